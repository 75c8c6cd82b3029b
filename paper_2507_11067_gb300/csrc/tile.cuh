// tile.cuh -- the shared-memory plane tile of the CUDA-core sweeps and of
// the fused wave kernels: its geometry and the per-plane star and box
// updates of a thread's register queue of partial sums.
#pragma once

#include "common.cuh"

namespace mms {

// The dynamic shared-memory base rounded up to 128 bytes (TMA destinations
// need 128-byte alignment; the launch adds 128 bytes of slack for this).
__device__ __forceinline__ unsigned char *smem_align128(unsigned char *p)
{
    const uint32_t a = ptx::smem_u32(p);  // offset in the shared window
    return p + ((128u - (a & 127u)) & 127u);
}

template <int R, int TX, int TY, int PY, int S>
struct Geom {
    static constexpr int W = 2 * R + 1;
    static constexpr int BX = (TX + 2 * R + 3) & ~3;  // TMA box x: a 16-byte multiple
    static constexpr int BY = TY + 2 * R;
    static constexpr int PLANE = BX * BY;             // floats one TMA box writes
    static constexpr int STAGE = (PLANE + 31) & ~31;  // ring stride: 128-byte multiple
    static constexpr int NTX = TX / 4;                // threads along x (4 points each)
    static constexpr int NT = NTX * (TY / PY);
    static constexpr int NV = (4 + 2 * R + 3) / 4;    // float4 per window row
    // 128 bytes of slack to align the dynamic base, the ring, its barriers
    // and the CTA's abort flag.
    static constexpr size_t SMEM = 128 + (size_t)S * STAGE * sizeof(float) + S * sizeof(uint64_t) + 16;
    static_assert(TX % 4 == 0 && TY % PY == 0, "tile");
    static_assert(BX <= 256 && BY <= 256, "TMA box dims are at most 256");
    static_assert(4 * (NTX - 1) + 4 * NV <= BX, "window inside the staged row");
};

// Loads the NV float4 of a window row starting at `p` (16-byte aligned).
template <int NV>
__device__ __forceinline__ void load_row(const float *p, float (&v)[4 * NV])
{
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        const float4 t = *reinterpret_cast<const float4 *>(p + 4 * q);
        v[4 * q + 0] = t.x;
        v[4 * q + 1] = t.y;
        v[4 * q + 2] = t.z;
        v[4 * q + 3] = t.w;
    }
}

// The 4 values at columns R..R+3 of a row whose column 0 is 16-byte aligned.
template <int R>
__device__ __forceinline__ void load_center(const float *p, float (&v)[4])
{
    constexpr int A = (R / 4) * 4;
    constexpr int o = R - A;
    const float4 t0 = *reinterpret_cast<const float4 *>(p + A);
    if constexpr (o == 0) {
        v[0] = t0.x; v[1] = t0.y; v[2] = t0.z; v[3] = t0.w;
    } else {
        const float4 t1 = *reinterpret_cast<const float4 *>(p + A + 4);
        const float tmp[8] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = tmp[o + k];
    }
}

// ---------------------------------------------------------------- pairs
// Two neighbouring points in one 64-bit register pair.  fma.rn.f32x2 is the
// same two IEEE FMAs in one instruction: the FP32 pipe does no more of them
// per clock (73 against 76 TFLOP/s measured), but a plane update issues half
// as many instructions, and issue is what binds these kernels (64 to 91 % of
// the cycles against 36 % for the pipe).
using f2 = float2;

__device__ __forceinline__ f2 pair(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ f2 pair(const W2 &w) { return make_float2(w.lo, w.hi); }
__device__ __forceinline__ f2 zero2() { return make_float2(0.f, 0.f); }
__device__ __forceinline__ void unpair(const f2 &v, float &a, float &b)
{
    a = v.x;
    b = v.y;
}
__device__ __forceinline__ f2 fma2(const f2 &a, const f2 &b, const f2 &c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ f2 mul2(const f2 &a, const f2 &b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ f2 add2(const f2 &a, const f2 &b) { return __fadd2_rn(a, b); }

// Whether a star update of radius R works on pairs: radius 3 and 4 are bound
// by issue (1024^3: r = 4 1.62 -> 1.39 ms, r = 3 1.40 -> 1.37 ms, HBM at 91
// %); at r = 1, 2 HBM binds already and pairs only cost registers (r = 2:
// 1.29 -> 1.55 ms).  The boxes are bound by the FMA pipe, which pairs do not
// relieve (r = 1, 512^3: 171 -> 188 us; 2D box r = 3: 117 -> 119 us).
template <int R>
constexpr bool kPairs = R >= 3;

// acc += w * v over a pair of points; point by point (WHOLE false) where v's
// halves do not share an aligned register pair: the moves that would pair them
// cost as much as the FMA they save, and take the FMA pipe as well.
template <bool WHOLE>
__device__ __forceinline__ void fma_pair(const W2 &w, const f2 &v, f2 &acc)
{
    if constexpr (WHOLE) {
        acc = fma2(pair(w), v, acc);
    } else {
        acc.x = fmaf(w.lo, v.x, acc.x);
        acc.y = fmaf(w.lo, v.y, acc.y);
    }
}

// acc (points 2h, 2h + 1) += w[d + R] * row[k + R + d]: tap d of the points'
// window row.  A tap whose columns start on an even register pairs with its
// neighbour.
template <int R>
__device__ __forceinline__ void tap_x(const W2 *w, const float *row, int d, int h, f2 &acc)
{
    const f2 v = pair(row[2 * h + R + d], row[2 * h + R + d + 1]);
    if (kPairs<R> && (R + d) % 2 == 0) fma_pair<true>(w[d + R], v, acc);
    else fma_pair<false>(w[d + R], v, acc);
}

// The four points' x line: every tap, d ascending.
template <int R>
__device__ __forceinline__ void line_x(const W2 *w, const float *row, f2 (&acc)[2])
{
#pragma unroll
    for (int d = -R; d <= R; ++d)
#pragma unroll
        for (int h = 0; h < 2; ++h) tap_x<R>(w, row, d, h, acc[h]);
}

// The centre values (columns R..R+3) of a staged row, as two pairs.
template <int R>
__device__ __forceinline__ void load_center2(const float *p, f2 (&v)[2])
{
    float c[4];
    load_center<R>(p, c);
    v[0] = pair(c[0], c[1]);
    v[1] = pair(c[2], c[3]);
}

// Queue slots: logical slot kk (output plane j - 2R + kk for input plane j)
// lives in acc[(kk + ROT) % (2R+1)]; ROT = 0 for a queue that is shifted
// after every plane, a compile-time rotation for one that is not.  A point's
// four x neighbours are two pairs.
//
// Star: plane j adds c_z[R-kk] * centre to the output plane at queue slot kk
// and its in-plane x/y part to slot R (the plane it centres).
template <int R, int PY, int BX, int NV, int ROT = 0>
__device__ __forceinline__ void star_plane(const float *pl, const StarCoef &cf, f2 (&acc)[2 * R + 1][PY][2], int tx,
                                           int ry0)
{
    constexpr int W = 2 * R + 1;
    f2 cen[PY + 2 * R][2];
#pragma unroll
    for (int rr = 0; rr < PY + 2 * R; ++rr) load_center2<R>(pl + (ry0 + rr) * BX + 4 * tx, cen[rr]);
#pragma unroll
    for (int i = 0; i < PY; ++i) {
        float win[4 * NV];
        load_row<NV>(pl + (ry0 + R + i) * BX + 4 * tx, win);
        f2 xy[2] = {zero2(), zero2()};
        line_x<R>(cf.c, win, xy);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
            for (int d = -R; d <= R; ++d) fma_pair<kPairs<R> && R % 2 == 0>(cf.c[1 * W + d + R], cen[i + R + d][h], xy[h]);
            acc[(R + ROT) % W][i][h] = add2(acc[(R + ROT) % W][i][h], xy[h]);
#pragma unroll
            for (int kk = 0; kk < W; ++kk)
                fma_pair<kPairs<R> && R % 2 == 0>(cf.c[2 * W + 2 * R - kk], cen[i + R][h], acc[(kk + ROT) % W][i][h]);
        }
    }
}

// Box: window row rr of the plane feeds output row i with dy = rr - R - i;
// slot kk (output plane z_o) takes the weights of dz = R - kk.
template <int R, int PY, int BX, int NV, int ROT = 0>
__device__ __forceinline__ void box_plane(const float *pl, const BoxCoef &cf, f2 (&acc)[2 * R + 1][PY][2], int tx,
                                          int ry0)
{
    constexpr int W = 2 * R + 1;
#pragma unroll
    for (int rr = 0; rr < PY + 2 * R; ++rr) {
        float row[4 * NV];
        load_row<NV>(pl + (ry0 + rr) * BX + 4 * tx, row);
#pragma unroll
        for (int i = 0; i < PY; ++i) {
            const int dy = rr - R - i;
            if (dy < -R || dy > R) continue;
#pragma unroll
            for (int kk = 0; kk < W; ++kk) {
                const int dz = R - kk;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    f2 &q = acc[(kk + ROT) % W][i][k / 2];
                    float a = k % 2 ? q.y : q.x;
#pragma unroll
                    for (int dx = -R; dx <= R; ++dx)
                        a = fmaf(cf.c[((dz + R) * W + dy + R) * W + dx + R], row[k + R + dx], a);
                    (k % 2 ? q.y : q.x) = a;
                }
            }
        }
    }
}

// Planar star (Table I's 2D kernels): the thread's 4 x PY outputs of a staged
// tile, x line (weights c[0..2R]) plus y line (weights c[2R+1..4R+1]); line
// after line, or (BY_TAP) tap d of both lines before tap d + 1, the order of
// the point-by-point kernel.
template <int R, int PY, int BX, int NV, bool BY_TAP = false>
__device__ __forceinline__ void star2d_tile(const float *pl, const StarCoef &cf, f2 (&o)[PY][2], int tx, int ry0)
{
    constexpr int W = 2 * R + 1;
    f2 cen[PY + 2 * R][2];
#pragma unroll
    for (int rr = 0; rr < PY + 2 * R; ++rr) load_center2<R>(pl + (ry0 + rr) * BX + 4 * tx, cen[rr]);
#pragma unroll
    for (int i = 0; i < PY; ++i) {
        float win[4 * NV];
        load_row<NV>(pl + (ry0 + R + i) * BX + 4 * tx, win);
        o[i][0] = o[i][1] = zero2();
        if constexpr (!BY_TAP) line_x<R>(cf.c, win, o[i]);
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int d = -R; d <= R; ++d) {
                if constexpr (BY_TAP) tap_x<R>(cf.c, win, d, h, o[i][h]);
                fma_pair<kPairs<R> && R % 2 == 0>(cf.c[W + d + R], cen[i + R + d][h], o[i][h]);
            }
    }
}

// Planar box: window row rr of the tile feeds output row i with dy = rr - R - i.
template <int R, int PY, int BX, int NV>
__device__ __forceinline__ void box2d_tile(const float *pl, const BoxCoef &cf, f2 (&o)[PY][2], int tx, int ry0)
{
    constexpr int W = 2 * R + 1;
#pragma unroll
    for (int i = 0; i < PY; ++i)
        for (int h = 0; h < 2; ++h) o[i][h] = zero2();
#pragma unroll
    for (int rr = 0; rr < PY + 2 * R; ++rr) {
        float row[4 * NV];
        load_row<NV>(pl + (ry0 + rr) * BX + 4 * tx, row);
#pragma unroll
        for (int i = 0; i < PY; ++i) {
            const int dy = rr - R - i;
            if (dy < -R || dy > R) continue;
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int dx = -R; dx <= R; ++dx) {
                    float &q = k % 2 ? o[i][k / 2].y : o[i][k / 2].x;
                    q = fmaf(cf.c[(dy + R) * W + dx + R], row[k + R + dx], q);
                }
        }
    }
}

}  // namespace mms
