// sweep_any.cu -- FP32 CUDA-core sweeps of grids whose rows TMA cannot read
// (a base or a pitch that is no multiple of 16 bytes: the dense grid of an odd
// nx, or nx + 2r = 514).
//
// The march of sweep_cc.cuh (a column of TX x TY outputs, a register queue
// along z) and of sweep_2d.cu (a strip of row blocks), with the ring filled by
// cp.async instead of TMA: every thread copies the same few elements of every
// plane, whose offsets it works out once, and a plane is waited for by its
// copy group and one CTA barrier.  The copies are 8 bytes where base and
// pitches are even, else 4 (cp.async's sizes that need no 16-byte alignment);
// the tile's padding and the columns and rows past the grid are not read, and
// feed no stored output.
//
// The one-thread-per-point kernel was bound by its loads (6r + 1 or (2r+1)^3 of
// them per point): star r = 2 on 301 x 260 x 230, 166 -> 43 us (3.4 TB/s of
// algorithmic bytes, half of HBM's rate); box r = 1 on a dense 512^3, 2.87 ->
// 0.22 ms.  What binds now is the copies: eleven of 4 bytes per thread and
// plane, whose instructions fill the load/store queue (star r = 2 on a dense
// 511 x 512 x 512: issue 47 %, DRAM 52 %, mio_throttle the top stall).
#include "common.cuh"
#include "tile.cuh"

namespace mms {
namespace {

// Copies n bytes (n <= N; the rest of the N is zeroed) from global to shared memory.
template <int N>
__device__ __forceinline__ void copy_async(float *dst, const void *src, int n)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(ptx::smem_u32(dst)), "l"(src), "n"(N), "r"(n)
                 : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// What a thread copies of every staged plane: V floats at each of NI places.
// FAST: tiles wholly inside the grid copy without looking at their places'
// bits (the 3D march: star r = 4, 512^3, 312 -> 289 us; the planar kernel is
// slower with the second copy of the code, 139 -> 165 us at r = 3).
template <typename G, int V, bool FAST>
struct Stager {
    static constexpr int ITEMS = G::BX / V * G::BY;
    static constexpr int NI = (ITEMS + G::NT - 1) / G::NT;
    uint32_t off[NI];      // from the plane's first element, in bytes
    uint32_t whole, part;  // places of V floats inside the grid; of one (the row's last)
    bool full;             // the whole tile is inside (no place needs its bits)

    // A plane of which the first `rows` rows and `cols` columns are inside the grid.
    __device__ __forceinline__ void aim(int rows, int cols, int pitch)
    {
        whole = part = 0u;
        full = rows >= G::BY && cols >= G::BX;
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const int e = threadIdx.x + i * G::NT;
            const int row = e / (G::BX / V), col = e % (G::BX / V) * V;
            off[i] = (uint32_t)(row * pitch + col) * 4u;
            if (e < ITEMS && row < rows) {
                if (col + V <= cols) whole |= 1u << i;
                else if (col < cols) part |= 1u << i;
            }
        }
    }
    __device__ __forceinline__ void copy(float *stage, const float *plane) const
    {
        const char *p = reinterpret_cast<const char *>(plane);
        if (FAST && full) {
#pragma unroll
            for (int i = 0; i < NI; ++i)
                if ((i + 1) * G::NT <= ITEMS || threadIdx.x + i * G::NT < ITEMS)
                    copy_async<V * 4>(stage + (threadIdx.x + i * G::NT) * V, p + off[i], V * 4);
        } else {
#pragma unroll
            for (int i = 0; i < NI; ++i)
                if ((whole | part) >> i & 1u)
                    copy_async<V * 4>(stage + (threadIdx.x + i * G::NT) * V, p + off[i], whole >> i & 1u ? V * 4 : 4);
        }
    }
};

template <int PY>
__device__ __forceinline__ void store_rows(const f2 (&o)[PY][2], float *out, int64_t opy, int y, int ny, int gx, int nx,
                                           int vec)
{
#pragma unroll
    for (int i = 0; i < PY; ++i) {
        if (y + i >= ny || gx >= nx) continue;
        float *p = out + (int64_t)(y + i) * opy + gx;
        float v[4];
        unpair(o[i][0], v[0], v[1]);
        unpair(o[i][1], v[2], v[3]);
        if (vec && gx + 3 < nx) {
            *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (gx + k < nx) p[k] = v[k];
        }
    }
}

template <int R, int TX, int TY, int PY, int S, int V, bool BOX, typename Coef>
__global__ void __launch_bounds__(Geom<R, TX, TY, PY, S>::NT)
    sweep_any_kernel(const float *__restrict__ in, int ipy, int64_t ipz, const __grid_constant__ Coef cf,
                     float *__restrict__ out, int nx, int ny, int nz, int64_t opy, int64_t opz,
                     const __grid_constant__ March march, int vec)
{
    using G = Geom<R, TX, TY, PY, S>;
    constexpr int W = G::W;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float *planes = reinterpret_cast<float *>(smem_align128(smem_raw));
    const int tx = threadIdx.x % G::NTX, ry0 = threadIdx.x / G::NTX * PY;
    const Leg leg = leg_of(march);
    const int x0 = leg.tx * TX, y0 = leg.ty * TY, zb = leg.zc * march.tz;
    const int P = min(march.tz, nz - zb) + 2 * R;  // padded planes this CTA consumes
    const int gx = x0 + 4 * tx;
    const float *src = in + (int64_t)zb * ipz + (int64_t)y0 * ipy + x0;

    Stager<G, V, true> st;
    st.aim(ny + 2 * R - y0, nx + 2 * R - x0, ipy);
#pragma unroll
    for (int j = 0; j < S - 1; ++j) {
        if (j < P) st.copy(planes + j * G::STAGE, src + j * ipz);
        copy_commit();
    }
    f2 acc[W][PY][2];
#pragma unroll
    for (int kk = 0; kk < W; ++kk)
#pragma unroll
        for (int i = 0; i < PY; ++i) acc[kk][i][0] = acc[kk][i][1] = zero2();

    for (int j = 0; j < P; ++j) {
        copy_wait<S - 2>();  // this thread's part of plane j has landed
        __syncthreads();     // everyone's has, and everyone is done with plane j - 1
        const int n = j + S - 1;
        if (n < P) st.copy(planes + n % S * G::STAGE, src + n * ipz);
        copy_commit();
        const float *pl = planes + j % S * G::STAGE;
        if constexpr (BOX)
            box_plane<R, PY, G::BX, G::NV>(pl, cf, acc, tx, ry0);
        else
            star_plane<R, PY, G::BX, G::NV>(pl, cf, acc, tx, ry0);
        if (j >= 2 * R) store_rows<PY>(acc[0], out + (int64_t)(zb + j - 2 * R) * opz, opy, y0 + ry0, ny, gx, nx, vec);
#pragma unroll
        for (int kk = 0; kk < W - 1; ++kk)
#pragma unroll
            for (int i = 0; i < PY; ++i)
#pragma unroll
                for (int h = 0; h < 2; ++h) acc[kk][i][h] = acc[kk + 1][i][h];
#pragma unroll
        for (int i = 0; i < PY; ++i) acc[W - 1][i][0] = acc[W - 1][i][1] = zero2();
    }
}

// Planar shapes: `blocks` row blocks of TY rows of one plane per CTA.
template <int R, int TX, int TY, int PY, int S, int V, bool BOX, typename Coef>
__global__ void __launch_bounds__(Geom<R, TX, TY, PY, S>::NT)
    plane_any_kernel(const float *__restrict__ in, int ipy, int64_t ipz, const __grid_constant__ Coef cf,
                     float *__restrict__ out, int nx, int ny, int64_t opy, int64_t opz, int blocks, int vec)
{
    using G = Geom<R, TX, TY, PY, S>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float *stages = reinterpret_cast<float *>(smem_align128(smem_raw));
    const int tx = threadIdx.x % G::NTX, ry0 = threadIdx.x / G::NTX * PY;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * blocks * TY, gx = x0 + 4 * tx;
    const int P = min(blocks, (ny - y0 + TY - 1) / TY);
    const float *src = in + (int64_t)blockIdx.z * ipz + (int64_t)y0 * ipy + x0;
    out += (int64_t)blockIdx.z * opz;

    Stager<G, V, false> st;
    st.aim(G::BY, nx + 2 * R - x0, ipy);
    auto copy = [&](int j) {
        // the block that reaches past the grid's last padded row
        if (ny + 2 * R - y0 - j * TY < G::BY) st.aim(ny + 2 * R - y0 - j * TY, nx + 2 * R - x0, ipy);
        st.copy(stages + j % S * G::STAGE, src + (int64_t)j * TY * ipy);
    };
#pragma unroll
    for (int j = 0; j < S - 1; ++j) {
        if (j < P) copy(j);
        copy_commit();
    }
    for (int j = 0; j < P; ++j) {
        copy_wait<S - 2>();
        __syncthreads();
        if (j + S - 1 < P) copy(j + S - 1);
        copy_commit();
        f2 o[PY][2];
        if constexpr (BOX)
            box2d_tile<R, PY, G::BX, G::NV>(stages + j % S * G::STAGE, cf, o, tx, ry0);
        else
            star2d_tile<R, PY, G::BX, G::NV, true>(stages + j % S * G::STAGE, cf, o, tx, ry0);
        store_rows<PY>(o, out, opy, y0 + j * TY + ry0, ny, gx, nx, vec);
    }
}

// The tuned tiles of the TMA forms: star and box r <= 2 two rows per thread,
// box r = 3, 4 one (their 343 and 729 weights leave no registers for two).
template <int R, int V, bool BOX, typename Coef>
cudaError_t launch_3d(const Sweep &s, const Coef &cf)
{
    constexpr int TX = 64, TY = 16, PY = BOX && R > 2 ? 1 : 2, S = 4;
    using G = Geom<R, TX, TY, PY, S>;
    auto kern = sweep_any_kernel<R, TX, TY, PY, S, V, BOX, Coef>;
    static SlotCache cache;
    Slots sl;
    cudaError_t e = kernel_slots(cache, reinterpret_cast<const void *>(kern), G::NT, G::SMEM, &sl);
    if (e != cudaSuccess) return e;
    int64_t ctas;
    size_t smem = G::SMEM;
    const March march = plan_march(sl, (s.nx + TX - 1) / TX, (s.ny + TY - 1) / TY, 1, s.nz, 2 * R, 128, G::NT, &smem,
                                   &ctas);
    if (ctas > INT32_MAX) return cudaErrorInvalidConfiguration;
    const int vec = s.opy % 4 == 0 && s.opz % 4 == 0 && reinterpret_cast<uintptr_t>(s.out) % 16 == 0;
    kern<<<(unsigned)ctas, G::NT, smem, s.stream>>>(s.in, (int)s.ipy, s.ipz, cf, s.out, (int)s.nx, (int)s.ny, (int)s.nz,
                                                    s.opy, s.opz, march, vec);
    return cudaGetLastError();
}

template <int R, int V, bool BOX, typename Coef>
cudaError_t launch_2d(const Sweep &s, const Coef &cf)
{
    constexpr int TX = 64, TY = 32, PY = 4, S = 3;
    using G = Geom<R, TX, TY, PY, S>;
    auto kern = plane_any_kernel<R, TX, TY, PY, S, V, BOX, Coef>;
    static SlotCache cache;
    Slots sl;
    cudaError_t e = kernel_slots(cache, reinterpret_cast<const void *>(kern), G::NT, G::SMEM, &sl);
    if (e != cudaSuccess) return e;
    const int64_t tiles_x = (s.nx + TX - 1) / TX, tiles_y = (s.ny + TY - 1) / TY;
    const int blocks = z_chunk(sl, tiles_x * s.nz, tiles_y, 0, 8, G::NT);
    note_planes(blocks);
    const dim3 grid((unsigned)tiles_x, (unsigned)((tiles_y + blocks - 1) / blocks), (unsigned)s.nz);
    const int vec = s.opy % 4 == 0 && s.opz % 4 == 0 && reinterpret_cast<uintptr_t>(s.out) % 16 == 0;
    kern<<<grid, G::NT, G::SMEM, s.stream>>>(s.in, (int)s.ipy, s.ipz, cf, s.out, (int)s.nx, (int)s.ny, s.opy, s.opz,
                                             blocks, vec);
    return cudaGetLastError();
}

template <int R, int V>
cudaError_t launch_shape(const Sweep &s)
{
    constexpr int w = 2 * R + 1;
    if (s.shape == MMS_BOX || s.shape == MMS_BOX2D) {
        BoxCoef cf{};
        const int n = s.shape == MMS_BOX ? w * w * w : w * w;
        for (int i = 0; i < n; ++i) cf.c[i] = s.coeffs[i];
        return s.shape == MMS_BOX ? launch_3d<R, V, true>(s, cf) : launch_2d<R, V, true>(s, cf);
    }
    StarCoef cf{};
    cf.set(s.coeffs, s.shape == MMS_STAR ? 3 * w : 2 * w);
    return s.shape == MMS_STAR ? launch_3d<R, V, false>(s, cf) : launch_2d<R, V, false>(s, cf);
}

template <int V>
cudaError_t launch_r(const Sweep &s)
{
    switch (s.r) {
        case 1: return launch_shape<1, V>(s);
        case 2: return launch_shape<2, V>(s);
        case 3: return launch_shape<3, V>(s);
        case 4: return launch_shape<4, V>(s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

// Points from which the staged kernels are the faster ones.  Below, a march's
// latency (its planes one after the other) is longer than the point-by-point
// kernel's single chain of loads.  Device time, point by point against staged:
// star r = 4, 9^3 3.0 and 4.7 us, 57^3 5.0 and 5.6, 65 x 67 x 63 (274 k points)
// 6.1 and 7.0, 129 x 33 x 65 6.2 and 7.4; 255 x 255 x 5 (325 k) and 95^3 the
// other way round, 79^3 8.1 and 8.9 at r = 3, at r = 1 even from 41^3 on; box r =
// 4, 31^3 38 and 42 us, 15 x 20 x 301 46 and 57, 47^3 the other way round (boxes
// of smaller radius at every size); planar star 17^2 2.0 and 2.2, 65^2 even.
static int64_t staged_from(int shape, int r)
{
    switch (shape) {
        case MMS_STAR: return 300000;
        case MMS_BOX: return r == 4 ? 100000 : 0;
        case MMS_STAR2D: return 4096;
        default: return 0;
    }
}

// Row offsets inside a staged tile (at most 40 rows) are 32-bit, input
// elements 4-byte aligned, and the planar grid's launch extents are CUDA's.
bool any_pitch_ok(const Sweep &s)
{
    return s.nx * s.ny * s.nz >= staged_from(s.shape, s.r) && s.ipy < (1 << 24) && reinterpret_cast<uintptr_t>(s.in) % 4 == 0 &&
           (!is_planar(s.shape) || (s.nz <= 65535 && s.ny <= (int64_t)65535 * 32));
}

cudaError_t launch_any(const Sweep &s)
{
    const bool even = s.ipy % 2 == 0 && s.ipz % 2 == 0 && reinterpret_cast<uintptr_t>(s.in) % 8 == 0;
    return even ? launch_r<2>(s) : launch_r<1>(s);
}

}  // namespace mms
