// wave.cu -- fused acoustic wave step, its discrete adjoint, and the small
// pointwise kernels around them (model, chain rule, FP64 dot product).
//
// The forward kernel is the star sweep of sweep_cc.cu with the leapfrog
// update fused into its epilogue: the Laplacian of a^n never leaves
// registers, so one step moves 12 bytes per point and shot (read a^n, a^{n-1};
// write a^{n+1}) and 4 of m for all of them, plus the L2-served halos.  Shots
// are independent; those of a tile are neighbours in launch order, so that they
// share m in L2.
//
// The adjoint kernel computes, per point and shot,
//   lam^n = R^T r^n + 2 g lam^{n+1} + L(m g lam^{n+1}) - g^2 lam^{n+2}
//   grad += g lam^{n+1} (L a^n)     (FP64, all shots)
// staging lam^{n+1}, m and a^n planes with TMA; the stencil input
// q = m g lam^{n+1} is formed plane by plane in shared memory.
//
// The gradient path runs the same recursion in the scaled variable
// mu = m g lam (pointwise).  Multiplying the update by m g at the output
// point gives
//   mu^n = g (2 mu^{n+1} + m L mu^{n+1} - g mu^{n+2} + m R^T r^n)
//   grad += mu^{n+1} (L a^n)          (= m times the lam-form term)
// -- the forward step's form (the stencil on the state itself, m and g after
// it) -- so it runs on the forward kernel with no per-plane product and
// no barrier between forming and reading it; the accumulated gradient is
// divided by m once at the end (divide_m_kernel).  It needs m > 0.
#include <type_traits>
#include <utility>

#include "common.cuh"
#include "tile.cuh"
#include "wave.cuh"

namespace mms {

__device__ unsigned g_error_word = 0;

unsigned *device_error_word()
{
    static PerContext<unsigned *> cache;
    unsigned *addr = nullptr;
    if (cache.find(context_id(), &addr)) return addr;
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, g_error_word) != cudaSuccess) return nullptr;
    addr = static_cast<unsigned *>(p);
    cache.keep(context_id(), addr);
    return addr;
}

namespace {

// Failure-path self-test: one CTA waits, bounded by limit_ns, on an mbarrier
// phase that nothing completes; the wait runs out, records the timeout in
// the error word and the kernel returns -- the path that every bounded wait
// of the library takes, exercised without a fault.
__global__ void wait_selftest_kernel(unsigned long long limit_ns, unsigned *err)
{
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        ptx::mbar_init(&bar, 1);
        ptx::fence_mbar_init();
    }
    __syncthreads();
    (void)ptx::mbar_wait_bounded(&bar, 0, err, limit_ns);
}

// FP32 -> FP64 by the IEEE-754 layouts (sign kept, exponent rebased by
// 1023 - 127, fraction shifted up 29 bits), on the integer units: GB300's
// FP64 pipe issues about two instructions per clock per SM, which a
// conversion per point and plane would saturate.  Exact for every FP32
// value: a denormal f (fraction field F, f = F 2^-149) is normalised by the
// position of F's leading one (FP64 reaches far below 2^-149).
__device__ __forceinline__ double widen(float f)
{
    const uint32_t u = __float_as_uint(f), a = u & 0x7fffffffu;
    uint32_t hi = (a >> 3) + (896u << 20), lo = u << 29;
    if (a - 0x00800000u >= 0x7f000000u) {  // not a normal number
        if (a >= 0x7f800000u) {
            hi = 0x7ff00000u | (a & 0x7fffffu) >> 3;
        } else if (a == 0u) {
            hi = 0u;
        } else {
            // leading one of F at bit b = 23 - s: f = 1.xxx 2^(-126 - s)
            const uint32_t sh = (uint32_t)__clz(a) - 8u, frac = (a << sh) & 0x7fffffu;
            hi = (897u - sh) << 20 | frac >> 3;
            lo = frac << 29;
        }
    }
    return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)lo);
}

// Ring stage s: [a^n plane + halo | m tile | a^{n-1} tile | a^n tile].  The
// interior tiles of output plane zo = j - 2R (m, a^{n-1} and the centre
// values of a^n) ride in the stage of input plane j, the plane that completes
// zo, so every operand arrives asynchronously and no register queue of
// centre values is needed.
// The kernel's three forms: the forward step; the forward step that also
// writes L a^n; the adjoint step in the scaled variable mu = m G lam, whose
// update has the forward step's form (the stencil acts on the state itself),
// with the receiver residual m r^n in place of the source and the FP64
// gradient term mu^{n+1} (L a^n) = m G lam^{n+1} (L a^n), L a^n read from a
// fifth tile -- K_ADJ_BULK where a plane's terms leave by bulk reductions (one
// shared slice, rows of 16 bytes), K_ADJ for the rest (no gradient, atomics,
// per-shot slices): the bulk form's registers decide how many CTAs an SM
// holds, so it carries nothing of the others.
enum { K_FWD = 0, K_FWD_LAP = 1, K_ADJ = 2, K_ADJ_BULK = 3 };

template <int R, int TX, int TY, int PY, int S, int MODE = K_FWD>
struct FwdGeom {
    using G = Geom<R, TX, TY, PY, S>;
    using I = Interior<R, TX>;
    static constexpr int MT = I::BXI * TY;                  // floats of one interior tile
    // sub-tile offsets rounded to 32 floats: every TMA destination is 128-byte aligned
    static constexpr int OFF_M = (G::PLANE + 31) & ~31;
    static constexpr int OFF_P = OFF_M + ((MT + 31) & ~31);
    static constexpr int OFF_C = OFF_P + ((MT + 31) & ~31);
    static constexpr int OFF_L = OFF_C + ((MT + 31) & ~31);  // adjoint: L a^n
    static constexpr int STAGE = OFF_L + (MODE >= K_ADJ ? ((MT + 31) & ~31) : 0);
    // K_ADJ_BULK: two FP64 buffers of an output plane's gradient terms (TY x
    // TX), 128-byte aligned after the ring's barriers and abort flag
    static constexpr size_t OFF_GB = ((size_t)S * STAGE * 4 + S * sizeof(uint64_t) + 16 + 127) / 128 * 128;
    static constexpr size_t GB_BYTES = MODE == K_ADJ_BULK ? 2 * (size_t)TY * TX * sizeof(double) : 0;
    static constexpr size_t SMEM = 128 + OFF_GB + GB_BYTES;
};

// Programmatic dependent launch: the next kernel of the stream (launched
// with the programmatic-serialization attribute) may start once every CTA
// of this grid has signalled; a kernel so launched waits, before it touches
// global memory another kernel wrote or reads, until the previous grid has
// completed and its writes are visible.  Both are no-ops without the
// attribute.
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_prior_grid() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launches a kernel whose prologue may overlap the previous kernel of the
// stream (programmatic stream serialization); the kernel calls
// wait_prior_grid() before its first dependent global access.  A stream
// being captured into a graph gets a plain launch (a replayed graph has no
// launch gaps to hide).
template <typename... KArgs, typename... Args>
cudaError_t launch_overlapped(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              Args &&...args)
{
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) cs = cudaStreamCaptureStatusNone;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = cs == cudaStreamCaptureStatusNone ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<Args &&>(args)...);
}

// Bulk reduction of an FP64 row from shared memory into global memory (the
// L2 adds it), in this thread's bulk groups; addresses 16-byte aligned, size
// a multiple of 16 bytes.
__device__ __forceinline__ void bulk_add_f64(double *dst, const double *src, uint32_t bytes)
{
    asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f64 [%0], [%1], %2;" ::"l"(dst),
                 "r"(ptx::smem_u32(src)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// at most the most recent group may still be reading its source
__device__ __forceinline__ void bulk_wait_read_1() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Operands of the scaled adjoint (unused by the forward forms).
struct AdjArgs {
    const float *resid;  // nshots*ny*nx on the receiver plane, or null
    double *grad;        // FP64 gradient, or null (no gradient term, tlap unused)
    int gvec;            // rows of four doubles 32-byte aligned
    int gbulk;           // one shared slice, nx even, grad 16-byte aligned: rows added by bulk reductions
};

template <int R, int TX, int TY, int PY, int S, int MODE>
__global__ void __launch_bounds__(Geom<R, TX, TY, PY, S>::NT)
    wave_fwd_kernel(const __grid_constant__ CUtensorMap tcur, const __grid_constant__ CUtensorMap tm,
                    const __grid_constant__ CUtensorMap tprev, const __grid_constant__ CUtensorMap tctr,
                    const __grid_constant__ CUtensorMap tlap, const __grid_constant__ StarCoef cf,
                    const __grid_constant__ WaveGeo geo, float *__restrict__ pnext,
                    const float *__restrict__ amp, float *__restrict__ rec, float *__restrict__ lapout,
                    const __grid_constant__ AdjArgs adj, const __grid_constant__ March march, int vec, unsigned *err)
{
    constexpr bool LAPOUT = MODE == K_FWD_LAP;
    constexpr bool ADJ = MODE >= K_ADJ, gbulk = MODE == K_ADJ_BULK;
    using G = Geom<R, TX, TY, PY, S>;
    using F = FwdGeom<R, TX, TY, PY, S, MODE>;
    using I = Interior<R, TX>;
    constexpr int W = G::W;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char *smem = smem_align128(smem_raw);
    float *stages = reinterpret_cast<float *>(smem);
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + (size_t)S * F::STAGE * sizeof(float));
    int &abort_flag = *reinterpret_cast<int *>(full + S);

    // the next step's kernel may set up while this one runs
    launch_dependents();
    const int tid = threadIdx.x;
    const int tx = tid % G::NTX, ty = tid / G::NTX;
    const int ry0 = ty * PY;
    const bool has_grad = gbulk || (ADJ && adj.grad != nullptr);
    // gbulk: the shots' terms go to one shared gradient; each output plane's
    // terms are gathered in shared memory and each row is added by one bulk
    // reduction (the L2 does the adds), instead of one FP64 atomic per point.
    [[maybe_unused]] double *gbuf = reinterpret_cast<double *>(smem + F::OFF_GB);
    const int ntiles = has_grad ? 4 : 3;

    if (tid == 0) {
        ptx::prefetch_tmap(&tcur);
        ptx::prefetch_tmap(&tm);
        ptx::prefetch_tmap(&tprev);
        ptx::prefetch_tmap(&tctr);
        if (has_grad) ptx::prefetch_tmap(&tlap);
#pragma unroll
        for (int s = 0; s < S; ++s) ptx::mbar_init(&full[s], 1);
        ptx::fence_mbar_init();
        abort_flag = 0;
    }
    // the previous step's fields are complete before any is read or written
    wait_prior_grid();
    const Leg leg = leg_of(march);
    const int sh = leg.shot, x0 = leg.tx * TX, y0 = leg.ty * TY, zb = leg.zc * march.tz;
    const int P = min(march.tz, geo.nz - zb) + 2 * R;
    const int gx = x0 + 4 * tx;
    const int sx = ADJ ? -1 : geo.src[sh][0], sy = ADJ ? -1 : geo.src[sh][1], sz = ADJ ? -1 : geo.src[sh][2];
    auto issue = [&](int j) {
        const int s = j % S;
        float *st = stages + (size_t)s * F::STAGE;
        const bool inner = j >= 2 * R;  // this plane completes output plane j - 2R
        ptx::mbar_arrive_expect_tx(&full[s], (G::PLANE + (inner ? ntiles * F::MT : 0)) * sizeof(float));
        ptx::tma_load_4d(st, &tcur, x0, y0, zb + j, sh, &full[s]);
        if (inner) {
            const int zp = zb + j - R;  // padded plane of output zo = j - 2R
            const int xs = x0 + (R & ~3);
            ptx::tma_load_3d(st + F::OFF_M, &tm, xs, y0 + R, zp, &full[s]);
            ptx::tma_load_4d(st + F::OFF_P, &tprev, xs, y0 + R, zp, sh, &full[s]);
            ptx::tma_load_4d(st + F::OFF_C, &tctr, xs, y0 + R, zp, sh, &full[s]);
            if (has_grad) ptx::tma_load_4d(st + F::OFF_L, &tlap, xs, y0 + R, zp, sh, &full[s]);
        }
    };
    __syncthreads();
    if (tid == 0)
        for (int j = 0; j < S && j < P; ++j) issue(j);
    f2 gxy[PY][2];  // sponge factors g(x) g(y) of the thread's points
    {
        float gxs[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) gxs[k] = sponge(gx + k, geo.nx, geo.sponge_w, geo.sponge_a);
#pragma unroll
        for (int i = 0; i < PY; ++i) {
            const float gy = sponge(y0 + ry0 + i, geo.ny, geo.sponge_w, geo.sponge_a);
#pragma unroll
            for (int h = 0; h < 2; ++h) gxy[i][h] = mul2(pair(gxs[2 * h], gxs[2 * h + 1]), pair(gy, gy));
        }
    }

    f2 acc[W][PY][2];
#pragma unroll
    for (int kk = 0; kk < W; ++kk)
#pragma unroll
        for (int i = 0; i < PY; ++i) acc[kk][i][0] = acc[kk][i][1] = zero2();

    const float samp = ADJ ? 0.f : amp[sh];
    const int64_t shot_off = (int64_t)sh * geo.ss;
    for (int j = 0; j < P; ++j) {
        const int s = j % S;
        const float *st = stages + (size_t)s * F::STAGE;
        const int zo = j - 2 * R;  // output plane completed by plane j
        float mv[PY][4], pv[PY][4], cv[PY][4];
        [[maybe_unused]] float lv[PY][4];
        if (ptx::mbar_wait_bounded(&full[s], (uint32_t)(j / S) & 1u, err)) {
            star_plane<R, PY, G::BX, G::NV>(st, cf, acc, tx, ry0);
            if (zo >= 0) {
#pragma unroll
                for (int i = 0; i < PY; ++i) {
                    // interior tiles: row ry0+i, columns 4tx+OFF .. +3
                    load_center<I::OFF>(st + F::OFF_M + (ry0 + i) * I::BXI + 4 * tx, mv[i]);
                    load_center<I::OFF>(st + F::OFF_P + (ry0 + i) * I::BXI + 4 * tx, pv[i]);
                    load_center<I::OFF>(st + F::OFF_C + (ry0 + i) * I::BXI + 4 * tx, cv[i]);
                    if constexpr (ADJ)
                        if (has_grad) load_center<I::OFF>(st + F::OFF_L + (ry0 + i) * I::BXI + 4 * tx, lv[i]);
                }
            }
        } else {
            abort_flag = 1;
        }
        __syncthreads();
        if (abort_flag) {
            if constexpr (gbulk) bulk_wait_all();  // no reduction still reads this CTA's buffers
            return;
        }
        if (tid == 0 && j + S < P) issue(j + S);
        if (zo >= 0) {
            const int z = zb + zo;
            const float gzv = sponge(z, geo.nz, geo.sponge_w, geo.sponge_a);
            // this output plane's gradient buffer; the reductions of the plane
            // before last, which read it, are done first
            [[maybe_unused]] double *gb = gbuf + (size_t)(zo & 1) * (TY * TX);
            if constexpr (gbulk) {
                if (tx == 0) bulk_wait_read_1();
                __syncwarp();
            }
#pragma unroll
            for (int i = 0; i < PY; ++i) {
                const int y = y0 + ry0 + i;
                if (y >= geo.ny || gx >= geo.nx) continue;
                const int64_t mp = (int64_t)(z + R) * geo.pz + (int64_t)(y + R) * geo.py + (gx + R);
                float *pp = pnext + shot_off + mp;
                float res[4], lap[4];
                unpair(acc[0][i][0], lap[0], lap[1]);
                unpair(acc[0][i][1], lap[2], lap[3]);
                [[maybe_unused]] double gd[4] = {0.0, 0.0, 0.0, 0.0};
                float g[4], v[4];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const f2 gg = mul2(gxy[i][h], pair(gzv, gzv));
                    const f2 c = pair(cv[i][2 * h], cv[i][2 * h + 1]), p = pair(pv[i][2 * h], pv[i][2 * h + 1]);
                    // (2 a + m L a) - g a', in this order of roundings and no
                    // other: a few roundings near the source decide the error
                    // of a whole run.  With fma(m, L a, 2 a) in the middle the
                    // gradient's error of 2 shots on 256^3, 40 steps, was
                    // 1.3e-6 where this has 5.4e-7.  (16 steps of 8 x 512^3
                    // take 42.08 ms, 41.77 with that; an add of 2 a to the
                    // product compiles into that fma again.)
                    const f2 t = mul2(pair(mv[i][2 * h], mv[i][2 * h + 1]), acc[0][i][h]);
                    const f2 u = fma2(pair(2.f, 2.f), c, t);
                    unpair(gg, g[2 * h], g[2 * h + 1]);
                    unpair(fma2(pair(-gg.x, -gg.y), p, u), v[2 * h], v[2 * h + 1]);
                }
                if constexpr (ADJ) {
                    if (adj.resid && z == geo.rec_z) {
                        const float *rs = adj.resid + ((int64_t)sh * geo.ny + y) * geo.nx + gx;
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            if (gx + k < geo.nx) v[k] += mv[i][k] * rs[k];
                    }
                    // mu^{n+1} (L a^n) = m G lam^{n+1} (L a^n): m is the same
                    // at every step, so the sum is divided by it once, at
                    // the end (mms_grad_divide_m).  The term in FP32 (its
                    // operands are FP32), accumulated in FP64.
                    if (has_grad)
#pragma unroll
                        for (int k = 0; k < 4; ++k) gd[k] = widen(cv[i][k] * lv[i][k]);
                } else if (z == sz && y == sy) {
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (gx + k == sx) v[k] += samp;
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) res[k] = g[k] * v[k];
                if (vec && gx + 3 < geo.nx) {
                    *reinterpret_cast<float4 *>(pp) = make_float4(res[0], res[1], res[2], res[3]);
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (gx + k < geo.nx) pp[k] = res[k];
                }
                if constexpr (LAPOUT) {  // L a^n itself, for the gradient's adjoint steps
                    float *lo = lapout + shot_off + mp;
                    if (vec && gx + 3 < geo.nx) {
                        *reinterpret_cast<float4 *>(lo) = make_float4(lap[0], lap[1], lap[2], lap[3]);
                    } else {
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            if (gx + k < geo.nx) lo[k] = lap[k];
                    }
                }
                if (rec && z == geo.rec_z) {
                    float *rp = rec + ((int64_t)sh * geo.ny + y) * geo.nx + gx;
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (gx + k < geo.nx) rp[k] = res[k];
                }
                if constexpr (ADJ) {
                    if (has_grad) {
                        const int64_t gi = ((int64_t)z * geo.ny + y) * geo.nx + gx;
                        if (gbulk) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) gb[(ry0 + i) * TX + 4 * tx + k] = gd[k];
                        } else if (geo.gss == 0) {
                            // one slice for all shots: other CTAs add to the same points
#pragma unroll
                            for (int k = 0; k < 4; ++k)
                                if (gx + k < geo.nx) atomicAdd(adj.grad + gi + k, gd[k]);
                        } else {
                            // this shot's own slice: no other thread touches these points
                            double *gp = adj.grad + (int64_t)sh * geo.gss + gi;
                            if (adj.gvec && gx + 3 < geo.nx) {
                                double2 *g2 = reinterpret_cast<double2 *>(gp);
                                double2 a = g2[0], b = g2[1];
                                a.x += gd[0]; a.y += gd[1]; b.x += gd[2]; b.y += gd[3];
                                g2[0] = a;
                                g2[1] = b;
                            } else {
#pragma unroll
                                for (int k = 0; k < 4; ++k)
                                    if (gx + k < geo.nx) gp[k] += gd[k];
                            }
                        }
                    }
                }
            }
            if constexpr (ADJ) {
                if (gbulk) {
                    // the terms reach the async proxy, then each row's first
                    // thread adds the row's valid points (an even count: nx
                    // and x0 are even) with one bulk reduction
                    ptx::fence_proxy_async_smem();
                    __syncwarp();
                    if (tx == 0) {
#pragma unroll
                        for (int i = 0; i < PY; ++i) {
                            const int y = y0 + ry0 + i;
                            if (y < geo.ny && x0 < geo.nx) {
                                const int n = min(TX, geo.nx - x0);
                                bulk_add_f64(adj.grad + ((int64_t)z * geo.ny + y) * geo.nx + x0, gb + (ry0 + i) * TX,
                                             (uint32_t)n * 8u);
                            }
                        }
                        bulk_commit();
                    }
                }
            }
        }
#pragma unroll
        for (int kk = 0; kk < W - 1; ++kk)
#pragma unroll
            for (int i = 0; i < PY; ++i)
#pragma unroll
                for (int h = 0; h < 2; ++h) acc[kk][i][h] = acc[kk + 1][i][h];
#pragma unroll
        for (int i = 0; i < PY; ++i) acc[W - 1][i][0] = acc[W - 1][i][1] = zero2();
    }
    // this thread's reductions are complete before the CTA exits
    if constexpr (ADJ)
        if (gbulk && tx == 0) bulk_wait_all();
}

// Adjoint step.  Ring stage s holds the planes lam^{n+1}, m, a^n (with halo)
// of input plane j and the interior tiles lam^{n+2} and lam^{n+1} of the
// output plane zo = j - 2R that plane j completes.
template <int R, int TX, int TY, int S>
struct AdjGeom {
    using G = Geom<R, TX, TY, 1, S>;
    using I = Interior<R, TX>;
    static constexpr int PL = (G::PLANE + 31) & ~31;   // padded plane stride
    static constexpr int MT = (I::BXI * TY + 31) & ~31;
    static constexpr int OFF_L2 = 3 * PL, OFF_L1 = OFF_L2 + MT;
    static constexpr int STAGE = OFF_L1 + MT;
    // [ring | q plane | sponge tables | barriers | abort flag]
    static constexpr size_t OFF_Q = (size_t)S * STAGE;
    static constexpr size_t OFF_GX = OFF_Q + PL;
    static constexpr size_t OFF_GY = OFF_GX + ((G::BX + 3) & ~3);
    static constexpr size_t OFF_BAR = OFF_GY + ((G::BY + 3) & ~3);
    static constexpr size_t SMEM = 128 + OFF_BAR * 4 + S * 8 + 16;
};

// LAPIN: the gradient term reads L a^n as a completed tile (written by the
// forward step that produced a^{n+1}) instead of staging a^n and applying
// the stencil here; the a^n plane's ring slot then holds that tile.
template <int R, int TX, int TY, int S, bool LAPIN>
__global__ void __launch_bounds__(Geom<R, TX, TY, 1, S>::NT, 2)
    wave_adj_kernel(const __grid_constant__ CUtensorMap tlam, const __grid_constant__ CUtensorMap tm,
                    const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tl2,
                    const __grid_constant__ CUtensorMap tl1, const __grid_constant__ StarCoef cf,
                    const __grid_constant__ WaveGeo geo, float *__restrict__ lprev,
                    const float *__restrict__ resid, double *__restrict__ grad, int has_a, int tz,
                    int nzc, int gvec, unsigned *err)
{
    constexpr int PY = 1;
    using G = Geom<R, TX, TY, PY, S>;
    using A = AdjGeom<R, TX, TY, S>;
    using I = Interior<R, TX>;
    constexpr int W = G::W;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float *base = reinterpret_cast<float *>(smem_align128(smem_raw));
    float *qbuf = base + A::OFF_Q;
    float *gxt = base + A::OFF_GX;
    float *gyt = base + A::OFF_GY;
    uint64_t *full = reinterpret_cast<uint64_t *>(base + A::OFF_BAR);
    int &abort_flag = *reinterpret_cast<int *>(full + S);

    const int tid = threadIdx.x;
    const int tx = tid % G::NTX, ty = tid / G::NTX;
    const int sh = blockIdx.z / nzc, zc = blockIdx.z % nzc;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, zb = zc * tz;
    const int nzt = min(tz, geo.nz - zb);
    const int P = nzt + 2 * R;
    const int ry0 = ty * PY;
    const int gx = x0 + 4 * tx;
    const uint32_t plane_bytes = (has_a && !LAPIN ? 3u : 2u) * G::PLANE * sizeof(float);

    for (int c = tid; c < G::BX; c += G::NT) gxt[c] = sponge(x0 + c - R, geo.nx, geo.sponge_w, geo.sponge_a);
    for (int rr = tid; rr < G::BY; rr += G::NT) gyt[rr] = sponge(y0 + rr - R, geo.ny, geo.sponge_w, geo.sponge_a);
    if (tid == 0) {
        ptx::prefetch_tmap(&tlam);
        ptx::prefetch_tmap(&tm);
        ptx::prefetch_tmap(&tl2);
        ptx::prefetch_tmap(&tl1);
        if (has_a) ptx::prefetch_tmap(&ta);  // a^n planes, or L a^n tiles
#pragma unroll
        for (int s = 0; s < S; ++s) ptx::mbar_init(&full[s], 1);
        ptx::fence_mbar_init();
        abort_flag = 0;
    }
    __syncthreads();
    auto issue = [&](int j, int s) {
        float *st = base + (size_t)s * A::STAGE;
        const bool inner = j >= 2 * R;
        const uint32_t tiles = inner ? (LAPIN && has_a ? 3u : 2u) : 0u;
        ptx::mbar_arrive_expect_tx(&full[s], plane_bytes + tiles * I::BXI * TY * 4u);
        ptx::tma_load_4d(st, &tlam, x0, y0, zb + j, sh, &full[s]);
        ptx::tma_load_3d(st + A::PL, &tm, x0, y0, zb + j, &full[s]);
        if (has_a && !LAPIN) ptx::tma_load_4d(st + 2 * A::PL, &ta, x0, y0, zb + j, sh, &full[s]);
        if (inner) {
            const int zp = zb + j - R;
            const int xs = x0 + (R & ~3);
            ptx::tma_load_4d(st + A::OFF_L2, &tl2, xs, y0 + R, zp, sh, &full[s]);
            ptx::tma_load_4d(st + A::OFF_L1, &tl1, xs, y0 + R, zp, sh, &full[s]);
            if (LAPIN && has_a) ptx::tma_load_4d(st + 2 * A::PL, &ta, xs, y0 + R, zp, sh, &full[s]);
        }
    };
    if (tid == 0)
        for (int j = 0; j < S && j < P; ++j) issue(j, j);

    f2 accq[W][PY][2], acca[W][PY][2];
#pragma unroll
    for (int kk = 0; kk < W; ++kk)
#pragma unroll
        for (int h = 0; h < 2; ++h) accq[kk][0][h] = acca[kk][0][h] = zero2();
    float gxs[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) gxs[k] = gxt[4 * tx + R + k];
    const float gys0 = gyt[ry0 + R];
    const int64_t shot_off = (int64_t)sh * geo.ss;

    // Input plane j; the oldest partial sums (output plane j - 2R) are in
    // queue slot 0.  Returns false when the CTA aborts.  (Rotating the two
    // queues instead of shifting them, as the sweeps do, spills registers
    // here and was measured slower.)
    auto plane = [&](int j) -> bool {
        constexpr int Q = 0;
        const int s = j % S;
        const float *st = base + (size_t)s * A::STAGE;
        const int zo = j - 2 * R;
        const bool ok = ptx::mbar_wait_bounded(&full[s], (uint32_t)(j / S) & 1u, err);
        if (ok) {
            // q = m * g * lam^{n+1} over the whole staged plane, four columns
            // per item (the staged rows are 16-byte multiples)
            const float gzp = sponge(zb + j - R, geo.nz, geo.sponge_w, geo.sponge_a);
            constexpr int BX4 = G::BX / 4;
            for (int e4 = tid; e4 < BX4 * G::BY; e4 += G::NT) {
                const int c4 = e4 % BX4, rr = e4 / BX4;
                const int e = rr * G::BX + 4 * c4;
                const float4 lv = *reinterpret_cast<const float4 *>(st + e);
                const float4 mv = *reinterpret_cast<const float4 *>(st + A::PL + e);
                const float4 gx = *reinterpret_cast<const float4 *>(gxt + 4 * c4);
                const float gy = gyt[rr];
                float4 q;
                q.x = mv.x * (gx.x * gy * gzp) * lv.x;
                q.y = mv.y * (gx.y * gy * gzp) * lv.y;
                q.z = mv.z * (gx.z * gy * gzp) * lv.z;
                q.w = mv.w * (gx.w * gy * gzp) * lv.w;
                *reinterpret_cast<float4 *>(qbuf + e) = q;
            }
        } else {
            abort_flag = 1;
        }
        __syncthreads();
        if (abort_flag) return false;
        float l2v[4], l1v[4], lav[4];
        {
            star_plane<R, PY, G::BX, G::NV, Q>(qbuf, cf, accq, tx, ry0);
            if (!LAPIN && has_a) star_plane<R, PY, G::BX, G::NV, Q>(st + 2 * A::PL, cf, acca, tx, ry0);
            if (zo >= 0) {
                load_center<I::OFF>(st + A::OFF_L2 + ry0 * I::BXI + 4 * tx, l2v);
                load_center<I::OFF>(st + A::OFF_L1 + ry0 * I::BXI + 4 * tx, l1v);
                if (LAPIN && has_a) load_center<I::OFF>(st + 2 * A::PL + ry0 * I::BXI + 4 * tx, lav);
            }
        }
        __syncthreads();
        if (tid == 0 && j + S < P) issue(j + S, s);
        if (zo >= 0) {
            const int z = zb + zo;
            const int y = y0 + ry0;
            if (y < geo.ny && gx < geo.nx) {
                const float gzv = sponge(z, geo.nz, geo.sponge_w, geo.sponge_a);
                const int64_t mp = (int64_t)(z + R) * geo.pz + (int64_t)(y + R) * geo.py + (gx + R);
                float *lp = lprev + shot_off + mp;
                const int64_t gi = ((int64_t)z * geo.ny + y) * geo.nx + gx;
                const bool at_rec = resid && z == geo.rec_z;
                double gd[4] = {0.0, 0.0, 0.0, 0.0};
                float lq[4], la[4];
                unpair(accq[Q][0][0], lq[0], lq[1]);
                unpair(accq[Q][0][1], lq[2], lq[3]);
                unpair(acca[Q][0][0], la[0], la[1]);
                unpair(acca[Q][0][1], la[2], la[3]);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (gx + k >= geo.nx) break;
                    const float g = gxs[k] * gys0 * gzv;
                    float v = 2.f * g * l1v[k] + lq[k] - g * g * l2v[k];
                    if (at_rec) v += resid[((int64_t)sh * geo.ny + y) * geo.nx + gx + k];
                    lp[k] = v;
                    // the step's term in FP32 (its operands are FP32), accumulated in FP64
                    if (has_a) gd[k] = widen(g * l1v[k] * (LAPIN ? lav[k] : la[k]));
                }
                if (has_a) {
                    if (geo.gss == 0) {
                        // one slice for all shots: other CTAs add to the same points
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            if (gx + k < geo.nx) atomicAdd(grad + gi + k, gd[k]);
                    } else {
                        // this shot's own slice: no other thread touches these points
                        double *gp = grad + (int64_t)sh * geo.gss + gi;
                        if (gvec && gx + 3 < geo.nx) {
                            double2 *g2 = reinterpret_cast<double2 *>(gp);
                            double2 a = g2[0], b = g2[1];
                            a.x += gd[0]; a.y += gd[1]; b.x += gd[2]; b.y += gd[3];
                            g2[0] = a;
                            g2[1] = b;
                        } else {
#pragma unroll
                            for (int k = 0; k < 4; ++k)
                                if (gx + k < geo.nx) gp[k] += gd[k];
                        }
                    }
                }
            }
        }
#pragma unroll
        for (int kk = 0; kk < W - 1; ++kk)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                accq[kk][0][h] = accq[kk + 1][0][h];
                acca[kk][0][h] = acca[kk + 1][0][h];
            }
#pragma unroll
        for (int h = 0; h < 2; ++h) accq[W - 1][0][h] = acca[W - 1][0][h] = zero2();
        return true;
    };
    for (int j = 0; j < P; ++j)
        if (!plane(j)) return;
}

// The pointwise kernels below run over rows of x, so that a point's place costs
// no division: with one per coordinate and point they took four times HBM's
// time (256^3: model 94 -> 26 us).  A block is 256 threads, 64 along each of
// four rows; narrow grids take fewer along more rows (5 x 300 x 300: model 17.5
// -> 7.4 us, division 25 -> 8.2).  T, the threads along x, is a template
// argument: with it in blockDim the loop along x is not unrolled (256^3: model
// 28 -> 45 us).
constexpr int kRowThreads = 256;
template <typename F>
void launch_rows(int64_t X, int64_t rows, F launch)
{
    const auto go = [&](auto t) {
        constexpr int T = decltype(t)::value, per = kRowThreads / T;
        const int64_t b = (rows + per - 1) / per;
        launch(t, (int)(b < 152 * 32 ? b : 152 * 32), dim3(T, per));
    };
    if (X <= 8) go(std::integral_constant<int, 8>{});
    else if (X <= 16) go(std::integral_constant<int, 16>{});
    else if (X <= 32) go(std::integral_constant<int, 32>{});
    else go(std::integral_constant<int, 64>{});
}

template <int T>
__global__ void __launch_bounds__(kRowThreads)
    model_kernel(const __grid_constant__ WaveGeo geo, const float *__restrict__ v, float *__restrict__ m, float s)
{
    const int r = geo.r, X = geo.nx + 2 * r;
    const int64_t Y = geo.ny + 2 * r, rows = Y * (geo.nz + 2 * r);
    for (int64_t row = (int64_t)blockIdx.x * (kRowThreads / T) + threadIdx.y; row < rows;
         row += (int64_t)gridDim.x * (kRowThreads / T)) {
        const int64_t zz = row / Y, yy = row - zz * Y, y = yy - r, z = zz - r;
        const bool inside = y >= 0 && y < geo.ny && z >= 0 && z < geo.nz;
        const float *vr = v + (z * geo.ny + y) * geo.nx;
        float *mr = m + zz * geo.pz + yy * geo.py;
        for (int xx = threadIdx.x; xx < X; xx += T) {
            const int x = xx - r;
            float val = 0.f;
            if (inside && x >= 0 && x < geo.nx) {
                const float vv = vr[x];
                val = vv * vv * s;
            }
            mr[xx] = val;
        }
    }
}

// grad[z][y][x] /= m at the interior point (FP64): the scaled adjoint's sum
// of mu^{n+1} (L a^n) turned into dJ/dm.  GB300's FP64 pipe makes an IEEE
// division per point the whole cost (256^3: 635 us, HBM's time is 49), so the
// quotient comes from a reciprocal of the FP32 m, kept as the sum of two FP32
// values (r + e, 47 bits, worked out on the FP32 pipe), and one FP64
// correction step: q = g r', q += (g - q m) r'.  That is the IEEE quotient: the
// first q is within 70 ulps, so g - q m (at most 32 bits) is exact, and the sum
// before its rounding is within 2^-40 ulp of g / m -- while a quotient of a
// 53-bit by a 24-bit number is at least 2^-25 ulp from every midpoint, so both
// round alike.  What this cannot serve (m outside 2^-60 .. 2^60, a quotient
// that is no number of moderate size) divides; the range is read off the bits,
// on the integer pipe.
__device__ __forceinline__ double divide_by_float(double g, float m)
{
    if (m >= 0x1p-60f && m <= 0x1p60f) {
        const float r = 1.f / m, e = r * fmaf(-m, r, 1.f);
        const double md = widen(m), rd = widen(r) + widen(e);
        const double q = g * rd;
        const uint32_t hi = (uint32_t)__double2hiint(q), ex = (hi >> 20) & 0x7ffu;
        if (ex - 123u < 1800u) return fma(fma(-q, md, g), rd, q);  // 2^-900 <= |q| < 2^900
        if (((uint32_t)__double2hiint(g) << 1 | (uint32_t)__double2loint(g)) == 0u) return g;
    }
    return g / (double)m;
}

template <int T>
__global__ void __launch_bounds__(kRowThreads)
    divide_m_kernel(const __grid_constant__ WaveGeo geo, const float *__restrict__ m, double *__restrict__ grad)
{
    const int r = geo.r;
    const int64_t rows = (int64_t)geo.ny * geo.nz;
    for (int64_t row = (int64_t)blockIdx.x * (kRowThreads / T) + threadIdx.y; row < rows;
         row += (int64_t)gridDim.x * (kRowThreads / T)) {
        const int64_t z = row / geo.ny, y = row - z * geo.ny;
        double *gr = grad + row * geo.nx;
        const float *mr = m + (z + r) * geo.pz + (y + r) * geo.py + r;
        for (int x = threadIdx.x; x < geo.nx; x += T) gr[x] = divide_by_float(gr[x], mr[x]);
    }
}

// gv = gm 2 v dt^2/h^2; s2 = 2 dt^2/h^2 (a factor of two rounds nothing)
__global__ void chain_kernel(const double *__restrict__ gm, const float *__restrict__ v,
                             double *__restrict__ gv, int64_t n, double s2)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        gv[i] = gm[i] * widen(v[i]) * s2;
}

__global__ void sum_kernel(const double *__restrict__ slices, int nslices, int64_t stride, int64_t n,
                           double *out)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double acc = slices[i];
        for (int s = 1; s < nslices; ++s) acc += slices[(int64_t)s * stride + i];
        out[i] = acc;
    }
}

__global__ void dot_kernel(const float *__restrict__ a, const float *__restrict__ b, int64_t n,
                           double *__restrict__ res)
{
    double acc = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        acc += (double)a[i] * (double)b[i];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    __shared__ double part[32];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        acc = threadIdx.x < blockDim.x / 32 ? part[threadIdx.x] : 0.0;
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (threadIdx.x == 0) atomicAdd(res, acc);
    }
}

constexpr int kFwdTX = 64, kFwdTY = 16, kFwdPY = 1, kFwdS = 3, kFwdTZ = 128;
constexpr int kAdjTX = 64, kAdjTY = 16, kAdjS = 2, kAdjTZ = 128;

// The march of a forward step (with L a^n out, `lap`, or without): the planes
// per CTA and the CTAs an SM may hold (*smem is raised to keep more off it)
// whose modelled time is least.  `filled`: the part of the tiles' points that
// are inside the grid.
//
// A plane step takes 0.69, 0.93, 1.16 us with one, two, three CTAs on an SM.
// The form that writes L a^n as well takes 0.72, 1.0, 1.33 us, and from 8 M
// points on (no longer served by L2) memory holds it up where the third CTA
// has whole tiles to do: 1.78 us at 95 % of the slots with points, 1.46 at 84
// %, 1.33 at 75 % (1 x 512^3: 519 us on two CTAs per SM, 568 on three).  CTAs
// of one length run in waves, a last wave that is not full hardly faster; a
// short last chunk fills the slots which that wave leaves, or runs after it.
// The scheduler does not spread the CTAs of one wave by itself: it may put the
// long ones on some SMs three at a time while others take the short ones (4 x
// 128 x 200 x 300 in chunks of 128, 128 and 44: 147 us, 117 with two per SM;
// in four of 75, 93).  Measured over 46 shapes of 1 to 8 shots, the plans take
// 0.5 % more time than the best ones (lap 1.8 %).  Over 110 others they take
// 0.50 of the time of 128 planes and two CTAs everywhere (lap 0.54), at most
// 0.97 (lap 1.06).
March plan_forward(const Slots &sl, int64_t tiles_x, int64_t tiles_y, const WaveGeo &g, int halo, int tz, bool lap,
                   double filled, size_t *smem, int64_t *ctas)
{
    const int64_t nz = g.nz, cols = tiles_x * tiles_y * g.nshots;
    const bool big = (double)g.nx * g.ny * (double)nz * g.nshots >= 8e6;
    // us of a plane step with `n` CTAs per SM of which `inflight` have work
    const auto step = [&](int n, int64_t inflight) {
        if (!lap) return 0.69 + 0.235 * (n - 1);
        if (n <= 2) return n == 1 ? 0.72 : 1.0;
        const double points = filled * (double)inflight / (double)(sl.sms * 3);
        return 1.33 * n / 3 + (big && points > 0.7 ? 1.5 * (points - 0.7) : 0.0);
    };
    if (tz > nz) tz = (int)nz;
    int64_t best = tz;
    int cap = sl.per_sm;
    double least = 1e300;
    const auto consider = [&](int64_t t) {
        if (t < 1 || t > tz) return;  // the tuned chunk is the longest
        int64_t full = cols * (nz / t), rem = nz % t;
        if (2 * rem > t) {  // all but as long as the others
            full += cols;
            rem = 0;
        }
        const double len = (double)(t + halo);
        for (int c = 1; c <= sl.per_sm; ++c) {
            const int64_t slots = (int64_t)sl.sms * c, waves = (full + slots - 1) / slots;
            double cost = waves == 1 ? len * step(c, full)
                                     : (0.8 * (double)waves + 0.2 * (double)full / (double)slots) * len * step(c, slots);
            if (rem) {
                const int64_t left = cols - (waves * slots - full) * ((t + halo) / (rem + halo));
                if (left > 0)
                    cost += ((double)left / (double)slots + 0.3) * (double)(rem + halo) *
                            step(c, left < slots ? left : slots);
            }
            if (cost < least) {
                least = cost;
                best = t;
                cap = c;
            }
        }
    };
    consider(tz);
    for (int k = 1; k <= 24; ++k) consider((nz + k - 1) / k);
    for (int c = 1; c <= sl.per_sm; ++c)  // few columns: one wave of c CTAs per SM
        if (const int64_t k = (int64_t)sl.sms * c / cols; k > 24) consider((nz + k - 1) / k);
    *ctas = cols * ((nz + best - 1) / best);
    if (cap < sl.per_sm) {
        const size_t room = kSmemPerSm / (size_t)(cap + 1) - kSmemReserved + 16;  // cap + 1 of these do not fit
        if (*smem < room) *smem = room < kSmemPerCta ? room : kSmemPerCta;
    }
    note_planes(best);
    return March{(int)tiles_x, (int)tiles_y, g.nshots, (int)best};
}

template <int R>
cudaError_t fwd_r(const WaveGeo &g, const StarCoef &cf, const float *m, const float *p_cur,
                  const float *p_prev, float *p_next, const float *amp, float *rec, float *lapout,
                  cudaStream_t st, const float *lap_in = nullptr, const AdjArgs *adj = nullptr)
{
    using G = Geom<R, kFwdTX, kFwdTY, kFwdPY, kFwdS>;
    using I = Interior<R, kFwdTX>;
    const int X = g.nx + 2 * R, Y = g.ny + 2 * R, Z = g.nz + 2 * R;
    CUtensorMap mcur, mm, mprev, mctr, mlap;
    if (!encode_tmap_4d(&mcur, p_cur, X, Y, Z, g.nshots, g.py, g.pz, g.ss, G::BX, G::BY, 1) ||
        !encode_tmap_3d(&mm, m, X, Y, Z, g.py, g.pz, I::BXI, kFwdTY, 1) ||
        !encode_tmap_4d(&mprev, p_prev, X, Y, Z, g.nshots, g.py, g.pz, g.ss, I::BXI, kFwdTY, 1) ||
        !encode_tmap_4d(&mctr, p_cur, X, Y, Z, g.nshots, g.py, g.pz, g.ss, I::BXI, kFwdTY, 1))
        return cudaErrorInvalidValue;
    if (lap_in) {
        if (!encode_tmap_4d(&mlap, lap_in, X, Y, Z, g.nshots, g.py, g.pz, g.ss, I::BXI, kFwdTY, 1))
            return cudaErrorInvalidValue;
    } else {
        mlap = mctr;  // not read
    }
    const int mode = adj ? (adj->grad && g.gss == 0 && adj->gbulk ? K_ADJ_BULK : K_ADJ) : lapout ? K_FWD_LAP : K_FWD;
    const auto form = [](auto m) {
        constexpr int M = decltype(m)::value;
        return std::make_pair(wave_fwd_kernel<R, kFwdTX, kFwdTY, kFwdPY, kFwdS, M>,
                              FwdGeom<R, kFwdTX, kFwdTY, kFwdPY, kFwdS, M>::SMEM);
    };
    auto [kern, smem] = mode == K_ADJ_BULK ? form(std::integral_constant<int, K_ADJ_BULK>{})
                        : mode == K_ADJ    ? form(std::integral_constant<int, K_ADJ>{})
                        : mode == K_FWD_LAP ? form(std::integral_constant<int, K_FWD_LAP>{})
                                            : form(std::integral_constant<int, K_FWD>{});
    static SlotCache caches[4];  // per form
    Slots sl;
    cudaError_t e = kernel_slots(caches[mode], reinterpret_cast<const void *>(kern), G::NT, smem, &sl);
    if (e != cudaSuccess) return e;
    const int tiles_x = (g.nx + kFwdTX - 1) / kFwdTX, tiles_y = (g.ny + kFwdTY - 1) / kFwdTY;
    int tz = kFwdTZ;
    if (adj) {
        // The adjoint step on a grid whose tuned chunks fill at most one wave
        // splits z finer, into about three waves, so that the SMs left with
        // one CTA do not idle while the others finish two (2 x 256^3: 219 ->
        // 207 us per step; the forward forms gained nothing).
        const int64_t cols = (int64_t)tiles_x * tiles_y * g.nshots, slots = (int64_t)sl.sms * sl.per_sm;
        if (cols * ((g.nz + tz - 1) / tz) <= slots) {
            const int64_t k = (3 * slots + cols / 2) / cols;  // chunks per column for about three waves
            tz = (int)((g.nz + k - 1) / k);
            if (tz < 2 * R) tz = 2 * R;
        }
    }
    int64_t ctas;
    const March march =
        adj ? plan_march(sl, tiles_x, tiles_y, g.nshots, g.nz, 2 * R, tz, G::NT, &smem, &ctas)
            : plan_forward(sl, tiles_x, tiles_y, g, 2 * R, tz, mode == K_FWD_LAP,
                           (double)g.nx * g.ny / ((double)tiles_x * kFwdTX * (double)tiles_y * kFwdTY), &smem, &ctas);
    if (ctas > INT32_MAX) return cudaErrorInvalidConfiguration;
    const int vec = (R % 4 == 0) && g.py % 4 == 0 && g.pz % 4 == 0 && g.ss % 4 == 0 &&
                    reinterpret_cast<uintptr_t>(p_next) % 16 == 0 && reinterpret_cast<uintptr_t>(lapout) % 16 == 0;
    const AdjArgs aa = adj ? *adj : AdjArgs{nullptr, nullptr, 0, 0};
    return launch_overlapped(kern, dim3((unsigned)ctas), dim3(G::NT), smem, st, mcur, mm, mprev, mctr, mlap, cf, g,
                             p_next, amp, rec, lapout, aa, march, vec, device_error_word());
}

template <int R, bool LAPIN>
cudaError_t adj_r(const WaveGeo &g, const StarCoef &cf, const float *m, const float *lam_cur,
                  float *lam_prev, const float *resid, const float *a_n, double *grad, cudaStream_t st)
{
    using G = Geom<R, kAdjTX, kAdjTY, 1, kAdjS>;
    using A = AdjGeom<R, kAdjTX, kAdjTY, kAdjS>;
    using I = Interior<R, kAdjTX>;
    CUtensorMap ml, mm, ma, m2, m1;
    const int X = g.nx + 2 * R, Y = g.ny + 2 * R, Z = g.nz + 2 * R;
    if (!encode_tmap_4d(&ml, lam_cur, X, Y, Z, g.nshots, g.py, g.pz, g.ss, G::BX, G::BY, 1) ||
        !encode_tmap_3d(&mm, m, X, Y, Z, g.py, g.pz, G::BX, G::BY, 1) ||
        !encode_tmap_4d(&m2, lam_prev, X, Y, Z, g.nshots, g.py, g.pz, g.ss, I::BXI, kAdjTY, 1) ||
        !encode_tmap_4d(&m1, lam_cur, X, Y, Z, g.nshots, g.py, g.pz, g.ss, I::BXI, kAdjTY, 1))
        return cudaErrorInvalidValue;
    if (a_n) {
        // a^n planes with halo, or (LAPIN) interior tiles of L a^n
        if (!encode_tmap_4d(&ma, a_n, X, Y, Z, g.nshots, g.py, g.pz, g.ss, LAPIN ? I::BXI : G::BX,
                            LAPIN ? kAdjTY : G::BY, 1))
            return cudaErrorInvalidValue;
    } else {
        ma = ml;
    }
    auto kern = wave_adj_kernel<R, kAdjTX, kAdjTY, kAdjS, LAPIN>;
    static SlotCache cache;
    Slots sl;
    cudaError_t e = kernel_slots(cache, reinterpret_cast<const void *>(kern), G::NT, A::SMEM, &sl);
    if (e != cudaSuccess) return e;
    const int tiles_x = (g.nx + kAdjTX - 1) / kAdjTX, tiles_y = (g.ny + kAdjTY - 1) / kAdjTY;
    const int tz = z_chunk(sl, (int64_t)tiles_x * tiles_y * g.nshots, g.nz, 2 * R, kAdjTZ, G::NT);
    note_planes(tz);
    const int nzc = (g.nz + tz - 1) / tz;
    const dim3 grid(tiles_x, tiles_y, nzc * g.nshots);
    // 32-byte aligned rows of four doubles: two double2 per thread
    const int gvec = g.nx % 4 == 0 && g.gss % 4 == 0 && reinterpret_cast<uintptr_t>(grad) % 32 == 0;
    kern<<<grid, G::NT, A::SMEM, st>>>(ml, mm, ma, m2, m1, cf, g, lam_prev, resid, grad, a_n ? 1 : 0,
                                       tz, nzc, gvec, device_error_word());
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_wave_fwd(const WaveGeo &g, const float *coeffs, const float *m, const float *p_cur,
                            const float *p_prev, float *p_next, const float *src_amp, float *rec,
                            cudaStream_t st, float *lapout)
{
    StarCoef cf{};
    cf.set(coeffs, 3 * (2 * g.r + 1));
    switch (g.r) {
        case 1: return fwd_r<1>(g, cf, m, p_cur, p_prev, p_next, src_amp, rec, lapout, st);
        case 2: return fwd_r<2>(g, cf, m, p_cur, p_prev, p_next, src_amp, rec, lapout, st);
        case 3: return fwd_r<3>(g, cf, m, p_cur, p_prev, p_next, src_amp, rec, lapout, st);
        case 4: return fwd_r<4>(g, cf, m, p_cur, p_prev, p_next, src_amp, rec, lapout, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_wave_adj_scaled(const WaveGeo &g, const float *coeffs, const float *m, const float *mu_cur,
                                   float *mu_prev, const float *resid, const float *lap_a, double *grad,
                                   cudaStream_t st)
{
    StarCoef cf{};
    cf.set(coeffs, 3 * (2 * g.r + 1));
    const AdjArgs adj{resid, lap_a ? grad : nullptr,
                      g.nx % 4 == 0 && g.gss % 4 == 0 && reinterpret_cast<uintptr_t>(grad) % 32 == 0,
                      g.nx % 2 == 0 && reinterpret_cast<uintptr_t>(grad) % 16 == 0};
    const float *lap = lap_a && grad ? lap_a : nullptr;
    switch (g.r) {
        case 1: return fwd_r<1>(g, cf, m, mu_cur, mu_prev, mu_prev, nullptr, nullptr, nullptr, st, lap, &adj);
        case 2: return fwd_r<2>(g, cf, m, mu_cur, mu_prev, mu_prev, nullptr, nullptr, nullptr, st, lap, &adj);
        case 3: return fwd_r<3>(g, cf, m, mu_cur, mu_prev, mu_prev, nullptr, nullptr, nullptr, st, lap, &adj);
        case 4: return fwd_r<4>(g, cf, m, mu_cur, mu_prev, mu_prev, nullptr, nullptr, nullptr, st, lap, &adj);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_wave_adj(const WaveGeo &g, const float *coeffs, const float *m, const float *lam_cur,
                            float *lam_prev, const float *resid, const float *a_n, double *grad,
                            cudaStream_t st, bool lapin)
{
    StarCoef cf{};
    cf.set(coeffs, 3 * (2 * g.r + 1));
#define MMS_ADJ(R_)                                                                              \
    return lapin ? adj_r<R_, true>(g, cf, m, lam_cur, lam_prev, resid, a_n, grad, st)            \
                 : adj_r<R_, false>(g, cf, m, lam_cur, lam_prev, resid, a_n, grad, st);
    switch (g.r) {
        case 1: MMS_ADJ(1)
        case 2: MMS_ADJ(2)
        case 3: MMS_ADJ(3)
        case 4: MMS_ADJ(4)
        default: return cudaErrorInvalidValue;
    }
#undef MMS_ADJ
}

cudaError_t launch_model_from_velocity(const WaveGeo &g, const float *v, float *m, float dt, float h,
                                       cudaStream_t st)
{
    const float s = (dt * dt) / (h * h);
    launch_rows(g.nx + 2 * g.r, (int64_t)(g.ny + 2 * g.r) * (g.nz + 2 * g.r), [&](auto t, int blocks, dim3 block) {
        model_kernel<decltype(t)::value><<<blocks, block, 0, st>>>(g, v, m, s);
    });
    return cudaGetLastError();
}

cudaError_t launch_grad_to_velocity(const double *gm, const float *v, double *gv, int64_t n, float dt,
                                    float h, cudaStream_t st)
{
    const double s = ((double)dt * dt) / ((double)h * h);
    chain_kernel<<<152 * 8, 256, 0, st>>>(gm, v, gv, n, 2.0 * s);
    return cudaGetLastError();
}

cudaError_t launch_grad_divide_m(const WaveGeo &g, const float *m, double *grad, cudaStream_t st)
{
    launch_rows(g.nx, (int64_t)g.ny * g.nz, [&](auto t, int blocks, dim3 block) {
        divide_m_kernel<decltype(t)::value><<<blocks, block, 0, st>>>(g, m, grad);
    });
    return cudaGetLastError();
}

cudaError_t launch_wait_selftest(unsigned long long limit_ns, cudaStream_t st)
{
    wait_selftest_kernel<<<1, 32, 0, st>>>(limit_ns, device_error_word());
    return cudaGetLastError();
}

cudaError_t launch_sum_f64(const double *slices, int nslices, int64_t stride, int64_t n, double *out,
                           cudaStream_t st)
{
    sum_kernel<<<152 * 8, 256, 0, st>>>(slices, nslices, stride, n, out);
    return cudaGetLastError();
}

cudaError_t launch_dot_f64(const float *a, const float *b, int64_t n, double *res, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(res, 0, sizeof(double), st);
    if (e != cudaSuccess) return e;
    dot_kernel<<<152 * 4, 256, 0, st>>>(a, b, n, res);
    return cudaGetLastError();
}

}  // namespace mms
