// common.cuh -- shared internals of the sm_103a stencil library: launch
// argument structs, the device error word, and inline-PTX helpers for
// mbarriers, TMA bulk-tensor copies and the global timer.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "../../include/mms.h"

namespace mms {

// Largest radius and coefficient counts (star: 3*(2r+1), box: (2r+1)^3).
constexpr int kMaxR = 4;
constexpr int kMaxStar = 3 * (2 * kMaxR + 1);
constexpr int kMaxBox = (2 * kMaxR + 1) * (2 * kMaxR + 1) * (2 * kMaxR + 1);

// Coefficients travel as kernel parameters (constant bank), so every FMA
// reads its weight as a uniform constant operand.  The star updates work on
// pairs of points (tile.cuh), so their weights come as pairs (c, c).
struct W2 {
    float lo, hi;
};
struct StarCoef {
    W2 c[kMaxStar];
    void set(const float *w, int n)
    {
        for (int i = 0; i < n; ++i) c[i] = W2{w[i], w[i]};
    }
};
struct BoxCoef { float c[kMaxBox]; };

// Device error word bits (read by mms_check_device).
constexpr unsigned kErrTimeout = 1u;
constexpr unsigned kErrIndex = 2u;

// Bound of every device-side wait (nanoseconds of %globaltimer).
constexpr unsigned long long kWaitLimitNs = 2000000000ull;

// One sweep, as validated by the ABI layer.
struct Sweep {
    int shape, r;
    int64_t nx, ny, nz;
    const float *in;
    int64_t ipy, ipz;
    float *out;
    int64_t opy, opz;
    const float *coeffs;  // host
    int variant;
    cudaStream_t stream;
};

// Host launchers (each returns a CUDA error code; validation happens above).
cudaError_t launch_naive(const Sweep &s);
cudaError_t launch_star_cc(const Sweep &s, const CUtensorMap &tmap, int variant);
cudaError_t launch_box_cc(const Sweep &s, const CUtensorMap &tmap, int variant);
int star_cc_variants();
int box_cc_variants();
// TMA box (x extent, y extent) that variant v of the CUDA-core sweeps loads.
void star_cc_box(int r, int v, int *bx, int *by);
void box_cc_box(int r, int v, int *bx, int *by);

// Planar (2D) CUDA-core sweeps (sweep_2d.cu).
cudaError_t launch_plane_cc(const Sweep &s, const CUtensorMap &tmap, int variant);
int plane_cc_variants();
void plane_cc_box(int r, int v, int *bx, int *by);

// Sweeps of inputs TMA cannot read (sweep_any.cu), and whether the grid is one they take.
bool any_pitch_ok(const Sweep &s);
cudaError_t launch_any(const Sweep &s);

// Planar shapes have no z halo.
__host__ __device__ constexpr bool is_planar(int shape) { return shape == MMS_STAR2D || shape == MMS_BOX2D; }

// Tensor-core banded sweeps (band_tc.cu).
int band_tc_supported(int shape, int r, int path);
// The star's two-pass variants run a planar tensor-core pass into `scratch`
// (nx*ny*nz floats, dense; band_tc_scratch_bytes of the sweep with its
// resolved variant in Sweep::variant) followed by a CUDA-core z pass; every
// other variant needs no scratch.
cudaError_t launch_band_tc(const Sweep &s, int path, const CUtensorMap &tmap, int variant, float *scratch);
size_t band_tc_scratch_bytes(const Sweep &s);
void band_tc_box(int shape, int r, int path, int v, int *bx, int *by, int *bz, int *swz);
int band_tc_variants(int shape, int r, int path);

// Error word helpers (wave.cu owns the symbol).
unsigned *device_error_word();

// Encodes a 3D FP32 tensor map over a padded grid (x extent X, pitches in
// elements) with box (bx, by, bz); returns false when the driver refuses.
bool encode_tmap_3d(CUtensorMap *map, const float *base, int64_t X, int64_t Y, int64_t Z,
                    int64_t py, int64_t pz, int bx, int by, int bz, bool swizzle128 = false);
// The same over nw stacked grids `pw` elements apart, box depth 1 in w.
bool encode_tmap_4d(CUtensorMap *map, const float *base, int64_t X, int64_t Y, int64_t Z,
                    int64_t W, int64_t py, int64_t pz, int64_t pw, int bx, int by, int bz);

// Shared memory of an SM, what the system keeps of it per CTA, and the most
// a CTA may ask for (sm_103).
constexpr size_t kSmemPerSm = 228 * 1024, kSmemReserved = 1024, kSmemPerCta = 227 * 1024;

// Id of the calling thread's current context, 0 if there is none yet.  A
// kernel's attributes and the address of a __device__ variable belong to a
// context, not to a device: what is remembered of them is kept by this id,
// which no later context has again (not the device's own after a reset either).
unsigned long long context_id();

// What was worked out last in each of a few contexts (the oldest gives way).
template <typename T>
class PerContext {
public:
    bool find(unsigned long long ctx, T *out)
    {
        std::lock_guard<std::mutex> lk(mu_);
        for (const Entry &e : e_)
            if (ctx != 0 && e.ctx == ctx) {
                *out = e.v;
                return true;
            }
        return false;
    }
    void keep(unsigned long long ctx, const T &v)
    {
        if (ctx == 0) return;
        std::lock_guard<std::mutex> lk(mu_);
        for (const Entry &e : e_)
            if (e.ctx == ctx) return;  // another thread was first
        e_[next_] = Entry{ctx, v};
        next_ = (next_ + 1) % kContexts;
    }

private:
    static constexpr int kContexts = 16;
    struct Entry {
        unsigned long long ctx = 0;
        T v{};
    };
    std::mutex mu_;
    Entry e_[kContexts];
    int next_ = 0;
};

// What one kernel instance can keep resident on the current device, asked once
// per context (with its dynamic shared-memory limit raised to the most there
// is): the SM count and the CTAs of `threads` threads and `smem` bytes one SM
// holds.  One static cache per kernel instance and size; concurrent first
// calls compute the same values.
struct Slots { int sms = 0, per_sm = 0; };
using SlotCache = PerContext<Slots>;
cudaError_t kernel_slots(SlotCache &cache, const void *kern, int threads, size_t smem, Slots *out);

// Planes per z chunk of a kernel whose CTAs each march one chunk of one of
// `cols` columns (reading `halo` extra planes), given the kernel's tuned chunk
// `tz`.  A grid whose tuned chunks keep every SM busy keeps them: it is bound
// by memory, and finer chunks only read more halo planes (box r = 1, 512^3:
// 172 us, 196 us in finer ones).  Otherwise the chunk is the one of least
// modelled time among those that fill one wave to 1, 2, ... CTAs per SM or run
// in one and a half to four waves: the VTI step on 2 x 250 x 230 x 190, 232
// columns on 456 CTA slots, takes 285 us as one chunk each, 171 us in five.
// Against the tuned chunk everywhere, over 36 random shapes per kernel (mean
// and worst time, kernels that changed in nothing else): star r = 1 0.54, 1.04;
// r = 2 0.53, 1.01; box r = 1 0.45, 1.04; r = 2 0.57, 1.00; planar star r = 2
// 0.88, 1.00; planar box r = 3 0.91, 1.00.  VTI and TTI, their paired updates
// included: 0.42, 0.98 and 0.64, 0.98.
int z_chunk(const Slots &sl, int64_t cols, int64_t nz, int halo, int tz, int threads);

// How a kernel's CTAs divide the columns they march along z: CTA b marches
// chunk zc (tz planes) of one x, y tile of one shot, the shots fastest, then
// x, y, chunks -- the shots of a tile read the same medium, so next to each
// other they read it from L2 (acoustic step, 8 x 512^3, shots slowest: 3.00
// ms, fastest: 2.83 ms).
struct March {
    int tiles_x, tiles_y, nshots, tz;
};
// The march of a launch of tuned chunk `tz`, and its grid size.  *smem, the
// kernel's dynamic shared memory, is raised where the grid is one wave of
// fewer CTAs than an SM holds, to what lets no SM take more than its share:
// the scheduler doubles up on some SMs while others run one CTA (232 CTAs of
// the VTI step on 152 SMs: one to three per SM).
March plan_march(const Slots &sl, int64_t tiles_x, int64_t tiles_y, int nshots, int64_t nz, int halo, int tz,
                 int threads, size_t *smem, int64_t *ctas);

// Keeps the planes (row blocks) per CTA of a launch for mms_last_planes.
void note_planes(int64_t planes);

// The tile, shot and z chunk of this CTA.
struct Leg {
    int tx, ty, shot, zc;
};
__device__ __forceinline__ Leg leg_of(const March &m)
{
    unsigned b = blockIdx.x;
    Leg g;
    g.shot = b % m.nshots;
    b /= m.nshots;
    g.tx = b % m.tiles_x;
    b /= m.tiles_x;
    g.ty = b % m.tiles_y;
    g.zc = b / m.tiles_y;
    return g;
}

}  // namespace mms

// ------------------------------------------------------------ PTX helpers
namespace ptx {

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// One lane of the (converged, full) warp is elected; true in that lane.
__device__ __forceinline__ bool elect_one()
{
    uint32_t pred = 0;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(pred));
    return pred != 0;
}

__device__ __forceinline__ unsigned long long globaltimer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
}

__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Waits for the phase with the given parity to complete; gives up after
// limit_ns (kWaitLimitNs by default), sets the timeout bit of the device
// error word and returns false.  Never traps.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity, unsigned *err,
                                                  unsigned long long limit_ns = mms::kWaitLimitNs)
{
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = globaltimer();
    for (uint32_t it = 0;; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 255u) == 255u && globaltimer() - t0 > limit_ns) {
            if (err) atomicOr(err, mms::kErrTimeout);
            return false;
        }
    }
}

// TMA: 3D tiled load global -> shared, completion counted on `bar`.
__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, int x, int y, int z,
                                            uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}

// TMA: 4D tiled load global -> shared (x, y, z, w coordinates).
__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *map, int x, int y, int z,
                                            int w, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void prefetch_tmap(const CUtensorMap *map)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

}  // namespace ptx
