// sweep_f64.cu -- FP64 star and box sweeps (3D and the planar 2D shapes).
//
// GB300's FP64 pipe issues about two FMAs per clock per SM, 1/64 of the
// FP32 rate, so an FP64 sweep is bound by that pipe long before HBM (star
// r = 4: 25 FMAs per 16 bytes moved).  The kernel therefore spends nothing
// on staging: one thread per output point, neighbours through the read-only
// L1 path (each input is reused from L1/L2 by the threads around it), and
// the FMA count cut to the minimum -- the star's three centre weights are
// folded into one, so a radius-r star costs 6r + 1 FMAs and a box (2r+1)^3.
#include "common.cuh"

namespace mms {

namespace {

struct F64Coef { double c[(2 * kMaxR + 1) * (2 * kMaxR + 1) * (2 * kMaxR + 1)]; };
struct F64Star {
    double c[kMaxStar], centre;
};

// The star, one point per thread.  Bound by the FP64 pipe, which does nothing
// but the 6R + 1 FMAs of a point: the centre weight is folded on the host (two
// FP64 adds per point before, 256^3 r = 4: 864 -> 802 us), and the weights sit
// in registers, for FMAs with a constant-bank operand run at five sixths of the
// pipe's rate whatever the tile (802 -> 698 us; the pipe's 25 FMAs take 667).
// Small CTAs spread evenly, and with one point per thread small grids fill the
// SMs (four points of a z column per thread, their z neighbours loaded once:
// r = 4, 256^3 715 us, 31 x 33 x 35 5.5 against 3.7, r = 3, 129 x 33 x 65 20.9
// against 13.7).
constexpr int kStarBY = 2;

template <int R>
__global__ void __launch_bounds__(32 * kStarBY)
    f64_star_kernel(const __grid_constant__ F64Star cf, const double *__restrict__ in, int64_t ipy, int64_t ipz,
                    double *__restrict__ out, int64_t opy, int64_t opz, int nx, int ny, int nz)
{
    constexpr int W = 2 * R + 1;
    // by way of shared memory, or the compiler takes them from the constant bank
    __shared__ double sw[3 * W + 1];
    for (int i = threadIdx.y * 32 + threadIdx.x; i <= 3 * W; i += 32 * kStarBY) sw[i] = i < 3 * W ? cf.c[i] : cf.centre;
    __syncthreads();
    double w[3 * W];
#pragma unroll
    for (int i = 0; i < 3 * W; ++i) w[i] = sw[i];
    const double centre = sw[3 * W];
    const int x = blockIdx.x * 32 + threadIdx.x;
    if (x >= nx) return;
    // y and z stride over the grid's extents (launch dims are capped at 65535)
    for (int z = blockIdx.z; z < nz; z += gridDim.z)
        for (int y = blockIdx.y * kStarBY + threadIdx.y; y < ny; y += gridDim.y * kStarBY) {
            const double *c = in + (int64_t)(z + R) * ipz + (int64_t)(y + R) * ipy + (x + R);
            double a = centre * __ldg(c);
#pragma unroll
            for (int d = 1; d <= R; ++d) {
                a = fma(w[R + d], __ldg(c + d), a);
                a = fma(w[R - d], __ldg(c - d), a);
                a = fma(w[W + R + d], __ldg(c + d * ipy), a);
                a = fma(w[W + R - d], __ldg(c - d * ipy), a);
                a = fma(w[2 * W + R + d], __ldg(c + d * ipz), a);
                a = fma(w[2 * W + R - d], __ldg(c - d * ipz), a);
            }
            out[(int64_t)z * opz + (int64_t)y * opy + x] = a;
        }
}

template <int SHAPE, int R>
__global__ void __launch_bounds__(256)
    f64_kernel(const __grid_constant__ F64Coef cf, const double *__restrict__ in, int64_t ipy, int64_t ipz,
               double *__restrict__ out, int64_t opy, int64_t opz, int nx, int ny, int nz)
{
    constexpr int W = 2 * R + 1;
    const int x = blockIdx.x * 32 + threadIdx.x;
    if (x >= nx) return;
    constexpr bool planar = SHAPE == MMS_STAR2D || SHAPE == MMS_BOX2D;
    // y and z stride over the grid's extents (launch dims are capped at 65535)
    for (int z = blockIdx.z; z < nz; z += gridDim.z)
        for (int y = blockIdx.y * 8 + threadIdx.y; y < ny; y += gridDim.y * 8) {
            const double *c0 = in + (int64_t)(z + (planar ? 0 : R)) * ipz + (int64_t)(y + R) * ipy + (x + R);
            double acc;
            if constexpr (SHAPE == MMS_STAR2D) {
                acc = (cf.c[R] + cf.c[W + R]) * __ldg(c0);
#pragma unroll
                for (int d = 1; d <= R; ++d) {
                    acc = fma(cf.c[R + d], __ldg(c0 + d), acc);
                    acc = fma(cf.c[R - d], __ldg(c0 - d), acc);
                    acc = fma(cf.c[W + R + d], __ldg(c0 + d * ipy), acc);
                    acc = fma(cf.c[W + R - d], __ldg(c0 - d * ipy), acc);
                }
            } else if constexpr (SHAPE == MMS_BOX2D) {
                acc = 0.0;
#pragma unroll
                for (int dy = -R; dy <= R; ++dy)
#pragma unroll
                    for (int dx = -R; dx <= R; ++dx)
                        acc = fma(cf.c[(dy + R) * W + dx + R], __ldg(c0 + dy * ipy + dx), acc);
            } else {
                acc = 0.0;
#pragma unroll 1
                for (int dz = -R; dz <= R; ++dz)
#pragma unroll
                    for (int dy = -R; dy <= R; ++dy)
#pragma unroll
                        for (int dx = -R; dx <= R; ++dx)
                            acc = fma(cf.c[((dz + R) * W + dy + R) * W + dx + R], __ldg(c0 + dz * ipz + dy * ipy + dx), acc);
            }
            out[(int64_t)z * opz + (int64_t)y * opy + x] = acc;
        }
}

cudaError_t f64_star(int r, const double *w, const double *in, int64_t ipy, int64_t ipz, double *out, int64_t opy,
                     int64_t opz, int nx, int ny, int nz, cudaStream_t st)
{
    F64Star cf{};
    const int W = 2 * r + 1;
    for (int i = 0; i < 3 * W; ++i) cf.c[i] = w[i];
    cf.centre = w[r] + w[W + r] + w[2 * W + r];
    const dim3 block(32, kStarBY), grid((nx + 31) / 32, min((ny + kStarBY - 1) / kStarBY, 65535), min(nz, 65535));
    switch (r) {
        case 1: f64_star_kernel<1><<<grid, block, 0, st>>>(cf, in, ipy, ipz, out, opy, opz, nx, ny, nz); break;
        case 2: f64_star_kernel<2><<<grid, block, 0, st>>>(cf, in, ipy, ipz, out, opy, opz, nx, ny, nz); break;
        case 3: f64_star_kernel<3><<<grid, block, 0, st>>>(cf, in, ipy, ipz, out, opy, opz, nx, ny, nz); break;
        case 4: f64_star_kernel<4><<<grid, block, 0, st>>>(cf, in, ipy, ipz, out, opy, opz, nx, ny, nz); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <int SHAPE>
cudaError_t f64_shape(int r, const F64Coef &cf, const double *in, int64_t ipy, int64_t ipz, double *out,
                      int64_t opy, int64_t opz, int nx, int ny, int nz, cudaStream_t st)
{
    const dim3 block(32, 8), grid((nx + 31) / 32, min((ny + 7) / 8, 65535), min(nz, 65535));
    switch (r) {
        case 1: f64_kernel<SHAPE, 1><<<grid, block, 0, st>>>(cf, in, ipy, ipz, out, opy, opz, nx, ny, nz); break;
        case 2: f64_kernel<SHAPE, 2><<<grid, block, 0, st>>>(cf, in, ipy, ipz, out, opy, opz, nx, ny, nz); break;
        case 3: f64_kernel<SHAPE, 3><<<grid, block, 0, st>>>(cf, in, ipy, ipz, out, opy, opz, nx, ny, nz); break;
        case 4: f64_kernel<SHAPE, 4><<<grid, block, 0, st>>>(cf, in, ipy, ipz, out, opy, opz, nx, ny, nz); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_f64(int shape, int r, const double *coeffs, int ncoef, const double *in, int64_t ipy, int64_t ipz,
                       double *out, int64_t opy, int64_t opz, int64_t nx, int64_t ny, int64_t nz, cudaStream_t st)
{
    const int X = (int)nx, Y = (int)ny, Z = (int)nz;
    if (shape == MMS_STAR) return f64_star(r, coeffs, in, ipy, ipz, out, opy, opz, X, Y, Z, st);
    F64Coef cf{};
    for (int i = 0; i < ncoef; ++i) cf.c[i] = coeffs[i];
    switch (shape) {
        case MMS_BOX: return f64_shape<MMS_BOX>(r, cf, in, ipy, ipz, out, opy, opz, X, Y, Z, st);
        case MMS_STAR2D: return f64_shape<MMS_STAR2D>(r, cf, in, ipy, ipz, out, opy, opz, X, Y, Z, st);
        case MMS_BOX2D: return f64_shape<MMS_BOX2D>(r, cf, in, ipy, ipz, out, opy, opz, X, Y, Z, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace mms
