// FP64 reductions (Section 4.1 plate Nusselt numbers, the divergence check of
// Section 3.2, the CFL limit), the upscale integration and dtype conversion
// (volume moments and profiles: mr_diag.cu).  Each block reduces with warp
// shuffles into one FP64 partial, and the partials are combined in a fixed order,
// so every result is deterministic.
#include <math.h>

#include "mr_internal.cuh"

namespace mr {
namespace {

constexpr int kRedThreads = 256;

__device__ __forceinline__ double warp_sum(double v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_max(double v)
{
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
    return v;
}

// Block reduction of NV values per thread (sum or max); thread 0 writes them.
template <int NV, bool MAX>
__device__ void block_reduce_store(double (&v)[NV], double* out)
{
    __shared__ double sh[NV][kRedThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int q = 0; q < NV; ++q) {
        double r = MAX ? warp_max(v[q]) : warp_sum(v[q]);
        if (lane == 0) sh[q][wid] = r;
    }
    __syncthreads();
    if (wid == 0) {
        for (int q = 0; q < NV; ++q) {
            double r = (lane < kRedThreads / 32) ? sh[q][lane] : (MAX ? 0.0 : 0.0);
            r = MAX ? warp_max(r) : warp_sum(r);
            if (lane == 0) out[q] = r;
        }
    }
}

// Plate Nusselt numbers: every block sums a fixed slice of both plates,
// sum (T_bottom - T) and sum (T - T_top), into two FP64 partials; the block
// that finishes last (an atomic count, nothing waits) adds the partials --
// thread t the partials t, t + 256, ..., then the block's fixed reduction tree,
// so the order of the additions never changes -- divides by the centre
// distance and the cell count, and resets the count for the next launch.
template <typename P>
__global__ void __launch_bounds__(256) k_plate_nu(Grid<P> g, const P* __restrict__ T, double zb, double zt,
                                                  double inv_plane, double* __restrict__ partials,
                                                  unsigned* __restrict__ count, double* __restrict__ out2)
{
    const size_t plane = (size_t)g.Nx * g.Ny;
    const P* top = T + (size_t)(g.Nz - 1) * plane;
    double v[2] = {0.0, 0.0};
    for (size_t m = (size_t)blockIdx.x * blockDim.x + threadIdx.x; m < plane; m += (size_t)gridDim.x * blockDim.x) {
        v[0] += 0.5 - (double)T[m];
        v[1] += (double)top[m] + 0.5;
    }
    block_reduce_store<2, false>(v, partials + 2 * blockIdx.x);
    __shared__ bool last;
    if (threadIdx.x == 0) {
        __threadfence();                     // this block's partials before its count
        last = atomicAdd(count, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double s2[2] = {0.0, 0.0};
    for (unsigned q = threadIdx.x; q < gridDim.x; q += blockDim.x) {
        s2[0] += __ldcg(partials + 2 * q);
        s2[1] += __ldcg(partials + 2 * q + 1);
    }
    __shared__ double tot[2];
    block_reduce_store<2, false>(s2, tot);
    if (threadIdx.x == 0) {                  // the thread that wrote tot
        out2[0] = tot[0] / zb * inv_plane;
        out2[1] = tot[1] / zt * inv_plane;
        *count = 0u;
    }
}

// FP64 values from mapped pinned host memory (read by the SMs over the host
// link) into the FP64 device copy and, where d32 is given, its FP32 rounding.
__global__ void k_fetch_f64(const double* __restrict__ src, double* __restrict__ d64, float* __restrict__ d32,
                            size_t n)
{
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    const size_t n2 = n / 2;
    const double2* s2 = reinterpret_cast<const double2*>(src);
    double2* o2 = reinterpret_cast<double2*>(d64);
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < n2; t += stride) {
        const double2 v = s2[t];
        o2[t] = v;
        if (d32) reinterpret_cast<float2*>(d32)[t] = make_float2((float)v.x, (float)v.y);
    }
    if ((n & 1) && blockIdx.x == 0 && threadIdx.x == 0) {
        d64[n - 1] = src[n - 1];
        if (d32) d32[n - 1] = (float)src[n - 1];
    }
}

// Max |divergence| of the dense refined faces (outward flux sum / volume).
// Blocks stride over dense rows (j, k), threads over x.
template <typename P>
__global__ void __launch_bounds__(kRedThreads) k_maxdiv(Grid<P> g, const P* __restrict__ Us,
                                                        const P* __restrict__ Vs, const P* __restrict__ Ws,
                                                        double* __restrict__ partials)
{
    const size_t plane = (size_t)g.Nx * g.Ny;
    const int rows = g.Ny * g.Nz;
    double v[1] = {0.0};
    for (int row = blockIdx.x; row < rows; row += gridDim.x) {
        const int k = row / g.Ny, j = row - k * g.Ny;
        const int fn = g.walls ? j + 1 : (j + 1 == g.Ny ? 0 : j + 1);
        const P* ur = Us + ((size_t)k * g.Ny + j) * g.ufx;
        const P* vs = Vs + ((size_t)k * g.vfy + j) * g.Nx;
        const P* vn = Vs + ((size_t)k * g.vfy + fn) * g.Nx;
        const P* wb = Ws + (size_t)row * g.Nx;
        const P* wt = wb + plane;
        const double idz = (double)g.inv_dz[k];
        for (int i = threadIdx.x; i < g.Nx; i += blockDim.x) {
            const int fe = g.walls ? i + 1 : (i + 1 == g.Nx ? 0 : i + 1);
            const double d = ((double)ur[fe] - (double)ur[i]) * (double)g.inv_dx +
                             ((double)vn[i] - (double)vs[i]) * (double)g.inv_dy + ((double)wt[i] - (double)wb[i]) * idz;
            v[0] = fmax(v[0], fabs(d));
        }
    }
    block_reduce_store<1, true>(v, partials + blockIdx.x);
}

// CFL rate max(|u|)/dx + max(|v|)/dy + max(|w|)/dz over the cell's faces, in
// precision P (|.| and max are exact; the rate is one sum of three products).
template <typename P>
__global__ void __launch_bounds__(kRedThreads) k_cfl(Grid<P> g, const P* __restrict__ Us,
                                                     const P* __restrict__ Vs, const P* __restrict__ Ws,
                                                     double* __restrict__ partials)
{
    const size_t plane = (size_t)g.Nx * g.Ny;
    const int rows = g.Ny * g.Nz;
    P m = 0;
    for (int row = blockIdx.x; row < rows; row += gridDim.x) {
        const int k = row / g.Ny, j = row - k * g.Ny;
        const int fn = g.walls ? j + 1 : (j + 1 == g.Ny ? 0 : j + 1);
        const P* ur = Us + ((size_t)k * g.Ny + j) * g.ufx;
        const P* vs = Vs + ((size_t)k * g.vfy + j) * g.Nx;
        const P* vn = Vs + ((size_t)k * g.vfy + fn) * g.Nx;
        const P* wb = Ws + (size_t)row * g.Nx;
        const P* wt = wb + plane;
        const P idz = g.inv_dz[k];
        for (int i = threadIdx.x; i < g.Nx; i += blockDim.x) {
            const int fe = g.walls ? i + 1 : (i + 1 == g.Nx ? 0 : i + 1);
            const P u = fmax(fabs(ur[i]), fabs(ur[fe]));
            const P vv = fmax(fabs(vs[i]), fabs(vn[i]));
            const P w = fmax(fabs(wb[i]), fabs(wt[i]));
            m = fmax(m, u * g.inv_dx + vv * g.inv_dy + w * idz);
        }
    }
    double v[1] = {(double)m};
    block_reduce_store<1, true>(v, partials + blockIdx.x);
}

// VEC contiguous values as one load (1, 2 or 4 of them; aligned to their size).
template <typename P, int VEC>
struct alignas(sizeof(P) * VEC) Pack {
    P v[VEC];
};

// Upscale integration (Section 3.3): volume average over every coarse cell, the
// sum over each dense layer in the working precision (GB300's FP64 pipe is 1/64
// of its FP32 rate), weighted in FP64 by upw[k] = dz_k / (mx my sum of the slab's
// dz): two FP64 operations per cell and layer.  A thread owns a coarse cell and
// reads its rows VEC values at a time.  FP32, 64 x 64 x 48 coarse cells at M = 4:
// 10.4 us; 19.5 us with scalar loads, the weights' sum and a division per cell.
template <typename P, int VEC, int M>
__global__ void __launch_bounds__(128) k_upscale(Grid<P> g, const P* __restrict__ T, const double* __restrict__ upw,
                                                 double* __restrict__ Tc)
{
    const size_t n = (size_t)g.nz * g.ny * g.nx;
    const int mx = M ? M : g.mx, my = M ? M : g.my, mz = M ? M : g.mz;
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x) {
        const int I = (int)(t % g.nx), J = (int)((t / g.nx) % g.ny), K = (int)(t / ((size_t)g.nx * g.ny));
        double s = 0.0;
#pragma unroll
        for (int c = 0; c < mz; ++c) {
            const int k = K * mz + c;
            P r = P(0);
            const P* row = T + ((size_t)k * g.Ny + (size_t)J * my) * g.Nx + (size_t)I * mx;
#pragma unroll
            for (int j = 0; j < my; ++j)
#pragma unroll
                for (int i = 0; i < mx; i += VEC) {
                    const Pack<P, VEC> q = *reinterpret_cast<const Pack<P, VEC>*>(row + (size_t)j * g.Nx + i);
#pragma unroll
                    for (int e = 0; e < VEC; ++e) r += q.v[e];
                }
            s = fma((double)r, upw[k], s);
        }
        Tc[t] = s;
    }
}

template <typename S, typename D>
__global__ void k_convert(const S* __restrict__ src, D* __restrict__ dst, size_t n)
{
    for (size_t m = (size_t)blockIdx.x * blockDim.x + threadIdx.x; m < n; m += (size_t)gridDim.x * blockDim.x)
        dst[m] = (D)src[m];
}

}  // namespace

template <typename P>
cudaError_t launch_plate_nu(const Grid<P>& g, const P* T, const double* zb_zt, double* work, double* out2,
                            cudaStream_t st)
{
    // work holds 3 + 2 * kPlateBlocks doubles: two for a caller's result, the block
    // count (zero between launches) and the partials
    k_plate_nu<P><<<kPlateBlocks, 256, 0, st>>>(g, T, zb_zt[0], zb_zt[1], 1.0 / ((double)g.Nx * g.Ny), work + 3,
                                                reinterpret_cast<unsigned*>(work + 2), out2);
    return cudaGetLastError();
}

template <typename P>
cudaError_t launch_upscale(const Grid<P>& g, const P* T, const double* upw, double* Tc, cudaStream_t st)
{
    const size_t n = (size_t)g.nz * g.ny * g.nx, want = (n + 127) / 128;
    const unsigned blocks = (unsigned)(want < 152 * 16 ? want : 152 * 16);
    const bool cube = g.mx == g.my && g.my == g.mz;       // unrolled: every load of a cell in flight
    // rows of a coarse cell start at multiples of mx: whole packs where mx allows
    // (16 bytes at most; the scalar's buffers are 256-byte aligned)
    if (cube && g.mx == 4) k_upscale<P, sizeof(P) == 4 ? 4 : 2, 4><<<blocks, 128, 0, st>>>(g, T, upw, Tc);
    else if (cube && g.mx == 2) k_upscale<P, 2, 2><<<blocks, 128, 0, st>>>(g, T, upw, Tc);
    else if (g.mx % 2 == 0) k_upscale<P, 2, 0><<<blocks, 128, 0, st>>>(g, T, upw, Tc);
    else k_upscale<P, 1, 0><<<blocks, 128, 0, st>>>(g, T, upw, Tc);
    return cudaGetLastError();
}

template <typename P>
cudaError_t launch_maxdiv(const Grid<P>& g, const P* Us, const P* Vs, const P* Ws, double* partials, int blocks,
                          cudaStream_t st)
{
    k_maxdiv<P><<<blocks, kRedThreads, 0, st>>>(g, Us, Vs, Ws, partials);
    return cudaGetLastError();
}

template <typename P>
cudaError_t launch_cfl(const Grid<P>& g, const P* Us, const P* Vs, const P* Ws, double* partials, int blocks,
                       cudaStream_t st)
{
    k_cfl<P><<<blocks, kRedThreads, 0, st>>>(g, Us, Vs, Ws, partials);
    return cudaGetLastError();
}

// src/dst dtypes: MR_F64 or MR_F32.  P is unused (kept for a uniform launcher signature).
template <typename P>
cudaError_t launch_convert(const void* src, int sd, void* dst, int dd, size_t n, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    const int threads = 256;
    size_t want = (n + threads - 1) / threads;
    const unsigned blocks = (unsigned)(want < 152 * 16 ? want : 152 * 16);
    if (sd == MR_F64 && dd == MR_F32)
        k_convert<double, float><<<blocks, threads, 0, st>>>((const double*)src, (float*)dst, n);
    else if (sd == MR_F32 && dd == MR_F64)
        k_convert<float, double><<<blocks, threads, 0, st>>>((const float*)src, (double*)dst, n);
    else if (sd == MR_F64 && dd == MR_F64)
        return cudaMemcpyAsync(dst, src, n * 8, cudaMemcpyDeviceToDevice, st);
    else
        return cudaMemcpyAsync(dst, src, n * 4, cudaMemcpyDeviceToDevice, st);
    return cudaGetLastError();
}

#define MR_INST(P)                                                                                           \
    template cudaError_t launch_plate_nu<P>(const Grid<P>&, const P*, const double*, double*, double*,              \
                                             cudaStream_t);                                                  \
    template cudaError_t launch_maxdiv<P>(const Grid<P>&, const P*, const P*, const P*, double*, int,          \
                                          cudaStream_t);                                                     \
    template cudaError_t launch_cfl<P>(const Grid<P>&, const P*, const P*, const P*, double*, int, cudaStream_t);    \
    template cudaError_t launch_upscale<P>(const Grid<P>&, const P*, const double*, double*, cudaStream_t);
MR_INST(double)
MR_INST(float)
#undef MR_INST
template cudaError_t launch_convert<double>(const void*, int, void*, int, size_t, cudaStream_t);

cudaError_t launch_fetch_f64(const double* src, double* d64, float* d32, size_t n, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    // 16-byte alignment for the pair loads and stores
    if ((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(d64)) & 15 ||
        reinterpret_cast<uintptr_t>(d32) & 7)
        return cudaErrorInvalidValue;
    k_fetch_f64<<<152 * 8, 256, 0, st>>>(src, d64, d32, n);
    return cudaGetLastError();
}

}  // namespace mr
