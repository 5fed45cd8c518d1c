// Volume moments and heat-flux profiles (Section 4.1) in one pass over the
// scalar each, to FP64 accuracy.
//
// GB300 issues FP64 arithmetic, and the conversion of an FP32 value to FP64, at
// 1/64 of its FP32 rate, so sums over an FP32 scalar are kept as unevaluated
// pairs of FP32 values (Sum<float>): the rounding error of every addition,
// product and difference is itself an FP32 value, found by the error-free
// transformations of Dekker and Knuth and added up beside the sum (the
// compensated dot product of Ogita, Rump and Oishi, 2005), which then is as good
// as if it had been formed with 48 bits.  A pair becomes FP64 once per thread's
// share of a block (at most kShare cells).  The transformations need room below
// and above the values: a block whose values leave that range, or are not
// finite, repeats its share in FP64 (Sum<double>), as FP64 scalars do anyway.
#include <math.h>

#include "mr_internal.cuh"

namespace mr {
namespace {

constexpr int kThreads = 256;
constexpr int kShare = 64;           // cells per thread of a block

template <typename A>
struct Sum;
template <>
struct Sum<double> {
    double s = 0.0;
    __device__ __forceinline__ void prod(double a, double b) { s = fma(a, b, s); }
    __device__ __forceinline__ void diff(double a, double b, Sum<double>& sq)
    {
        const double d = a - b;
        s += d;
        sq.s = fma(d, d, sq.s);
    }
    __device__ __forceinline__ void sqdiff(double a, double b)
    {
        const double d = a - b;
        s = fma(d, d, s);
    }
    // the warp's sum, in lane 0
    __device__ __forceinline__ void warp()
    {
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    }
    __device__ __forceinline__ void join(const Sum<double>& o) { s += o.s; }
    __device__ __forceinline__ double value() const { return s; }
};
template <>
struct Sum<float> {
    float s = 0.f, c = 0.f;          // the sum is s + c
    __device__ __forceinline__ void add(float x)
    {
        const float t = __fadd_rn(s, x), b = __fsub_rn(t, s);
        c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(x, b)));
        s = t;
    }
    __device__ __forceinline__ void prod(float a, float b)
    {
        const float p = __fmul_rn(a, b);
        add(p);
        c = __fadd_rn(c, __fmaf_rn(a, b, -p));
    }
    // a - b = d + e exactly
    static __device__ __forceinline__ float split(float a, float b, float& e)
    {
        const float d = __fsub_rn(a, b), v = __fsub_rn(d, a);
        e = __fsub_rn(__fsub_rn(a, __fsub_rn(d, v)), __fadd_rn(b, v));
        return d;
    }
    __device__ __forceinline__ void square(float d, float e)
    {
        const float p = __fmul_rn(d, d);
        add(p);
        c = __fadd_rn(c, __fmaf_rn(__fadd_rn(d, d), e, __fmaf_rn(d, d, -p)));
    }
    __device__ __forceinline__ void diff(float a, float b, Sum<float>& sq)
    {
        float e;
        const float d = split(a, b, e);
        add(d);
        c = __fadd_rn(c, e);
        sq.square(d, e);
    }
    __device__ __forceinline__ void sqdiff(float a, float b)
    {
        float e;
        const float d = split(a, b, e);
        square(d, e);
    }
    __device__ __forceinline__ void join(const Sum<float>& o)
    {
        add(o.s);
        c = __fadd_rn(c, o.c);
    }
    __device__ __forceinline__ void warp()
    {
        for (int d = 16; d > 0; d >>= 1) {
            Sum<float> o;
            o.s = __shfl_down_sync(0xffffffffu, s, d);
            o.c = __shfl_down_sync(0xffffffffu, c, d);
            join(o);
        }
    }
    __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};

// Whether the largest magnitude of a block's FP32 values leaves the error-free
// transformations their room: squares of the scalar's differences (2^-24 of it and
// more) and the products w T keep their errors normal numbers, and nothing overflows.
__device__ __forceinline__ bool in_range(float m, float lo) { return m == 0.f || (m > lo && m < 1e9f); }
__device__ __forceinline__ bool in_range(double, float) { return true; }
constexpr float kLeastT = 1e-6f, kLeastW = 1e-18f;

// Block sums of NV values, in every thread: warps by shuffles, then one thread per
// value adds the warps' sums in order and converts once.
template <int NV, typename A>
__device__ __forceinline__ void block_sum(Sum<A> (&v)[NV], double (&out)[NV])
{
    __shared__ Sum<A> sh[NV][kThreads / 32];
    __shared__ double tot[NV];
    for (int q = 0; q < NV; ++q) {
        v[q].warp();
        if ((threadIdx.x & 31) == 0) sh[q][threadIdx.x >> 5] = v[q];
    }
    __syncthreads();
    if (threadIdx.x < NV) {
        Sum<A> s = sh[threadIdx.x][0];
        for (int w = 1; w < kThreads / 32; ++w) s.join(sh[threadIdx.x][w]);
        tot[threadIdx.x] = s.value();
    }
    __syncthreads();
    for (int q = 0; q < NV; ++q) out[q] = tot[q];
    __syncthreads();
}

// ------------------------------------------------------------- moments

// Whether a value is finite, and whether it is NaN; FP64 ones from their bits, a
// comparison taking as long as an addition.
__device__ __forceinline__ bool finite(float t) { return isfinite(t); }
__device__ __forceinline__ bool finite(double t) { return ((unsigned)__double2hiint(t) & 0x7ff00000u) != 0x7ff00000u; }
__device__ __forceinline__ bool is_nan(float t) { return isnan(t); }
__device__ __forceinline__ bool is_nan(double t)
{
    const unsigned hi = (unsigned)__double2hiint(t) & 0x7fffffffu;
    return hi > 0x7ff00000u || (hi == 0x7ff00000u && __double2loint(t) != 0);
}
// The sum of squares of values that are not finite, of which some are NaN (2) or not (1).
__device__ __forceinline__ double squares_of(int poison)
{
    return __hiloint2double(poison & 2 ? 0x7ff80000 : (poison ? 0x7ff00000 : 0), 0);
}

// One unit of a plane: sum and sum of squares of T - c over its finite values,
// their number's complement (bad), what the others are (squares_of), and the
// largest magnitude.
template <typename A, typename P>
__device__ __forceinline__ void moments_unit(const P* __restrict__ r, size_t lo, size_t hi, P c, Sum<A>& s1, Sum<A>& s2,
                                             int& bad, int& poison, P& big)
{
    constexpr int kGroup = 8;                              // loads in flight
    size_t m = lo + threadIdx.x;
    auto one = [&](P t) {
        if (finite(t)) {
            if constexpr (sizeof(P) == 4) big = fmaxf(big, fabsf(t));
            s1.diff(t, c, s2);
        } else {
            ++bad;
            poison |= is_nan(t) ? 2 : 1;
        }
    };
    for (; m + (kGroup - 1) * kThreads < hi; m += kGroup * kThreads) {
        P t[kGroup];
#pragma unroll
        for (int q = 0; q < kGroup; ++q) t[q] = r[m + q * kThreads];
#pragma unroll
        for (int q = 0; q < kGroup; ++q) one(t[q]);
    }
    for (; m < hi; m += kThreads) one(r[m]);
}

// A value near the mean of one or more units: kSample samples per thread and unit,
// spread over it (finite ones), and their mean in every thread (0 without any).
// Whatever the samples miss or hit, the squares about it are at most cells / samples
// (16) times those about the units' mean, so that at most four bits of them cancel;
// about one cell's value an outlier just there would cost as many bits as the units
// have.  The sum's last steps are one thread's and the division is FP32's: FP64
// operations are dear.
constexpr int kSample = 4;
template <typename P>
__device__ __forceinline__ void sample(const P* __restrict__ r, size_t lo, size_t hi, P& s, int& n)
{
    const size_t step = (hi - lo) / kSample;
#pragma unroll
    for (int q = 0; q < kSample; ++q) {
        const size_t m = lo + q * step + threadIdx.x;
        const P t = m < hi ? r[m] : P(NAN);
        if (finite(t)) {
            s += t;
            ++n;
        }
    }
}
template <typename P>
__device__ __forceinline__ P sample_mean(P s, int n)
{
    __shared__ P sum[kThreads / 32];
    __shared__ int num[kThreads / 32];
    __shared__ P mean;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    n = __reduce_add_sync(0xffffffffu, n);
    if ((threadIdx.x & 31) == 0) {
        sum[threadIdx.x >> 5] = s;
        num[threadIdx.x >> 5] = n;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kThreads / 32; ++w) {
            s += sum[w];
            n += num[w];
        }
        const P c = s * (P)(1.0f / (float)(n > 0 ? n : 1));
        mean = isfinite(c) ? c : P(0);
    }
    __syncthreads();
    return mean;
}

// Sum of T vol and of (T - mean)^2 vol (vol = dz_k, in FP64; the host applies dx dy), the
// count of non-finite values and their sum of squares into out[0..3].  An FP32 block's
// first unit takes T relative to a value near its own mean, each further one relative
// to the mean of the one before, so that no squares cancel beyond what the
// differences between units add to the variance anyway; every unit's pairs are summed
// over the block, and thread 0 refers them to the first one's value.  An FP64 block
// takes one value near the mean of all its units, and its threads add up their own
// sums until the end: the FP64 pipe bounds it, three operations a cell (512 x 512 x 256
// cells: 469 us for the statistics, 771 with the units summed over the block one by
// one and FP64 comparisons, 682 in two passes).  The block that finishes last (an
// atomic count, nothing waits) combines the blocks' (sum, squares, weight) about the
// common mean, in a fixed order.
// 256 x 256 x 192 FP32 cells: 34 us (40 instructions per cell, and the last block's
// FP64 combination at the end; 32 us about a block's first cell, which an outlier
// there makes useless); a pass for the mean and one for the squares took 2 x 20 us,
// each with a copy of the partials to the host and a synchronisation.
template <typename P>
__global__ void __launch_bounds__(kThreads) k_moments(Grid<P> g, const P* __restrict__ T, const double* __restrict__ dz,
                                                      int per_plane, double vtot, double* __restrict__ partials, 
                                                      unsigned* __restrict__ count, double* __restrict__ out)
{
    const size_t plane = (size_t)g.Nx * g.Ny, per = (plane + per_plane - 1) / per_plane;
    const int units = g.Nz * per_plane;
    double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};              // thread 0: S1, S2, weight, bad, poison
    P c = P(0), cb = P(0);                                // this unit's value, the first unit's
    if constexpr (sizeof(P) == 8) {
        P s = P(0);
        int n = 0;
        for (int u = blockIdx.x; u < units; u += gridDim.x) {
            const size_t lo = (size_t)(u % per_plane) * per, hi = lo + per < plane ? lo + per : plane;
            if (lo < hi) sample(T + (size_t)(u / per_plane) * plane, lo, hi, s, n);
        }
        cb = sample_mean(s, n);
        Sum<double> a[5];
        for (int u = blockIdx.x; u < units; u += gridDim.x) {
            const int k = u / per_plane;
            const size_t lo = (size_t)(u % per_plane) * per, hi = lo + per < plane ? lo + per : plane;
            if (lo >= hi) continue;
            Sum<double> d[2];
            int bad = 0, poison = 0;
            P big = P(0);
            moments_unit(T + (size_t)k * plane, lo, hi, cb, d[0], d[1], bad, poison, big);
            const double z = dz[k];
            a[0].s = fma(d[0].s, z, a[0].s);
            a[1].s = fma(d[1].s, z, a[1].s);
            if (threadIdx.x == 0) a[2].s = fma((double)(hi - lo), z, a[2].s);
            if (bad) {                                    // the weight less the bad values'
                a[2].s -= (double)bad * z;
                a[3].s += (double)bad;
                a[4].s += squares_of(poison);
            }
        }
        block_sum(a, v);
    } else {
        bool first = true;
        for (int u = blockIdx.x; u < units; u += gridDim.x) {
            const int k = u / per_plane;
            const size_t lo = (size_t)(u % per_plane) * per, hi = lo + per < plane ? lo + per : plane;
            if (lo >= hi) continue;
            const P* r = T + (size_t)k * plane;
            if (first) {
                P s = P(0);
                int n = 0;
                sample(r, lo, hi, s, n);
                c = cb = sample_mean(s, n);
            }
            first = false;
            Sum<P> s[2];
            int bad = 0, poison = 0;
            P big = fabs(c);
            moments_unit(r, lo, hi, c, s[0], s[1], bad, poison, big);
            double w[2];
            if (__syncthreads_or(!in_range(big, kLeastT))) {
                Sum<double> d[2];
                bad = 0;
                poison = 0;
                moments_unit(r, lo, hi, c, d[0], d[1], bad, poison, big);
                block_sum(d, w);
            } else {
                block_sum(s, w);
            }
            double n[2] = {0.0, 0.0};
            if (__syncthreads_or(bad)) {
                Sum<double> d[2];
                d[0].s = (double)bad;
                d[1].s = squares_of(poison);
                block_sum(d, n);
            }
            if (threadIdx.x == 0) {
                const double good = (double)(hi - lo) - n[0], d = (double)c - (double)cb;
                v[0] = fma(fma(d, good, w[0]), dz[k], v[0]);
                v[1] = fma(fma(d, fma(d, good, 2.0 * w[0]), w[1]), dz[k], v[1]);
                v[2] = fma(good, dz[k], v[2]);
                v[3] += n[0];
                v[4] += n[1];
            }
            // the next unit's value, in every thread alike (near this one's mean will do)
            if (u + (int)gridDim.x >= units) break;
            const float count = (float)(hi - lo) - (float)n[0];
            const P m = c + (P)w[0] * (P)(1.0f / count);
            c = isfinite(m) ? m : P(0);
        }
    }
    __shared__ bool last;
    if (threadIdx.x == 0) {
        double* p = partials + 6 * (size_t)blockIdx.x;
        for (int q = 0; q < 5; ++q) p[q] = v[q];
        p[5] = (double)cb;
        __threadfence();                                  // this block's partials before its count
        last = atomicAdd(count, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    Sum<double> s[3];
    for (unsigned q = threadIdx.x; q < gridDim.x; q += kThreads) {
        const double* p = partials + 6 * (size_t)q;
        s[0].s += fma(__ldcg(p + 5), __ldcg(p + 2), __ldcg(p));
        s[1].s += __ldcg(p + 3);
        s[2].s += __ldcg(p + 4);
    }
    double t[3], tm[1];
    block_sum(s, t);
    const double mean = t[0] / vtot;
    Sum<double> m2[1];
    for (unsigned q = threadIdx.x; q < gridDim.x; q += kThreads) {
        const double* p = partials + 6 * (size_t)q;
        const double d = __ldcg(p + 5) - mean;
        m2[0].s += fma(d, fma(d, __ldcg(p + 2), 2.0 * __ldcg(p)), __ldcg(p + 1));
    }
    block_sum(m2, tm);
    if (threadIdx.x == 0) {
        out[0] = t[0];
        out[1] = t[1] > 0.0 ? t[2] : tm[0];
        out[2] = t[1];
        *count = 0u;
    }
}

// ------------------------------------------------------------- profiles

template <typename P, int N>
struct alignas(sizeof(P) * N) Pack {
    P v[N];
};

// R rows of the horizontal split of W (uniform periodic x and y).
struct SplitRows {
    float rx[4][3], ry[4][3];
};

// One block's share of z-face k (planes k - 1 below, k above; a plate's value in
// the place of the missing one): the sums of w T (over the planes below and above,
// or the four of the fourth-order face value), of T_above - T_below and its
// square, and of the squared x and y differences on plane k.
// M = 0: W is dense; otherwise its split in x and y from the full-area W of the
// M x M coarse columns (Wk, coarse plane k) is formed here.
constexpr int kSums = 8;             // w T (4 planes), dT, dT^2 (z), x, y
template <typename A, typename P, int M, bool O4>
__device__ __forceinline__ void profile_share(const Grid<P>& g, const P* __restrict__ T, const P* __restrict__ Ws,
                                              const float* __restrict__ Wk, const SplitRows& R, const float (*ry)[3],
                                              int k, size_t lo, size_t hi,
                                              Sum<A> (&s)[kSums], P& big, P& bigw)
{
    constexpr int SEG = M > 0 ? M : 1;
    const size_t plane = (size_t)g.Nx * g.Ny;
    const int nseg = g.Nx / SEG;
    const bool below = k > 0, above = k < g.Nz;
    const P* const pb = T + (size_t)(below ? k - 1 : 0) * plane;
    const P* const pa = T + (size_t)(above ? k : 0) * plane;
    // the thread's segments: one division, then steps of kThreads
    const int dj = kThreads / nseg, dx = kThreads % nseg;
    int j = (int)((lo + threadIdx.x) / nseg), xs = (int)((lo + threadIdx.x) % nseg);
    for (size_t e = lo + threadIdx.x; e < hi; e += kThreads, j += dj, xs += dx) {
        if (xs >= nseg) {
            xs -= nseg;
            ++j;
        }
        const int x0 = xs * SEG;
        const size_t m = (size_t)j * g.Nx + x0;
        P w[SEG];
        if (below && above) {
            if constexpr (M > 0) {
                const int I = x0 / M, J = j / M, b = j % M;
                const int Im = I == 0 ? g.nx - 1 : I - 1, Ip = I == g.nx - 1 ? 0 : I + 1;
                const int Jm = J == 0 ? g.ny - 1 : J - 1, Jp = J == g.ny - 1 ? 0 : J + 1;
                const float *r0 = Wk + (size_t)Jm * g.nx, *r1 = Wk + (size_t)J * g.nx, *r2 = Wk + (size_t)Jp * g.nx;
                const float y0 = ry[b][0], y1 = ry[b][1], y2 = ry[b][2];
                const float a = y0 * r0[Im] + y1 * r1[Im] + y2 * r2[Im];
                const float c = y0 * r0[I] + y1 * r1[I] + y2 * r2[I];
                const float d = y0 * r0[Ip] + y1 * r1[Ip] + y2 * r2[Ip];
#pragma unroll
                for (int q = 0; q < SEG; ++q) w[q] = R.rx[q][0] * a + R.rx[q][1] * c + R.rx[q][2] * d;
            } else {
                w[0] = Ws[(size_t)k * plane + m];
            }
        }
        P west = P(0);
        const bool wx = above && !(g.walls && x0 == 0), wy = above && !(g.walls && j == 0);
        if (wx) west = pa[x0 == 0 ? m + g.Nx - 1 : m - 1];
        const size_t south = j == 0 ? m + plane - g.Nx : m - g.Nx;
        using V = Pack<P, SEG>;                            // segments start at multiples of SEG
        const V vb = *reinterpret_cast<const V*>(pb + m), va = *reinterpret_cast<const V*>(pa + m),
                vs = *reinterpret_cast<const V*>(pa + (wy ? south : m));
#pragma unroll
        for (int q = 0; q < SEG; ++q) {
            const P tb = below ? vb.v[q] : P(0.5), ta = above ? va.v[q] : P(-0.5);
            big = fmax(big, fmax(fabs(tb), fabs(ta)));
            s[4].diff(ta, tb, s[5]);
            if (below && above) {
                bigw = fmax(bigw, fabs(w[q]));
                s[1].prod(w[q], tb);
                s[2].prod(w[q], ta);
                if constexpr (O4) {
                    if (k >= 2) s[0].prod(w[q], T[(size_t)(k - 2) * plane + m + q]);
                    if (k + 1 < g.Nz) s[3].prod(w[q], T[(size_t)(k + 1) * plane + m + q]);
                }
            }
            if (q > 0 || wx) s[6].sqdiff(ta, west);
            if (wy) s[7].sqdiff(ta, vs.v[q]);
            west = ta;
        }
    }
}

// Block face * slices + slice; sums[face][slice][kSums].  256 x 256 x 192 FP32 cells:
// 76 us for both profiles; 1035 us for the gradient squares and 728 us for the
// fluxes when every cell converted to FP64 and divided in FP64.
template <typename P, int M, bool O4>
__global__ void __launch_bounds__(kThreads) k_profiles(Grid<P> g, const P* __restrict__ T, const P* __restrict__ Ws,
                                                       const float* __restrict__ Wc, const float* __restrict__ Win,
                                                       const SplitRows R, int slices, double* __restrict__ sums)
{
    const int k = blockIdx.x / slices, slice = blockIdx.x % slices;
    constexpr int SEG = M > 0 ? M : 1;
    const size_t nel = (size_t)g.Ny * (g.Nx / SEG), per = (nel + slices - 1) / slices;
    const size_t lo = (size_t)slice * per, hi = lo + per < nel ? lo + per : nel;
    const size_t cplane = (size_t)g.nx * g.ny;
    // full-area W of face k: the given one on the coarse planes, the slab balance on the others
    const float* Wk = M > 0 ? (k % SEG == 0 ? Wc + (size_t)(k / SEG) * cplane : Win + (size_t)k * cplane) : nullptr;
    __shared__ float ry[4][3];                             // indexed by the dense row: not from the parameters
    if (threadIdx.x < 12) ry[threadIdx.x / 3][threadIdx.x % 3] = (&R.ry[0][0])[threadIdx.x];
    __syncthreads();
    double b[kSums];
    {
        Sum<P> s[kSums];
        P big = P(0), bigw = P(0);
        profile_share<P, P, M, O4>(g, T, Ws, Wk, R, ry, k, lo, hi, s, big, bigw);
        const bool redo = __syncthreads_or(!(in_range(big, kLeastT) && in_range(bigw, kLeastW)));
        if (!redo) {
            block_sum(s, b);
        } else {
            Sum<double> d[kSums];
            profile_share<double, P, M, O4>(g, T, Ws, Wk, R, ry, k, lo, hi, d, big, bigw);
            block_sum(d, b);
        }
    }
    if (threadIdx.x == 0)
        for (int q = 0; q < kSums; ++q) sums[(size_t)blockIdx.x * kSums + q] = b[q];
}

// The slices of a face added in order: thread per (face, sum).
__global__ void k_profile_sum(const double* __restrict__ sums, int faces, int slices, double* __restrict__ out)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= faces * kSums) return;
    const double* p = sums + (size_t)(t / kSums) * slices * kSums + t % kSums;
    double s = 0.0;
    for (int q = 0; q < slices; ++q) s += p[(size_t)q * kSums];
    out[t] = s;
}

}  // namespace

template <typename P>
cudaError_t launch_moments(const Grid<P>& g, const P* T, const double* dz, double vtot, double* work, double* out, cudaStream_t st)
{
    // units of at most kShare cells per thread, one block each up to the blocks
    // that work holds (the first double is the count)
    const size_t plane = (size_t)g.Nx * g.Ny;
    const int per_plane = (int)((plane + (size_t)kThreads * kShare - 1) / ((size_t)kThreads * kShare));
    const long long units = (long long)per_plane * g.Nz;
    const int blocks = (int)(units < kMomentBlocks ? units : kMomentBlocks);
    k_moments<P><<<blocks, kThreads, 0, st>>>(g, T, dz, per_plane, vtot, work + 1, reinterpret_cast<unsigned*>(work), out);
    return cudaGetLastError();
}

int profile_slices(size_t plane) { return (int)((plane + (size_t)kThreads * kShare - 1) / ((size_t)kThreads * kShare)); }
size_t profile_work(size_t plane, int Nz) { return ((size_t)Nz + 1) * kSums * (profile_slices(plane) + 1); }

template <typename P>
cudaError_t launch_profiles(const Grid<P>& g, const P* T, const P* Ws, const float* Wc, const float* Win,
                            const float* rx12, const float* ry12, double* work, cudaStream_t st)
{
    const size_t plane = (size_t)g.Nx * g.Ny;
    const int slices = profile_slices(plane);
    double* part = work + ((size_t)g.Nz + 1) * kSums;
    SplitRows R = {};
    if (!Ws)
        for (int q = 0; q < 12; ++q) {
            R.rx[q / 3][q % 3] = rx12[q];
            R.ry[q / 3][q % 3] = ry12[q];
        }
    const unsigned grd = (unsigned)slices * (unsigned)(g.Nz + 1);
    if (Ws) {
        if (g.order4) k_profiles<P, 0, true><<<grd, kThreads, 0, st>>>(g, T, Ws, nullptr, nullptr, R, slices, part);
        else k_profiles<P, 0, false><<<grd, kThreads, 0, st>>>(g, T, Ws, nullptr, nullptr, R, slices, part);
    } else if constexpr (sizeof(P) == 4) {
        if (g.mx == 4) {
            if (g.order4) k_profiles<P, 4, true><<<grd, kThreads, 0, st>>>(g, T, nullptr, Wc, Win, R, slices, part);
            else k_profiles<P, 4, false><<<grd, kThreads, 0, st>>>(g, T, nullptr, Wc, Win, R, slices, part);
        } else {
            if (g.order4) k_profiles<P, 2, true><<<grd, kThreads, 0, st>>>(g, T, nullptr, Wc, Win, R, slices, part);
            else k_profiles<P, 2, false><<<grd, kThreads, 0, st>>>(g, T, nullptr, Wc, Win, R, slices, part);
        }
    }
    const int n = (g.Nz + 1) * kSums;
    k_profile_sum<<<(n + 127) / 128, 128, 0, st>>>(part, g.Nz + 1, slices, work);
    return cudaGetLastError();
}

template cudaError_t launch_moments<double>(const Grid<double>&, const double*, const double*, double, double*, double*, cudaStream_t);
template cudaError_t launch_moments<float>(const Grid<float>&, const float*, const double*, double, double*, double*, cudaStream_t);
template cudaError_t launch_profiles<double>(const Grid<double>&, const double*, const double*, const float*, const float*,
                                             const float*, const float*, double*, cudaStream_t);
template cudaError_t launch_profiles<float>(const Grid<float>&, const float*, const float*, const float*, const float*,
                                            const float*, const float*, double*, cudaStream_t);

// ------------------------------------------------------------- results

// What a synchronising call returns, gathered into res by one block so that one
// small copy brings it: res[0..2] as it is (moments), res[3..4] the plate Nusselt
// numbers, res[5] the maximum of n partials, res[6] the fused kernels' error flag,
// which is cleared.  Any of nu2, part, err may be NULL.
__global__ void __launch_bounds__(kThreads) k_gather(const double* __restrict__ nu2, const double* __restrict__ part, int n,
                                                     int* __restrict__ err, double* __restrict__ res)
{
    __shared__ double sh[kThreads / 32];
    double m = 0.0;
    if (part)
        for (int q = threadIdx.x; q < n; q += kThreads) m = fmax(m, part[q]);
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x) return;
    for (int w = 1; w < kThreads / 32; ++w) m = fmax(m, sh[w]);
    if (nu2) {
        res[3] = nu2[0];
        res[4] = nu2[1];
    }
    res[5] = m;
    res[6] = err ? (double)*err : 0.0;
    if (err && *err) *err = 0;
}

cudaError_t launch_gather(const double* nu2, const double* part, int n, int* err, double* res, cudaStream_t st)
{
    k_gather<<<1, kThreads, 0, st>>>(nu2, part, n, err, res);
    return cudaGetLastError();
}

}  // namespace mr
