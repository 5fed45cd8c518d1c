// 64-bit fixed-point arithmetic on the integer pipes, for the FP64 path.
//
// GB300 issues FP64 arithmetic (and every conversion from or to FP64) at 2
// lanes per clock and SM, 1/64 of its FP32 rate, but 32 x 32 + 64-bit integer
// multiply-adds at ~50 and 32-bit integer operations at 64 lanes per clock and
// SM (measured).  So a stencil over values of one scale is several times faster
// in integers: every value becomes a 60- or 62-bit integer relative to the
// largest one of its neighbourhood, sums of integers are exact, and a product
// of two of them is three multiply-adds of balanced 32-bit halves with an error
// of 2^-60 of its largest value, where FP64 rounds at 2^-53 of its own.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace mr {
namespace fix {

// x = hi 2^32 + lo with both halves signed
struct Bal {
    int hi, lo;
};
__host__ __device__ __forceinline__ Bal bal(long long x)
{
    const unsigned lo = (unsigned)x;
    return {(int)(x >> 32) + (int)(lo >> 31), (int)lo};
}

// a sum of products: H 2^64 + M 2^32 (the products of the low halves are left out)
struct Acc {
    long long H, M;
};
__host__ __device__ __forceinline__ long long madw(int a, int b, long long c)
{
#ifdef __CUDA_ARCH__
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return (long long)a * b + c;
#endif
}
__host__ __device__ __forceinline__ void mac(Acc& s, Bal a, Bal b)
{
    s.M = madw(a.hi, b.lo, s.M);
    s.M = madw(a.lo, b.hi, s.M);
    s.H = madw(a.hi, b.hi, s.H);
}
// the product in units of 2^64
__host__ __device__ __forceinline__ long long mul(Bal a, Bal b)
{
    Acc s{0, 0};
    mac(s, a, b);
    return madw((int)(s.M >> 32), 1, s.H);
}

// The double with words (hi, lo) as an integer of at most BITS bits relative to
// the exponent field E >= its own: trunc(|x| 2^(BITS - (E - 1022))), the sign by
// complement (so negative values come out one unit lower; negating them costs 2 % of
// a step and makes no result more accurate).  Zeros and subnormals, whose field is 0,
// come out as 0 (or -1) for every E >= 80; where a cell and its neighbours are all
// zeros of either sign, what that leaves is below a quarter of a unit of the step's
// sum, and the cell stays zero.
template <int BITS>
__host__ __device__ __forceinline__ long long dec(int hi, int lo, int E)
{
    constexpr int L = BITS - 53;
    // E - e from the magnitude's high word, which a caller may have taken already
    const int d = (int)((((unsigned)E << 20) | 0xfffffu) - ((unsigned)hi & 0x7fffffffu)) >> 20;
    const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u, ml = (unsigned)lo;
    const int s = hi >> 31;
#ifdef __CUDA_ARCH__
    const unsigned long long m = ((unsigned long long)__funnelshift_l(ml, mh, L) << 32) | (ml << L);
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(m), "r"(d));       // 0 from 64 on
#else
    const unsigned long long m = ((unsigned long long)mh << 32 | ml) << L, r = d > 63 ? 0ull : m >> d;
#endif
    return (long long)((unsigned long long)(unsigned)((int)(r >> 32) ^ s) << 32 | (unsigned)((int)r ^ s));
}

// Columns of a band of rows on the line that the warps of a step share out, 30 each:
// a neighbour column at both ends of the band and, where that adds 5 % at most, a
// rounding to whole warps, whose reads then do not cross bands (256 columns: 212
// against 213 us per step on 256 x 256 x 192 cells; without rounding 123 columns,
// 125 instead of 150, 41 -> 35 us on 123 x 74 x 148, and 128 columns, 130 instead of 150,
// 40 -> 37 us on 128 x 128 x 96).
__host__ __device__ __forceinline__ int band_span(int nx)
{
    const int n = nx + 2, whole = (n + 29) / 30 * 30;
    return whole - n <= n / 20 ? whole : n;
}

#ifdef __CUDACC__
__device__ __forceinline__ double pow2(int n) { return __hiloint2double((n + 1023) << 20, 0); }
__device__ __forceinline__ Bal fixed(double v) { return bal(__double2ll_rn(v)); }
// the magnitude of a double, ordered like its high word without the sign
__device__ __forceinline__ unsigned mag(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }

template <int BITS>
__device__ __forceinline__ long long dec(double v, int E)
{
    return fix::dec<BITS>(__double2hiint(v), __double2loint(v), E);
}

// the least e with v < 2^e, v positive and normal
__device__ __forceinline__ int exponent(double v) { return ((__double2hiint(v) >> 20) & 0x7ff) - 1022; }

// 2^-900 <= v < 2^900, without an FP64 comparison
__device__ __forceinline__ bool ordinary(double v)
{
    return (unsigned)__double2hiint(v) - (123u << 20) < (1800u << 20);
}

// asynchronous 8-byte copies into shared memory
__device__ __forceinline__ void copy8(double* dst, const double* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ const double* at(const double* base, unsigned bytes)
{
    return reinterpret_cast<const double*>(reinterpret_cast<const char*>(base) + bytes);
}
#endif

}  // namespace fix
}  // namespace mr
