// Scalar time step with the dense velocity read from HBM (MR_VEL_STORED),
// FP64 or FP32.  Eq. (5) in flux form, second-order (linear) face values,
// Euler-leapfrog with the averaging step (Section 2.2):
//   T^{s+1} = a T^{s-1} + b T^s + gdt [C(T^s) + D(T^{s-1})]
// C = -(1/Vol) sum_faces u_f T_f A_f (outward), D = (1/Vol) sum kappa A dT/dn.
// Per-layer coefficients (1/dz, interpolation weights, kappa/(dz d)) come
// from the handle's grid, so a stretched z costs no extra arithmetic.
#include <mutex>
#include <unordered_map>

#include "mr_internal.cuh"

namespace mr {
namespace {

constexpr double kTBottom = 0.5;
constexpr double kTTop = -0.5;
constexpr size_t kAloneCells = (size_t)4 << 20;

// Dense face velocity of a step: one stored field, or (LERP) the linear
// interpolation A + alpha (B - A) between the fields of two coarse time
// levels (temporal refinement, Section 3.4).
template <typename P, bool LERP>
struct FaceVel {
    const P* A;
    const P* B;
    P alpha;
    __device__ __forceinline__ P operator[](size_t f) const
    {
        if (!LERP) return A[f];
        const P a = A[f];
        return a + alpha * (B[f] - a);
    }
};

// Fourth-order value at face f of an axis of N cells (Section 2.2): the cells
// f-2 .. f+1 at T[base + c * stride] with the grid's weights; periodic cells
// wrap, cells beyond a wall carry zero weight and are not read.
template <typename P>
__device__ __forceinline__ P face4(const P* w, int f, int N, bool periodic, const P* T, size_t base, size_t stride)
{
    P s = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        int c = f - 2 + q;
        if (periodic) c = c < 0 ? c + N : (c >= N ? c - N : c);
        else if (c < 0 || c >= N) continue;
        s += w[4 * f + q] * T[base + (size_t)c * stride];
    }
    return s;
}

// One thread per dense cell.  IMPLZ: vertical diffusion enters as
// (D_z(T^{s-1}) + plate terms) / 2; the implicit half follows in k_zsolve.
// O4: fourth-order face values of the advected scalar.
template <typename P, bool IMPLZ, bool LERP, bool O4>
__device__ __forceinline__ void step_cell(const Grid<P>& g, const FaceVel<P, LERP>& Us, const FaceVel<P, LERP>& Vs,
                                          const FaceVel<P, LERP>& Ws, const P* Tm1, const P* T, P* Tp1, P a, P b, P gdt)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= g.Nx || j >= g.Ny) return;
    const size_t plane = (size_t)g.Nx * g.Ny;
    const size_t m = (size_t)k * plane + (size_t)j * g.Nx + i;
    const P Tc = T[m], Dc = Tm1[m];
    const P half = P(0.5);
    P cx = 0, dx_ = 0, cy = 0, dy_ = 0;
    // x faces
    const size_t urow = ((size_t)k * g.Ny + j) * g.ufx;
    if (!(g.walls && i == 0)) {
        const int iw = (i == 0) ? g.Nx - 1 : i - 1;
        const size_t mw = m - i + iw;
        cx += Us[urow + i] * (O4 ? face4(g.f4x, i, g.Nx, !g.walls, T, m - i, 1) : half * (T[mw] + Tc));
        dx_ -= Dc - Tm1[mw];
    }
    if (!(g.walls && i == g.Nx - 1)) {
        const int ie = (i == g.Nx - 1) ? 0 : i + 1;
        const int fe = g.walls ? i + 1 : ie;
        const size_t me = m - i + ie;
        cx -= Us[urow + fe] * (O4 ? face4(g.f4x, i + 1, g.Nx, !g.walls, T, m - i, 1) : half * (Tc + T[me]));
        dx_ += Tm1[me] - Dc;
    }
    // y faces
    if (!(g.walls && j == 0)) {
        const int js = (j == 0) ? g.Ny - 1 : j - 1;
        const size_t ms = m + ((ptrdiff_t)js - j) * g.Nx;
        cy += Vs[((size_t)k * g.vfy + j) * g.Nx + i] *
              (O4 ? face4(g.f4y, j, g.Ny, !g.walls, T, m - (size_t)j * g.Nx, g.Nx) : half * (T[ms] + Tc));
        dy_ -= Dc - Tm1[ms];
    }
    if (!(g.walls && j == g.Ny - 1)) {
        const int jn = (j == g.Ny - 1) ? 0 : j + 1;
        const int fn = g.walls ? j + 1 : jn;
        const size_t mn = m + ((ptrdiff_t)jn - j) * g.Nx;
        cy -= Vs[((size_t)k * g.vfy + fn) * g.Nx + i] *
              (O4 ? face4(g.f4y, j + 1, g.Ny, !g.walls, T, m - (size_t)j * g.Nx, g.Nx) : half * (Tc + T[mn]));
        dy_ += Tm1[mn] - Dc;
    }
    // z faces (plates: no advective flux; Dirichlet or zero diffusive flux)
    P cz = 0, dz_ = 0;
    if (k > 0) {
        const P Tb = T[m - plane];
        cz += Ws[m] * (O4 ? face4(g.f4z, k, g.Nz, false, T, m - k * plane, plane) : g.wlo[k] * Tb + g.whi[k] * Tc);
        dz_ -= g.cdn[k] * (Dc - Tm1[m - plane]);
    } else {
        dz_ -= g.cdn[0] * (Dc - P(kTBottom));    // cdn[0] = 0 when adiabatic
    }
    if (k < g.Nz - 1) {
        const P Tt = T[m + plane];
        cz -= Ws[m + plane] *
              (O4 ? face4(g.f4z, k + 1, g.Nz, false, T, m - k * plane, plane) : g.wlo[k + 1] * Tc + g.whi[k + 1] * Tt);
        dz_ += g.cup[k] * (Tm1[m + plane] - Dc);
    } else {
        dz_ += g.cup[k] * (P(kTTop) - Dc);        // cup[Nz-1] = 0 when adiabatic
    }
    if (IMPLZ) {
        // (Lz T^{s-1} + bz)/2 + bz/2: the plate terms count in full
        P bz = 0;
        if (k == 0) bz += g.cdn[0] * P(kTBottom);
        if (k == g.Nz - 1) bz += g.cup[k] * P(kTTop);
        dz_ = half * dz_ + half * bz;
    }
    const P C = cx * g.inv_dx + cy * g.inv_dy + cz * g.inv_dz[k];
    const P D = g.kx2 * dx_ + g.ky2 * dy_ + dz_;
    Tp1[m] = a * Dc + b * Tc + gdt * (C + D);
}
template <typename P, bool IMPLZ, bool LERP, bool O4>
__global__ void __launch_bounds__(256) k_step_stored(Grid<P> g, const FaceVel<P, LERP> Us, const FaceVel<P, LERP> Vs,
                                                     const FaceVel<P, LERP> Ws, const P* Tm1, const P* T,
                                                     P* __restrict__ Tp1, P a, P b, P gdt)
{
    after_previous();
    let_next();
    step_cell<P, IMPLZ, LERP, O4>(g, Us, Vs, Ws, Tm1, T, Tp1, a, b, gdt);
}
// Not launched ahead, so that the scalar is read-only while it lives and may be loaded
// as such.
template <typename P, bool IMPLZ, bool LERP, bool O4>
__global__ void __launch_bounds__(256) k_step_stored_alone(Grid<P> g, const FaceVel<P, LERP> Us, const FaceVel<P, LERP> Vs,
                                                           const FaceVel<P, LERP> Ws, const P* __restrict__ Tm1,
                                                           const P* __restrict__ T, P* __restrict__ Tp1, P a, P b, P gdt)
{
    step_cell<P, IMPLZ, LERP, O4>(g, Us, Vs, Ws, Tm1, T, Tp1, a, b, gdt);
}

// The same step (Eq. 5) for the common case -- periodic x and y, explicit
// diffusion, second-order faces, one velocity level -- with the arithmetic
// folded for the FP64 pipe (25 FP operations per cell instead of 39):
// 1/(2 dx), 1/(2 dy) scale the summed x and y flux differences, the z-face
// weights carry 1/dz_k (the top face's negated), the opposite diffusion
// neighbours are summed before kx2, ky2, and the diagonal and the plate
// terms come from the per-layer table g.lz.  LF: a plain leapfrog step.
template <typename P, bool LF>
__global__ void __launch_bounds__(256) k_step_periodic(Grid<P> g, const P* Us, const P* Vs, const P* Ws,
                                                       const P* Tm1, const P* T, P* __restrict__ Tp1, P a, P b, P gdt)
{
    after_previous();
    let_next();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= g.Nx || j >= g.Ny) return;
    const size_t plane = (size_t)g.Nx * g.Ny;
    const size_t row = (size_t)j * g.Nx, m = (size_t)k * plane + row + i;
    const P* L = g.lz + 8 * k;
    const int iw = i == 0 ? g.Nx - 1 : i - 1, ie = i == g.Nx - 1 ? 0 : i + 1;
    const int js = j == 0 ? g.Ny - 1 : j - 1, jn = j == g.Ny - 1 ? 0 : j + 1;
    const size_t mw = m - i + iw, me = m - i + ie;
    const size_t ms = m - row + (size_t)js * g.Nx, mn = m - row + (size_t)jn * g.Nx;
    const P Tc = T[m], Dc = Tm1[m];
    // beyond the plates: zero (W is zero there; the plate values enter through L[7])
    const bool lo = k > 0, hi = k < g.Nz - 1;
    const P Tb = lo ? T[m - plane] : P(0), Db = lo ? Tm1[m - plane] : P(0);
    const P Tt = hi ? T[m + plane] : P(0), Dt = hi ? Tm1[m + plane] : P(0);
    const size_t urow = ((size_t)k * g.Ny + j) * g.Nx, vrow = (size_t)k * g.Ny * g.Nx;
    const P ax = Us[urow + i] * (T[mw] + Tc) - Us[urow + ie] * (Tc + T[me]);
    const P ay = Vs[vrow + row + i] * (T[ms] + Tc) - Vs[vrow + (size_t)jn * g.Nx + i] * (Tc + T[mn]);
    const P az = Ws[m] * (L[0] * Tb + L[1] * Tc) + Ws[m + plane] * (L[2] * Tc + L[3] * Tt);
    const P D = L[7] + g.kx2 * (Tm1[mw] + Tm1[me]) + g.ky2 * (Tm1[ms] + Tm1[mn]) + L[4] * Db + L[5] * Dt + L[6] * Dc;
    const P C = g.hx * ax + g.hy * ay + az;
    Tp1[m] = LF ? Dc + gdt * (C + D) : a * Dc + b * Tc + gdt * (C + D);
}

// The FP32 form of k_step_periodic on rows of whole quads: a thread marches four
// cells of a row through kMarch layers, so that its loads are 16 bytes wide and the
// planes above become the current ones and those below in registers.  The
// operations are k_step_periodic's in its order and with its contractions (spelt
// out here), so that the results are the same to the last bit: the FP32 adjoint's
// coarse gradients magnify any other rounding of the forward run by 1e4.
// Bound by L2 and the loads' latency on grids that fit L2: 128 x 128 x 96 cells
// 7.6 us per step, 14.8 us with a cell per thread (back to back); 512 x 512 x 384:
// 467 and 870 us.
constexpr int kMarch = 4;
__device__ __forceinline__ float get(const float4& v, int q) { return q == 0 ? v.x : (q == 1 ? v.y : (q == 2 ? v.z : v.w)); }
__device__ __forceinline__ void put(float4& v, int q, float x) { (q == 0 ? v.x : (q == 1 ? v.y : (q == 2 ? v.z : v.w))) = x; }
template <bool LF>
__global__ void __launch_bounds__(128) k_step_periodic4(Grid<float> g, const float* Us, const float* Vs,
                                                        const float* Ws, const float* Tm1, const float* T,
                                                        float* __restrict__ Tp1, float a, float b, float gdt, int march)
{
    after_previous();
    let_next();
    const unsigned quads = (unsigned)g.Nx / 4, s = blockIdx.x * 128u + threadIdx.x;
    if (s >= quads * (unsigned)g.Ny) return;
    const int j = (int)(s / quads), i = (int)(s % quads) * 4;
    const int k0 = blockIdx.y * march, k1 = min(k0 + march, g.Nz);
    const size_t plane = (size_t)g.Nx * g.Ny, row = (size_t)j * g.Nx + i;
    const size_t west = row - i + (i == 0 ? g.Nx - 1 : i - 1), east = row - i + (i + 4 == g.Nx ? 0 : i + 4);
    const size_t south = (size_t)(j == 0 ? g.Ny - 1 : j - 1) * g.Nx + i, north = (size_t)(j == g.Ny - 1 ? 0 : j + 1) * g.Nx + i;
    auto quad = [](const float* p) { return *reinterpret_cast<const float4*>(p); };
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    size_t m = (size_t)k0 * plane;
    float4 tb = k0 > 0 ? quad(T + m - plane + row) : zero, db = k0 > 0 ? quad(Tm1 + m - plane + row) : zero;
    float4 tc = quad(T + m + row), dc = quad(Tm1 + m + row), wb = quad(Ws + m + row);
    for (int k = k0; k < k1; ++k, m += plane) {
        const float* L = g.lz + 8 * k;
        const bool hi = k < g.Nz - 1;
        const float4 tt = hi ? quad(T + m + plane + row) : zero, dt = hi ? quad(Tm1 + m + plane + row) : zero;
        const float4 wt = quad(Ws + m + plane + row);
        const float4 ts = quad(T + m + south), tn = quad(T + m + north), ds = quad(Tm1 + m + south), dn = quad(Tm1 + m + north);
        const float4 u = quad(Us + m + row), vs = quad(Vs + m + row), vn = quad(Vs + m + north);
        const float tw = T[m + west], te = T[m + east], dw = Tm1[m + west], de = Tm1[m + east], ue = Us[m + east];
        float4 out;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float Tc = get(tc, q), Dc = get(dc, q);
            const float Tw = q ? get(tc, q - 1) : tw, Te = q < 3 ? get(tc, q + 1) : te;
            const float Dw = q ? get(dc, q - 1) : dw, De = q < 3 ? get(dc, q + 1) : de;
            const float U0 = get(u, q), U1 = q < 3 ? get(u, q + 1) : ue;
            const float ax = __fmaf_rn(U0, __fadd_rn(Tw, Tc), -__fmul_rn(U1, __fadd_rn(Tc, Te)));
            const float ay = __fmaf_rn(get(vs, q), __fadd_rn(get(ts, q), Tc), -__fmul_rn(get(vn, q), __fadd_rn(Tc, get(tn, q))));
            const float az = __fmaf_rn(get(wb, q), __fmaf_rn(L[0], get(tb, q), __fmul_rn(L[1], Tc)),
                                       __fmul_rn(get(wt, q), __fmaf_rn(L[2], Tc, __fmul_rn(L[3], get(tt, q)))));
            float D = __fmaf_rn(g.kx2, __fadd_rn(Dw, De), L[7]);
            D = __fmaf_rn(g.ky2, __fadd_rn(get(ds, q), get(dn, q)), D);
            D = __fmaf_rn(L[4], get(db, q), D);
            D = __fmaf_rn(L[5], get(dt, q), D);
            D = __fmaf_rn(L[6], Dc, D);
            const float C = __fadd_rn(__fmaf_rn(g.hx, ax, __fmul_rn(g.hy, ay)), az), S = __fadd_rn(C, D);
            put(out, q, LF ? __fmaf_rn(gdt, S, Dc) : __fmaf_rn(gdt, S, __fmaf_rn(a, Dc, __fmul_rn(b, Tc))));
        }
        *reinterpret_cast<float4*>(Tp1 + m + row) = out;
        tb = tc;
        db = dc;
        tc = tt;
        dc = dt;
        wb = wt;
    }
}

// Opt-in implicit vertical diffusion: per (x, y) column solve
//   (1 + h (cup + cdn)) x_k - h cdn_k x_{k-1} - h cup_k x_{k+1} = r_k,
// h = gdt / 2, by elimination from both plates at once: lanes 0..15 of a warp
// eliminate the lower halves of 16 columns upwards, lanes 16..31 their upper
// halves downwards, the two middle values follow from one exchange, and both
// substitute back towards their plate.  The eliminated coefficients do not
// depend on the column, so the host forms them (ZTable, in FP64) and they come
// with the launch: per layer, counted from the lane's plate,
//   y_n = id r_n + e y_{n-1},   then   x_n = y_n + f x_{n+1},
// three multiply-adds per cell and no division.  The loads of eight layers are
// in flight ahead of the chain, and y stays in shared memory where a block's
// columns fit (SM), so that X is read and written once; blocks of one warp
// spread the columns over the SMs.  What bounds it is the FP64 pipe, which takes
// 64 clocks per instruction of a warp, so half the layers per warp on twice the
// warps is what fills the chip's pipes on small planes.
// Measured on 123 x 74 x 148 cells in FP64 (ncu): 19.4 us; 29.7 us with a whole
// column per lane, 224 us with two FP64 divisions per cell and the coefficients
// in global memory.
constexpr int kZBatch = 8;
template <typename P, int N>
struct ZTable {
    P id[N], e[N], f[N];
    P mid;                                                 // 1 / (1 - f f) of the middle pair
};
template <typename P, int N, bool SM>
__global__ void __launch_bounds__(32) k_zsolve(P* __restrict__ X, size_t plane, int Nz,
                                               const __grid_constant__ ZTable<P, N> z)
{
    extern __shared__ __align__(16) unsigned char zsm[];
    const int lane = threadIdx.x;
    const bool up = lane >= 16;                            // from the upper plate
    const size_t m = (size_t)blockIdx.x * 16 + (lane & 15);
    const bool on = m < plane;                             // off: a column of the domain, read but not written
    P* const x = X + (on ? m : plane - 1) + (up ? (size_t)(Nz - 1) * plane : 0);
    const ptrdiff_t step = up ? -(ptrdiff_t)plane : (ptrdiff_t)plane;
    const int cnt = up ? Nz - Nz / 2 : Nz / 2, k0 = up ? Nz - 1 : 0, dk = up ? -1 : 1;
    P* const y = reinterpret_cast<P*>(zsm) + lane;
    P r[kZBatch], v = P(0);
#pragma unroll
    for (int q = 0; q < kZBatch; ++q) r[q] = q < cnt ? x[q * step] : P(0);
    for (int n0 = 0; n0 < cnt; n0 += kZBatch) {
        P c[kZBatch];
#pragma unroll
        for (int q = 0; q < kZBatch; ++q) {
            c[q] = r[q];
            const int n = n0 + kZBatch + q;
            if (n < cnt) r[q] = x[n * step];
        }
#pragma unroll
        for (int q = 0; q < kZBatch; ++q) {
            const int n = n0 + q, k = k0 + n * dk;
            if (n < cnt) {
                v = z.id[k] * c[q] + z.e[k] * v;
                if (SM) y[n * 32] = v;
                else if (on) x[n * step] = v;
            }
        }
    }
    __syncwarp();
    // the middle pair: x = y + f x_other on both sides
    const P vo = __shfl_xor_sync(0xffffffffu, v, 16);
    if (cnt == 0) return;
    v = (v + z.f[k0 + (cnt - 1) * dk] * vo) * z.mid;
    if (on) x[(cnt - 1) * step] = v;
    for (int n0 = cnt - 2; n0 >= 0; n0 -= kZBatch) {
        P c[kZBatch];
#pragma unroll
        for (int q = 0; q < kZBatch; ++q) c[q] = n0 - q >= 0 ? (SM ? y[(n0 - q) * 32] : x[(n0 - q) * step]) : P(0);
#pragma unroll
        for (int q = 0; q < kZBatch; ++q) {
            const int n = n0 - q;
            if (n >= 0) {
                v = c[q] + z.f[k0 + n * dk] * v;
                if (on) x[n * step] = v;
            }
        }
    }
}

// The same for columns whose coefficients exceed a launch's parameters: formed
// per column, the eliminated super-diagonal in work (one value per cell).
template <typename P>
__global__ void k_zsolve_tall(Grid<P> g, P* __restrict__ X, P h, P* __restrict__ work)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (i >= g.Nx) return;
    const size_t plane = (size_t)g.Nx * g.Ny;
    const size_t base = (size_t)j * g.Nx + i;
    const int N = g.Nz;
    P prev_c = 0, prev_x = 0;
    for (int k = 0; k < N; ++k) {
        const P lo = (k > 0) ? -h * g.cdn[k] : P(0);
        const P up = (k < N - 1) ? -h * g.cup[k] : P(0);
        const P di = P(1) + h * (g.cup[k] + g.cdn[k]);
        const P den = di - lo * prev_c;
        const P c = up / den;
        const P x = (X[base + k * plane] - lo * prev_x) / den;
        work[base + k * plane] = c;
        X[base + k * plane] = x;
        prev_c = c;
        prev_x = x;
    }
    for (int k = N - 2; k >= 0; --k) {
        prev_x = X[base + k * plane] - work[base + k * plane] * prev_x;
        X[base + k * plane] = prev_x;
    }
}

template <typename P, int N>
cudaError_t zsolve_table(const Grid<P>& g, P* X, double h, const double* cdn, const double* cup, cudaStream_t st)
{
    ZTable<P, N> z;
    const int M = g.Nz / 2;                                // layers of the lower half
    double c = 0.0, fb = 0.0, ft = 0.0;                    // what the layer nearer to the plate left on this one
    for (int k = 0; k < M; ++k) {
        const double lo = k > 0 ? h * cdn[k] : 0.0, id = 1.0 / (1.0 + h * (cup[k] + cdn[k]) - lo * c);
        c = (k < g.Nz - 1 ? h * cup[k] : 0.0) * id;
        z.id[k] = (P)id;
        z.e[k] = (P)(lo * id);
        z.f[k] = (P)(fb = c);
    }
    c = 0.0;
    for (int k = g.Nz - 1; k >= M; --k) {
        const double up = k < g.Nz - 1 ? h * cup[k] : 0.0, id = 1.0 / (1.0 + h * (cup[k] + cdn[k]) - up * c);
        c = (k > 0 ? h * cdn[k] : 0.0) * id;
        z.id[k] = (P)id;
        z.e[k] = (P)(up * id);
        z.f[k] = (P)(ft = c);
    }
    z.mid = (P)(1.0 / (1.0 - fb * ft));
    const size_t plane = (size_t)g.Nx * g.Ny;
    const unsigned blocks = (unsigned)((plane + 15) / 16);
    const int bytes = (g.Nz - M) * 32 * (int)sizeof(P);
    // Launched when the step has finished: one-warp blocks that come up while it still
    // runs gather on the SMs that empty first, several to a scheduler, whose FP64 pipe
    // bounds them (70 instead of 57 us per step on 123 x 74 x 148 cells).
    // At least four blocks of one warp per SM (one per scheduler); beyond that y goes
    // through global memory
    if (bytes <= 56 * 1024) {
        static unsigned long long done = 0;                // one bit per device
        const cudaError_t e = smem_optin(reinterpret_cast<const void*>(k_zsolve<P, N, true>), 56 * 1024, &done);
        if (e != cudaSuccess) return e;
        k_zsolve<P, N, true><<<blocks, 32, bytes, st>>>(X, plane, g.Nz, z);
    } else {
        k_zsolve<P, N, false><<<blocks, 32, 0, st>>>(X, plane, g.Nz, z);
    }
    return cudaGetLastError();
}

template <typename P, bool LERP>
cudaError_t step_stored(const Grid<P>& g, const FaceVel<P, LERP>& u, const FaceVel<P, LERP>& v,
                        const FaceVel<P, LERP>& w, const P* Tm1, const P* T, P* Tp1, StepCoef c, bool implz,
                        cudaStream_t st)
{
    dim3 blk(64, 4);
    dim3 grd((g.Nx + blk.x - 1) / blk.x, (g.Ny + blk.y - 1) / blk.y, g.Nz);
    const P a = (P)c.a, b = (P)c.b, gdt = (P)c.gdt;
    if (!LERP && !implz && !g.order4 && !g.walls) {
        if constexpr (sizeof(P) == 4) {
            // whole quads, 16-byte aligned
            const uintptr_t all = reinterpret_cast<uintptr_t>(u.A) | reinterpret_cast<uintptr_t>(v.A) |
                                  reinterpret_cast<uintptr_t>(w.A) | reinterpret_cast<uintptr_t>(Tm1) |
                                  reinterpret_cast<uintptr_t>(T) | reinterpret_cast<uintptr_t>(Tp1);
            const size_t quads = (size_t)(g.Nx / 4) * g.Ny;
            // fewer layers per thread where the grid would not give every SM 256 threads
            int march = kMarch;
            while (march > 1 && quads * ((g.Nz + march - 1) / march) < 152 * 256) march /= 2;
            const size_t layers = (g.Nz + march - 1) / march;
            if (g.Nx % 4 == 0 && !(all & 15) && quads < (1u << 31) && layers <= 65535)
                return launch_after(c.a == 1.0 && c.b == 0.0 ? k_step_periodic4<true> : k_step_periodic4<false>,
                                    dim3((unsigned)((quads + 127) / 128), (unsigned)layers), 128, 0, st, g, u.A, v.A, w.A,
                                    Tm1, T, Tp1, a, b, gdt, march);
        }
        const auto k = c.a == 1.0 && c.b == 0.0 ? k_step_periodic<P, true> : k_step_periodic<P, false>;
        const bool ahead = sizeof(P) == 4 || fp64_gains_ahead(reinterpret_cast<const void*>(k), grd, 256);
        return launch_after_if(ahead, k, grd, blk, 0, st, g, u.A, v.A, w.A, Tm1, T, Tp1, a, b, gdt);
    }
    if constexpr (sizeof(P) == 4) {
        // FP32 at fourth order: from 4 M cells on read-only loads gain more than an early
        // start, which does not allow them (us per step: 3.1 M cells 63.5 and 62.7,
        // 4.2 M 84.2 and 87.5, 33.6 M 638 and 683)
        if (g.order4 && (size_t)g.Nx * g.Ny * g.Nz >= kAloneCells) {
            (implz ? k_step_stored_alone<P, true, LERP, true> : k_step_stored_alone<P, false, LERP, true>)
                <<<grd, blk, 0, st>>>(g, u, v, w, Tm1, T, Tp1, a, b, gdt);
            return cudaGetLastError();
        }
    }
    // (with implicit z the solve lies between the steps)
    const auto k = g.order4 ? (implz ? k_step_stored<P, true, LERP, true> : k_step_stored<P, false, LERP, true>)
                            : (implz ? k_step_stored<P, true, LERP, false> : k_step_stored<P, false, LERP, false>);
    const bool ahead = sizeof(P) == 4 || implz || fp64_gains_ahead(reinterpret_cast<const void*>(k), grd, 256);
    return launch_after_if(ahead, k, grd, blk, 0, st, g, u, v, w, Tm1, T, Tp1, a, b, gdt);
}

__global__ void k_lerp(const float* A, const float* B, float alpha, float* __restrict__ out,
                       size_t n)
{
    after_previous();
    let_next();
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x) {
        const float a = A[t];
        out[t] = a + alpha * (B[t] - a);
    }
}

}  // namespace

cudaError_t launch_lerp_f32(const float* A, const float* B, double alpha, float* out, size_t n, cudaStream_t st)
{
    if (!n) return cudaSuccess;
    const size_t want = (n + 255) / 256;
    const unsigned blocks = (unsigned)(want < 152 * 16 ? want : 152 * 16);
    return launch_after(k_lerp, blocks, 256, 0, st, A, B, (float)alpha, out, n);
}

bool fp64_gains_ahead(const void* kernel, dim3 grid, int threads)
{
    static std::mutex mu;
    static std::unordered_map<const void*, int> resident;     // blocks per SM
    int r = 0;
    {
        std::lock_guard<std::mutex> lock(mu);
        const auto it = resident.find(kernel);
        if (it != resident.end()) {
            r = it->second;
        } else if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&r, kernel, threads, 0) == cudaSuccess) {
            resident[kernel] = r;
        } else {
            cudaGetLastError();
            return true;
        }
    }
    const size_t blocks = (size_t)grid.x * grid.y * grid.z, slots = (size_t)152 * r;
    return 2 * blocks <= slots || 4 * blocks > 3 * slots;
}

template <typename P>
cudaError_t launch_step_stored(const Grid<P>& g, const P* Us, const P* Vs, const P* Ws, const P* Tm1,
                               const P* T, P* Tp1, StepCoef c, bool implz, cudaStream_t st)
{
    return step_stored<P, false>(g, {Us, nullptr, P(0)}, {Vs, nullptr, P(0)}, {Ws, nullptr, P(0)}, Tm1, T, Tp1,
                                 c, implz, st);
}

template <typename P>
cudaError_t launch_step_stored_lerp(const Grid<P>& g, const P* const velA[3], const P* const velB[3], double alpha,
                                    const P* Tm1, const P* T, P* Tp1, StepCoef c, bool implz, cudaStream_t st)
{
    const P al = (P)alpha;
    return step_stored<P, true>(g, {velA[0], velB[0], al}, {velA[1], velB[1], al}, {velA[2], velB[2], al}, Tm1,
                                T, Tp1, c, implz, st);
}

// The largest table is 3 x 1280 doubles (30 KB of the 32,764 bytes of parameters a
// launch may have); the small one keeps the usual launches short.
bool zsolve_needs_work(int Nz) { return Nz > 1280; }

template <typename P>
cudaError_t launch_zsolve(const Grid<P>& g, P* Tp1, double half_gdt, const double* cdn, const double* cup, P* work,
                          cudaStream_t st)
{
    if (g.Nz <= 256) return zsolve_table<P, 256>(g, Tp1, half_gdt, cdn, cup, st);
    if (!zsolve_needs_work(g.Nz)) return zsolve_table<P, 1280>(g, Tp1, half_gdt, cdn, cup, st);
    dim3 blk(128);
    dim3 grd((g.Nx + 127) / 128, g.Ny);
    k_zsolve_tall<P><<<grd, blk, 0, st>>>(g, Tp1, (P)half_gdt, work);
    return cudaGetLastError();
}

template cudaError_t launch_step_stored<double>(const Grid<double>&, const double*, const double*,
                                                const double*, const double*, const double*, double*,
                                                StepCoef, bool, cudaStream_t);
template cudaError_t launch_step_stored<float>(const Grid<float>&, const float*, const float*, const float*,
                                               const float*, const float*, float*, StepCoef, bool,
                                               cudaStream_t);
template cudaError_t launch_step_stored_lerp<double>(const Grid<double>&, const double* const[3],
                                                     const double* const[3], double, const double*,
                                                     const double*, double*, StepCoef, bool, cudaStream_t);
template cudaError_t launch_step_stored_lerp<float>(const Grid<float>&, const float* const[3], const float* const[3],
                                                    double, const float*, const float*, float*, StepCoef, bool,
                                                    cudaStream_t);
template cudaError_t launch_zsolve<double>(const Grid<double>&, double*, double, const double*, const double*, double*,
                                           cudaStream_t);
template cudaError_t launch_zsolve<float>(const Grid<float>&, float*, double, const double*, const double*, float*,
                                          cudaStream_t);

}  // namespace mr
