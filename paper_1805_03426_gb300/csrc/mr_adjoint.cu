// Hand-written discrete adjoint of the scalar path (stored-velocity mode).
//
// Loss L = sum_s wnu[s] Nu_bot(T^s) + wvar[s] Var(T^s) over the levels
// s = 0..S of an S-step run.  The forward scheme (Section 2.2, Eq. 5) is
//   T^{s+1} = a_s T^{s-1} + b_s T^s + g_s dt [C(u; T^s) + D(T^{s-1})],
// affine in T for fixed u and bilinear in (u, T) through C.  The backward sweep
// carries mu = lambda / Vol (adjoint per unit volume):
//   mu^s     += b_s mu^{s+1} + g_s dt C^T mu^{s+1}
//   mu^{s-1}  = direct_{s-1} + a_s mu^{s+1} + g_s dt D^T mu^{s+1}
// (Euler start: mu^0 += mu^1 + dt (C^T + D^T) mu^1).  In this form D^T is the
// forward diffusion stencil itself (D is symmetric in the volume-weighted inner
// product, plate values zero), and C^T is gathered per cell:
//   (C^T mu)_c = sum_faces (A_f / Vol_c) u_f w_{c,f} (mu_R - mu_L),
// w_{c,f} being the weight of T_c in the face value T_f.  The face gradient is
//   dL/du_f += g_s dt A_f T^s_f (mu_R - mu_L),
// accumulated by the cell that owns the face (its west, south and bottom
// faces), so no atomics are needed: in the working precision over one
// checkpoint segment, then added into FP64 totals (GB300's FP64 pipe is a
// small fraction of its FP32 one).  The coarse gradient is the
// transpose of the refinement (Section 3.2), applied once at the end (it is
// linear and fixed, so sum_s P^T g_s = P^T sum_s g_s).
//
// Checkpoints: the forward stores (T^{s-1}, T^s) every k steps; the backward
// recomputes each segment's levels from its checkpoint before sweeping it.
#include <math.h>

#include <algorithm>
#include <vector>

#include "mr_internal.cuh"

namespace mr {
namespace {

constexpr int kThreads = 256;
inline unsigned nblk(size_t n) { return (unsigned)((n + kThreads - 1) / kThreads); }

// direct term of one level: mu = s_nu * (k == 0) + s_var * (T - mean)
template <typename P>
__global__ void k_adj_direct(Grid<P> g, const P* __restrict__ T, double s_nu_bottom, double s_var, double mean,
                             P* __restrict__ mu)
{
    const size_t plane = (size_t)g.Nx * g.Ny, n = plane * g.Nz;
    for (size_t m = (size_t)blockIdx.x * blockDim.x + threadIdx.x; m < n; m += (size_t)gridDim.x * blockDim.x) {
        double v = 0.0;
        if (m < plane) v += s_nu_bottom;
        if (s_var != 0.0) v += s_var * ((double)T[m] - mean);
        mu[m] = (P)v;
    }
}

// One backward step (thread per cell).  Mn = mu^{s+1} (complete), Mc = mu^s
// (accumulated), Mp = mu^{s-1} (written: its direct term -- s_nu on the bottom
// layer, s_var (T^{s-1} - mean) everywhere -- plus this step's share);
// EULER: the s = 0 start, which feeds everything into Mc.
template <typename P, bool EULER>
__global__ void __launch_bounds__(256) k_adj_step(Grid<P> g, const P* __restrict__ Us, const P* __restrict__ Vs,
                                                  const P* __restrict__ Ws, const P* __restrict__ T,
                                                  const P* __restrict__ Tprev, const P* __restrict__ Mn,
                                                  P* __restrict__ Mc, P* __restrict__ Mp, double s_nu, double s_var,
                                                  double mean_prev, P* __restrict__ gU,
                                                  P* __restrict__ gV, P* __restrict__ gW, P a, P b, P gdt)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= g.Nx || j >= g.Ny) return;
    const size_t plane = (size_t)g.Nx * g.Ny;
    const size_t m = (size_t)k * plane + (size_t)j * g.Nx + i;
    const P half = P(0.5);
    const P mc = Mn[m], tc = T[m];
    P ct = 0, dxs = 0, dys = 0, dzs = 0, cy = 0, cz = 0;
    const size_t urow = ((size_t)k * g.Ny + j) * g.ufx;
    // x faces
    if (!(g.walls && i == 0)) {
        const int iw = (i == 0) ? g.Nx - 1 : i - 1;
        const size_t mw = m - i + iw;
        const P uw = Us[urow + i], mw_ = Mn[mw];
        ct += uw * half * (mc - mw_);
        dxs -= mc - mw_;
        gU[urow + i] += gdt * (g.dy * g.dz[k]) * (half * (T[mw] + tc)) * (mc - mw_);
    }
    if (!(g.walls && i == g.Nx - 1)) {
        const int ie = (i == g.Nx - 1) ? 0 : i + 1;
        const int fe = g.walls ? i + 1 : ie;
        const P me_ = Mn[m - i + ie];
        ct += Us[urow + fe] * half * (me_ - mc);
        dxs += me_ - mc;
    }
    // y faces
    const size_t vrow = ((size_t)k * g.vfy + j) * g.Nx + i;
    if (!(g.walls && j == 0)) {
        const int js = (j == 0) ? g.Ny - 1 : j - 1;
        const size_t ms = m + ((ptrdiff_t)js - j) * g.Nx;
        const P ms_ = Mn[ms];
        cy += Vs[vrow] * half * (mc - ms_);
        dys -= mc - ms_;
        gV[vrow] += gdt * (g.dx * g.dz[k]) * (half * (T[ms] + tc)) * (mc - ms_);
    }
    if (!(g.walls && j == g.Ny - 1)) {
        const int jn = (j == g.Ny - 1) ? 0 : j + 1;
        const int fn = g.walls ? j + 1 : jn;
        const P mn_ = Mn[m + ((ptrdiff_t)jn - j) * g.Nx];
        cy += Vs[((size_t)k * g.vfy + fn) * g.Nx + i] * half * (mn_ - mc);
        dys += mn_ - mc;
    }
    // z faces (plates: no advective flux, Dirichlet / zero-flux diffusion with zero plate value)
    if (k > 0) {
        const P mb_ = Mn[m - plane];
        cz += Ws[m] * g.whi[k] * (mc - mb_);
        dzs -= g.cdn[k] * (mc - mb_);
        gW[m] += gdt * (g.dx * g.dy) * (g.wlo[k] * T[m - plane] + g.whi[k] * tc) * (mc - mb_);
    } else {
        dzs -= g.cdn[0] * mc;
    }
    if (k < g.Nz - 1) {
        const P mt_ = Mn[m + plane];
        cz += Ws[m + plane] * g.wlo[k + 1] * (mt_ - mc);
        dzs += g.cup[k] * (mt_ - mc);
    } else {
        dzs -= g.cup[k] * mc;
    }
    const P CT = ct * g.inv_dx + cy * g.inv_dy + cz * g.inv_dz[k];
    const P DT = g.kx2 * dxs + g.ky2 * dys + dzs;
    if (EULER) {
        Mc[m] = Mc[m] + mc + gdt * (CT + DT);
    } else {
        Mc[m] = Mc[m] + b * mc + gdt * CT;
        double d = (k == 0) ? s_nu : 0.0;
        if (s_var != 0.0) d += s_var * ((double)Tprev[m] - mean_prev);
        Mp[m] = (P)d + a * mc + gdt * DT;
    }
}

// The same backward step for periodic x and y, folded for the FP64 pipe
// like the forward's k_step_periodic (about 42 FP operations per cell instead
// of 60): the adjoint differences of the six neighbours are formed once, the
// planes beyond the plates read as zero (which gives the plate terms of D^T),
// the z weights times 1/dz come from g.lz, and the face-gradient factors
// gdt A_f / 2 (x, y) and gdt A_z arrive as cx, cy, cz per unit dz.
template <typename P, bool EULER>
__global__ void __launch_bounds__(256) k_adj_step_periodic(Grid<P> g, const P* Us, const P* Vs, const P* Ws,
                                                           const P* T, const P* Tprev, const P* Mn, P* __restrict__ Mc,
                                                           P* __restrict__ Mp, double s_nu, double s_var,
                                                           double mean_prev, P* __restrict__ gU, P* __restrict__ gV,
                                                           P* __restrict__ gW, P a, P b, P gdt, P cx, P cy, P cz)
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
    const bool lo = k > 0, hi = k < g.Nz - 1;
    const P mc = Mn[m], tc = T[m];
    const P dw = mc - Mn[mw], de = Mn[me] - mc, ds = mc - Mn[ms], dn = Mn[mn] - mc;
    const P db = mc - (lo ? Mn[m - plane] : P(0)), dt = (hi ? Mn[m + plane] : P(0)) - mc;
    const size_t urow = ((size_t)k * g.Ny + j) * g.Nx, vrow = (size_t)k * plane;
    const P uw = Us[urow + i], wb = Ws[m];
    const P CT = g.hx * (uw * dw + Us[urow + ie] * de) + g.hy * (Vs[vrow + row + i] * ds + Vs[vrow + (size_t)jn * g.Nx + i] * dn) +
                 ((wb * L[1]) * db - (Ws[m + plane] * L[2]) * dt);
    const P DT = g.kx2 * (de - dw) + g.ky2 * (dn - ds) + L[5] * dt - L[4] * db;
    // face gradients of the cell's west, south and bottom faces
    const P dzk = g.dz[k];
    gU[urow + i] += (cx * dzk) * (T[mw] + tc) * dw;
    gV[vrow + row + i] += (cy * dzk) * (T[ms] + tc) * ds;
    if (lo) gW[m] += (cz * dzk) * (L[0] * T[m - plane] + L[1] * tc) * db;
    if (EULER) {
        Mc[m] = Mc[m] + mc + gdt * (CT + DT);
    } else {
        Mc[m] = Mc[m] + b * mc + gdt * CT;
        double d = (k == 0) ? s_nu : 0.0;
        if (s_var != 0.0) d += s_var * ((double)Tprev[m] - mean_prev);
        Mp[m] = (P)d + a * mc + gdt * DT;
    }
}

// The FP32 form of k_adj_step_periodic on rows of whole quads: a thread marches
// four cells of a row through a few layers (16-byte loads, the planes of mu, T and
// W above become the current ones in registers).  The operations are those of
// k_adj_step_periodic in its order and with its contractions (spelt out), so that
// the gradients, which magnify rounding, are the same to the last bit.
// 128 x 128 x 96 cells: the 40-step gradient (three of its launches per step are this
// kernel and the FP32 step) 2.6 ms, 3.2 ms with a cell per thread in both.
__device__ __forceinline__ float get(const float4& v, int q) { return q == 0 ? v.x : (q == 1 ? v.y : (q == 2 ? v.z : v.w)); }
__device__ __forceinline__ void put(float4& v, int q, float x) { (q == 0 ? v.x : (q == 1 ? v.y : (q == 2 ? v.z : v.w))) = x; }
template <bool EULER>
__global__ void __launch_bounds__(128) k_adj_step_periodic4(Grid<float> g, const float* Us, const float* Vs,
                                                            const float* Ws, const float* T, const float* Tprev,
                                                            const float* Mn, float* __restrict__ Mc,
                                                            float* __restrict__ Mp, double s_nu, double s_var,
                                                            double mean_prev, float* __restrict__ gU, float* __restrict__ gV,
                                                            float* __restrict__ gW, float a, float b, float gdt, float cx,
                                                            float cy, float cz, int march)
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
    float4 mb = k0 > 0 ? quad(Mn + m - plane + row) : zero, tb = k0 > 0 ? quad(T + m - plane + row) : zero;
    float4 mc = quad(Mn + m + row), wb = quad(Ws + m + row);
    for (int k = k0; k < k1; ++k, m += plane) {
        const float* L = g.lz + 8 * k;
        const bool lo = k > 0, hi = k < g.Nz - 1;
        const float4 tc = quad(T + m + row), mt = hi ? quad(Mn + m + plane + row) : zero, wt = quad(Ws + m + plane + row);
        const float4 ms = quad(Mn + m + south), mn = quad(Mn + m + north), ts = quad(T + m + south);
        const float4 u = quad(Us + m + row), vs = quad(Vs + m + row), vn = quad(Vs + m + north);
        const float mw = Mn[m + west], me = Mn[m + east], tw = T[m + west], ue = Us[m + east];
        float4 hu = quad(gU + m + row), hv = quad(gV + m + row), hw = lo ? quad(gW + m + row) : zero;
        float4 oc = quad(Mc + m + row), op = zero;
        const float dzk = g.dz[k], ex = __fmul_rn(cx, dzk), ey = __fmul_rn(cy, dzk), ez = __fmul_rn(cz, dzk);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float M = get(mc, q), Tc = get(tc, q);
            const float dw = __fsub_rn(M, q ? get(mc, q - 1) : mw), de = __fsub_rn(q < 3 ? get(mc, q + 1) : me, M);
            const float ds = __fsub_rn(M, get(ms, q)), dn = __fsub_rn(get(mn, q), M);
            const float db = __fsub_rn(M, get(mb, q)), dt = __fsub_rn(get(mt, q), M);
            const float X = __fmaf_rn(get(u, q), dw, __fmul_rn(q < 3 ? get(u, q + 1) : ue, de));
            const float Y = __fmaf_rn(get(vs, q), ds, __fmul_rn(get(vn, q), dn));
            const float Z = __fmaf_rn(__fmul_rn(get(wb, q), L[1]), db, -__fmul_rn(__fmul_rn(get(wt, q), L[2]), dt));
            const float CT = __fadd_rn(__fmaf_rn(g.hx, X, __fmul_rn(g.hy, Y)), Z);
            float DT = __fmaf_rn(g.kx2, __fsub_rn(de, dw), __fmul_rn(g.ky2, __fsub_rn(dn, ds)));
            DT = __fmaf_rn(L[5], dt, DT);
            DT = __fmaf_rn(-L[4], db, DT);
            put(hu, q, __fmaf_rn(__fmul_rn(ex, __fadd_rn(q ? get(tc, q - 1) : tw, Tc)), dw, get(hu, q)));
            put(hv, q, __fmaf_rn(__fmul_rn(ey, __fadd_rn(get(ts, q), Tc)), ds, get(hv, q)));
            if (lo)
                put(hw, q, __fmaf_rn(__fmul_rn(ez, __fmaf_rn(L[0], get(tb, q), __fmul_rn(L[1], Tc))), db, get(hw, q)));
            if (EULER) {
                put(oc, q, __fmaf_rn(gdt, __fadd_rn(CT, DT), __fadd_rn(get(oc, q), M)));
            } else {
                put(oc, q, __fmaf_rn(gdt, CT, __fmaf_rn(b, M, get(oc, q))));
                double d = (k == 0) ? s_nu : 0.0;
                if (s_var != 0.0) d += s_var * ((double)Tprev[m + row + q] - mean_prev);
                put(op, q, __fmaf_rn(gdt, DT, __fmaf_rn(a, M, (float)d)));
            }
        }
        *reinterpret_cast<float4*>(gU + m + row) = hu;
        *reinterpret_cast<float4*>(gV + m + row) = hv;
        if (lo) *reinterpret_cast<float4*>(gW + m + row) = hw;
        *reinterpret_cast<float4*>(Mc + m + row) = oc;
        if (!EULER) *reinterpret_cast<float4*>(Mp + m + row) = op;
        mb = mc;
        mc = mt;
        tb = tc;
        wb = wt;
    }
}

// totals (FP64) += segment sums (FP32), which are cleared
__global__ void k_flush_faces(float* __restrict__ seg, double* __restrict__ tot, size_t n)
{
    after_previous();
    let_next();
    for (size_t m = (size_t)blockIdx.x * blockDim.x + threadIdx.x; m < n; m += (size_t)gridDim.x * blockDim.x) {
        tot[m] += (double)seg[m];
        seg[m] = 0.f;
    }
}

template <typename P>
__global__ void k_times_volume(Grid<P> g, const P* __restrict__ mu, int dst_f64, void* __restrict__ out)
{
    const size_t plane = (size_t)g.Nx * g.Ny, n = plane * g.Nz;
    const double dxdy = (double)g.dx * (double)g.dy;
    for (size_t m = (size_t)blockIdx.x * blockDim.x + threadIdx.x; m < n; m += (size_t)gridDim.x * blockDim.x) {
        const double v = (double)mu[m] * dxdy * (double)g.dz[m / plane];
        if (dst_f64) ((double*)out)[m] = v;
        else ((float*)out)[m] = (float)v;
    }
}

// ------------------------------------------------------------- refinement transpose (FP64)
// The transpose of the refinement axis by axis (the stages of launch_refine in
// mr_refine.cu in reverse order).  A balance's transpose is a running sum over the
// faces it formed, which takes the place of their gradients; each neighbour then
// gathers its differences.  A split's transpose sums a coarse cell's dense values
// with the R columns first (t_p = sum_a R[a][p] x_a) and adds the three t_p to the
// window's cells with FP64 atomics, one for each coarse value at the resolution
// still left instead of nine products and atomics per dense face.
//   aUs (per coarse cell in x)  -> h_a = sum_{a' >= a} aU_a'     (h_0: aUO)
//   aVs, aWs + differences of h -> R_x^T -> aVR, aWY
//   aVR (per coarse row)        -> g_b = sum_{b' >= b} aVR_b'    (g_0: aVZ)
//   aUO, aWY + differences of g -> R_y^T -> aUZ, aWC
//   aWC (per coarse slab)       -> S_c = dz_c sum_{c' <= c} aWC_c', their last sum to gW
//   aUZ, aVZ + differences of S -> R_z^T -> gU, gV
// 128 x 128 x 96 dense cells at M = 2: 91 us; 300 us face by face, nine atomics each.

struct Transpose {
    Grid<double> g;
    double *aUs, *aVs, *aWs;         // dense face gradients (consumed)
    double *aVR, *aWY, *aUZ, *aWC;   // zero before
    double *gU, *gV, *gW;            // zero before
};

__device__ __forceinline__ void add(double* p, double v) { atomicAdd(p, v); }

// Running sums of the x balances: thread per (layer, dense row, coarse column).
__global__ void k_t_sum_x(const Transpose A)
{
    const Grid<double>& g = A.g;
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x, n = (size_t)g.Nz * g.Ny * g.nx;
    if (t >= n) return;
    const size_t row = t / g.nx;
    double* u = A.aUs + row * g.ufx + (t - row * g.nx) * g.mx;
    double h = u[g.mx - 1];
    for (int a = g.mx - 2; a >= 0; --a) u[a] = h += u[a];
}

// R_x^T: thread per (layer, V face row, coarse column), then (plane, dense row, coarse column).
__global__ void k_t_split_x(const Transpose A)
{
    const Grid<double>& g = A.g;
    const size_t nv = (size_t)g.Nz * g.vfy * g.nx, nw = (size_t)(g.Nz + 1) * g.Ny * g.nx;
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nv + nw) return;
    const bool v = t < nv;
    const size_t e = v ? t : t - nv, row = e / g.nx;
    const int I = (int)(e - row * g.nx), rows = v ? g.vfy : g.Ny, k = (int)(row / rows), j = (int)(row - (size_t)k * rows);
    // the two balances that read the face: with its coefficient in the first one
    const double *h0 = nullptr, *h1 = nullptr;
    double c0 = 0.0, c1 = 0.0;
    if (v) {
        const int js = j > 0 ? j - 1 : (g.walls ? -1 : g.Ny - 1);
        if (j < g.Ny) h0 = A.aUs + ((size_t)k * g.Ny + j) * g.ufx;
        if (js >= 0) h1 = A.aUs + ((size_t)k * g.Ny + js) * g.ufx;
        c0 = c1 = g.dx / g.dy;
    } else {
        if (k < g.Nz) h0 = A.aUs + ((size_t)k * g.Ny + j) * g.ufx, c0 = g.dx * g.inv_dz[k];
        if (k > 0) h1 = A.aUs + ((size_t)(k - 1) * g.Ny + j) * g.ufx, c1 = g.dx * g.inv_dz[k - 1];
    }
    const double* x = (v ? A.aVs : A.aWs) + row * g.Nx + (size_t)I * g.mx;
    const double* r = g.Rx + 3 * (size_t)I * g.mx;
    double s[3] = {0.0, 0.0, 0.0};
    for (int a = 0; a < g.mx; ++a) {
        double y = x[a];
        if (a < g.mx - 1) {
            const size_t f = (size_t)I * g.mx + a + 1;
            if (h0) y = fma(c0, h0[f], y);
            if (h1) y = fma(-c1, h1[f], y);
        }
        for (int p = 0; p < 3; ++p) s[p] = fma(r[3 * a + p], y, s[p]);
    }
    double* o = (v ? A.aVR : A.aWY) + row * g.nx;
    for (int p = 0; p < 3; ++p) add(o + g.wx[3 * I + p], s[p]);
}

// Running sums of the row balances: thread per (layer, coarse row, coarse column).
__global__ void k_t_sum_y(const Transpose A)
{
    const Grid<double>& g = A.g;
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x, n = (size_t)g.Nz * g.ny * g.nx;
    if (t >= n) return;
    const size_t row = t / g.nx, k = row / g.ny;
    double* v = A.aVR + (k * g.vfy + (row - k * g.ny) * g.my) * g.nx + (t - row * g.nx);
    double s = v[(size_t)(g.my - 1) * g.nx];
    for (int b = g.my - 2; b >= 0; --b) v[(size_t)b * g.nx] = s += v[(size_t)b * g.nx];
}

// R_y^T: thread per (layer, coarse row, U face column), then (plane, coarse row, coarse column).
__global__ void k_t_split_y(const Transpose A)
{
    const Grid<double>& g = A.g;
    const size_t nu = (size_t)g.Nz * g.ny * g.cux, nw = (size_t)(g.Nz + 1) * g.ny * g.nx;
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nu + nw) return;
    const bool u = t < nu;
    const int cols = u ? g.cux : g.nx;
    const size_t e = u ? t : t - nu, row = e / cols;
    const int I = (int)(e - row * cols), k = (int)(row / g.ny), J = (int)(row - (size_t)k * g.ny);
    const double *g0 = nullptr, *g1 = nullptr;            // running sums of V, [dense row][coarse column]
    double c0 = 0.0, c1 = 0.0;
    if (u) {
        const int Iw = I > 0 ? I - 1 : (g.walls ? -1 : g.nx - 1);
        if (I < g.nx) g0 = A.aVR + (size_t)k * g.vfy * g.nx + I;
        if (Iw >= 0) g1 = A.aVR + (size_t)k * g.vfy * g.nx + Iw;
        c0 = c1 = g.dy / g.DX;
    } else {
        if (k < g.Nz) g0 = A.aVR + (size_t)k * g.vfy * g.nx + I, c0 = g.dy * g.inv_dz[k];
        if (k > 0) g1 = A.aVR + (size_t)(k - 1) * g.vfy * g.nx + I, c1 = g.dy * g.inv_dz[k - 1];
    }
    // U's values are the running sums' first ones of each coarse cell
    const double* x = u ? A.aUs + (size_t)k * g.Ny * g.ufx + (size_t)I * g.mx : A.aWY + (size_t)k * g.Ny * g.nx + I;
    const size_t xs = u ? g.ufx : g.nx;
    const double* r = g.Ry + 3 * (size_t)J * g.my;
    double s[3] = {0.0, 0.0, 0.0};
    for (int b = 0; b < g.my; ++b) {
        const size_t j = (size_t)J * g.my + b;
        double y = x[j * xs];
        if (b < g.my - 1) {
            if (g0) y = fma(c0, g0[(j + 1) * g.nx], y);
            if (g1) y = fma(-c1, g1[(j + 1) * g.nx], y);
        }
        for (int p = 0; p < 3; ++p) s[p] = fma(r[3 * b + p], y, s[p]);
    }
    double* o = (u ? A.aUZ : A.aWC) + (size_t)k * g.ny * cols + I;
    for (int p = 0; p < 3; ++p) add(o + (size_t)g.wy[3 * J + p] * cols, s[p]);
}

// Running sums of the slab balances, and W's gradient: thread per coarse cell.
__global__ void k_t_sum_z(const Transpose A)
{
    const Grid<double>& g = A.g;
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x, plane = (size_t)g.ny * g.nx, n = (size_t)g.nz * plane;
    if (t >= n) return;
    const size_t K = t / plane;
    double* w = A.aWC + K * g.mz * plane + (t - K * plane);
    add(A.gW + t, w[0]);
    if (K + 1 == (size_t)g.nz) add(A.gW + t + plane, w[(size_t)g.mz * plane]);
    double s = 0.0;
    for (int c = 1; c < g.mz; ++c) {
        s += w[(size_t)c * plane];
        w[(size_t)c * plane] = s * g.dz[K * g.mz + c];
    }
    add(A.gW + t + plane, s);
}

// R_z^T: thread per coarse U face, then per coarse V face.
__global__ void k_t_split_z(const Transpose A)
{
    const Grid<double>& g = A.g;
    const size_t pu = (size_t)g.ny * g.cux, pv = (size_t)g.cvy * g.nx, nu = g.nz * pu, nv = g.nz * pv;
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nu + nv) return;
    const bool u = t < nu;
    const size_t e = u ? t : t - nu, pl = u ? pu : pv;
    const int K = (int)(e / pl), cols = u ? g.cux : g.nx, J = (int)(e % pl / cols), I = (int)(e % pl % cols);
    // the cells east / north (coefficient -) and west / south (+) of the face
    const int Ie = u ? (I < g.nx ? I : -1) : I, Iw = u ? (I > 0 ? I - 1 : (g.walls ? -1 : g.nx - 1)) : I;
    const int Jn = u ? J : (J < g.ny ? J : -1), Js = u ? J : (J > 0 ? J - 1 : (g.walls ? -1 : g.ny - 1));
    const double c = u ? 1.0 / g.DX : 1.0 / g.DY;
    const size_t wp = (size_t)g.ny * g.nx;
    const double* x = u ? A.aUZ + (size_t)J * g.cux + I : A.aVR + (size_t)J * g.my * g.nx + I;
    const size_t xs = u ? pu : (size_t)g.vfy * g.nx;
    double s[3] = {0.0, 0.0, 0.0};
    for (int b = 0; b < g.mz; ++b) {
        const size_t k = (size_t)K * g.mz + b;
        double y = x[k * xs];
        if (b > 0) {
            const double* S = A.aWC + k * wp;
            double d = 0.0;
            if (Iw >= 0 && Js >= 0) d += S[(size_t)Js * g.nx + Iw];
            if (Ie >= 0 && Jn >= 0) d -= S[(size_t)Jn * g.nx + Ie];
            y = fma(c, d, y);
        }
        for (int p = 0; p < 3; ++p) s[p] = fma(g.Rz[3 * k + p], y, s[p]);
    }
    double* o = (u ? A.gU : A.gV) + e % pl;
    for (int p = 0; p < 3; ++p) add(o + (size_t)g.wz[3 * K + p] * pl, s[p]);
}

}  // namespace

size_t transpose_work(const Grid<double>& g)
{
    return (size_t)g.Nz * g.vfy * g.nx + (size_t)(g.Nz + 1) * g.ny * g.nx;
}
size_t transpose_wy(const Grid<double>& g) { return (size_t)(g.Nz + 1) * g.Ny * g.nx; }

// P^T: dense face gradients (U, V and W one after the other; consumed) -> coarse
// gradients (zeroed first).  The gradient of the faces refined in z alone takes the
// place of the V and W faces, which are no longer needed by then.
cudaError_t launch_refine_transpose(const Grid<double>& g, double* faces, double* work, double* wy, double* gU, double* gV,
                                    double* gW, size_t ncU, size_t ncV, size_t ncW, cudaStream_t st)
{
    Transpose A{g, faces, nullptr, nullptr, work, wy, nullptr, nullptr, gU, gV, gW};
    A.aVs = faces + (size_t)g.Nz * g.Ny * g.ufx;
    A.aWs = A.aVs + (size_t)g.Nz * g.vfy * g.Nx;
    A.aWC = work + (size_t)g.Nz * g.vfy * g.nx;
    A.aUZ = A.aVs;
    cudaError_t e;
    if ((e = cudaMemsetAsync(gU, 0, ncU * 8, st)) || (e = cudaMemsetAsync(gV, 0, ncV * 8, st)) ||
        (e = cudaMemsetAsync(gW, 0, ncW * 8, st)) || (e = cudaMemsetAsync(work, 0, transpose_work(g) * 8, st)) ||
        (e = cudaMemsetAsync(wy, 0, transpose_wy(g) * 8, st)))
        return e;
    k_t_sum_x<<<nblk((size_t)g.Nz * g.Ny * g.nx), kThreads, 0, st>>>(A);
    k_t_split_x<<<nblk((size_t)g.Nz * g.vfy * g.nx + (size_t)(g.Nz + 1) * g.Ny * g.nx), kThreads, 0, st>>>(A);
    if ((e = cudaMemsetAsync(A.aUZ, 0, (size_t)g.Nz * g.ny * g.cux * 8, st))) return e;
    k_t_sum_y<<<nblk((size_t)g.Nz * g.ny * g.nx), kThreads, 0, st>>>(A);
    k_t_split_y<<<nblk((size_t)g.Nz * g.ny * g.cux + (size_t)(g.Nz + 1) * g.ny * g.nx), kThreads, 0, st>>>(A);
    k_t_sum_z<<<nblk((size_t)g.nz * g.ny * g.nx), kThreads, 0, st>>>(A);
    k_t_split_z<<<nblk(g.nz * ((size_t)g.ny * g.cux + (size_t)g.cvy * g.nx)), kThreads, 0, st>>>(A);
    return cudaGetLastError();
}

template <typename P>
cudaError_t launch_adj_direct(const Grid<P>& g, const P* T, double s_nu_bottom, double s_var, double mean, P* mu,
                              cudaStream_t st)
{
    k_adj_direct<P><<<152 * 8, kThreads, 0, st>>>(g, T, s_nu_bottom, s_var, mean, mu);
    return cudaGetLastError();
}

cudaError_t launch_flush_faces(float* seg, double* tot, size_t n, cudaStream_t st)
{
    return launch_after(k_flush_faces, 152 * 8, kThreads, 0, st, seg, tot, n);
}

template <typename P>
cudaError_t launch_adj_step(const Grid<P>& g, const P* Us, const P* Vs, const P* Ws, const P* T, const P* Tprev,
                            const P* Mn, P* Mc, P* Mp, double s_nu, double s_var, double mean_prev, P* gU,
                            P* gV, P* gW, StepCoef c, bool euler, cudaStream_t st)
{
    dim3 blk(64, 4);
    dim3 grd((g.Nx + blk.x - 1) / blk.x, (g.Ny + blk.y - 1) / blk.y, g.Nz);
    if (!g.walls) {
        // face-gradient factors: gdt dy / 2 and gdt dx / 2 per unit dz_k (x and y
        // faces), gdt dx dy (z faces, times dz_k in the kernel to undo the 1/dz_k
        // of the g.lz weights)
        const double dx = (double)g.dx, dy = (double)g.dy;
        const P cx = (P)(c.gdt * 0.5 * dy), cy = (P)(c.gdt * 0.5 * dx), cz = (P)(c.gdt * dx * dy);
        if constexpr (sizeof(P) == 4) {
            // whole quads, 16-byte aligned; fewer layers per thread where the grid would
            // not give every SM 256 threads
            const void* ptrs[] = {Us, Vs, Ws, T, Tprev, Mn, Mc, Mp, gU, gV, gW};
            uintptr_t all = 0;
            for (const void* p : ptrs) all |= reinterpret_cast<uintptr_t>(p);
            const size_t quads = (size_t)(g.Nx / 4) * g.Ny;
            int march = 4;
            while (march > 1 && quads * ((g.Nz + march - 1) / march) < 152 * 256) march /= 2;
            const size_t layers = (g.Nz + march - 1) / march;
            if (g.Nx % 4 == 0 && !(all & 15) && quads < (1u << 31) && layers <= 65535)
                return launch_after(euler ? k_adj_step_periodic4<true> : k_adj_step_periodic4<false>,
                                    dim3((unsigned)((quads + 127) / 128), (unsigned)layers), 128, 0, st, g, Us, Vs, Ws, T,
                                    Tprev, Mn, Mc, Mp, s_nu, s_var, mean_prev, gU, gV, gW, (P)c.a, (P)c.b, (P)c.gdt, cx, cy,
                                    cz, march);
        }
        const auto k = euler ? k_adj_step_periodic<P, true> : k_adj_step_periodic<P, false>;
        const bool ahead = sizeof(P) == 4 || fp64_gains_ahead(reinterpret_cast<const void*>(k), grd, 256);
        return launch_after_if(ahead, k, grd, blk, 0, st, g, Us, Vs, Ws, T, Tprev, Mn, Mc, Mp, s_nu, s_var, mean_prev, gU, gV,
                               gW, (P)c.a, (P)c.b, (P)c.gdt, cx, cy, cz);
    }
    if (euler)
        k_adj_step<P, true><<<grd, blk, 0, st>>>(g, Us, Vs, Ws, T, Tprev, Mn, Mc, Mp, s_nu, s_var, mean_prev, gU, gV,
                                                 gW, (P)c.a, (P)c.b, (P)c.gdt);
    else
        k_adj_step<P, false><<<grd, blk, 0, st>>>(g, Us, Vs, Ws, T, Tprev, Mn, Mc, Mp, s_nu, s_var, mean_prev, gU,
                                                  gV, gW, (P)c.a, (P)c.b, (P)c.gdt);
    return cudaGetLastError();
}

template <typename P>
cudaError_t launch_times_volume(const Grid<P>& g, const P* mu, int dst_dtype, void* out, cudaStream_t st)
{
    k_times_volume<P><<<152 * 8, kThreads, 0, st>>>(g, mu, dst_dtype == MR_F64 ? 1 : 0, out);
    return cudaGetLastError();
}

#define MR_INST(P)                                                                                                 \
    template cudaError_t launch_adj_direct<P>(const Grid<P>&, const P*, double, double, double, P*, cudaStream_t); \
    template cudaError_t launch_adj_step<P>(const Grid<P>&, const P*, const P*, const P*, const P*, const P*,        \
                                            const P*, P*, P*, double, double, double, P*, P*, P*,                  \
                                            StepCoef, bool, cudaStream_t);                                         \
    template cudaError_t launch_times_volume<P>(const Grid<P>&, const P*, int, void*, cudaStream_t);
MR_INST(double)
MR_INST(float)
#undef MR_INST

}  // namespace mr
