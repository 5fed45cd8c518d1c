// Divergence-free refinement of the coarse staggered velocity onto the dense
// grid (Section 3.2), used by MR_VEL_STORED and to export dense faces.  The fused
// FP32 step kernel (mr_fused.cu) performs the same stages inside shared memory
// instead.  Two chains: launch_refine, axis by axis with intermediates at coarse
// resolution in the axes not yet refined (below), for FP64 handles, and
// launch_refine_in_place, whose intermediates live in the outputs, for callers with
// next to no memory and for FP32 handles: another order of the operations would
// change the FP32 faces in their last bits, which the FP32 adjoint magnifies to
// 2e-5 of the coarse gradients (its own error against FP64 being 6e-5), and the
// runs are to stay comparable.
//
// Stages (3-D reading of the paper's 2-D procedure, z first, then y, then x):
//   0  every coarse face value is split over its sub-faces with the tensor
//      product of the two tangential R matrices (V_s = R V, R = A_s A^-1);
//   Z  per coarse cell, the full-area W on the inner dense z-planes follows
//      from the mass balance of each dense slab, top-down, and is split over
//      the sub-faces with R_x (x) R_y applied to the neighbouring columns;
//   Y  per dense layer, the full-width V on the inner y-planes follows from
//      the balance of each row, south to north, and is split along x with R_x;
//   X  per dense row, U on the inner x-faces follows from each dense cell's
//      balance, west to east.
#include <algorithm>

#include "mr_internal.cuh"

namespace mr {
namespace {

constexpr int kThreads = 256;

inline unsigned blocks_for(size_t n) { return (unsigned)((n + kThreads - 1) / kThreads); }

// Stage 0, x-normal faces on the coarse x-planes: thread per (k, j, I).
template <typename P>
__global__ void k_outer_u(Grid<P> g, const P* __restrict__ U, P* __restrict__ Us)
{
    size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    size_t n = (size_t)g.Nz * g.Ny * g.cux;
    if (t >= n) return;
    int I = (int)(t % g.cux);
    int j = (int)((t / g.cux) % g.Ny);
    int k = (int)(t / ((size_t)g.cux * g.Ny));
    int J = j / g.my, K = k / g.mz;
    P s = P(0);
    for (int p = 0; p < 3; ++p) {
        int Jp = g.wy[3 * J + p];
        for (int q = 0; q < 3; ++q) {
            int Kq = g.wz[3 * K + q];
            s += g.Ry[3 * j + p] * g.Rz[3 * k + q] * U[((size_t)Kq * g.ny + Jp) * g.cux + I];
        }
    }
    Us[((size_t)k * g.Ny + j) * g.ufx + (size_t)I * g.mx] = s;
}

// Stage 0, y-normal faces on the coarse y-planes: thread per (k, J, i).
template <typename P>
__global__ void k_outer_v(Grid<P> g, const P* __restrict__ V, P* __restrict__ Vs)
{
    size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    size_t n = (size_t)g.Nz * g.cvy * g.Nx;
    if (t >= n) return;
    int i = (int)(t % g.Nx);
    int J = (int)((t / g.Nx) % g.cvy);
    int k = (int)(t / ((size_t)g.Nx * g.cvy));
    int I = i / g.mx, K = k / g.mz;
    P s = P(0);
    for (int p = 0; p < 3; ++p) {
        int Ip = g.wx[3 * I + p];
        for (int q = 0; q < 3; ++q) {
            int Kq = g.wz[3 * K + q];
            s += g.Rx[3 * i + p] * g.Rz[3 * k + q] * V[((size_t)Kq * g.cvy + J) * g.nx + Ip];
        }
    }
    Vs[((size_t)k * g.vfy + (size_t)J * g.my) * g.Nx + i] = s;
}

// Stage 0, z-normal faces on the coarse z-planes: thread per (K, j, i).
template <typename P>
__global__ void k_outer_w(Grid<P> g, const P* __restrict__ W, P* __restrict__ Ws)
{
    size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    size_t n = (size_t)(g.nz + 1) * g.Ny * g.Nx;
    if (t >= n) return;
    int i = (int)(t % g.Nx);
    int j = (int)((t / g.Nx) % g.Ny);
    int K = (int)(t / ((size_t)g.Nx * g.Ny));
    int I = i / g.mx, J = j / g.my;
    P s = P(0);
    for (int p = 0; p < 3; ++p) {
        int Ip = g.wx[3 * I + p];
        for (int q = 0; q < 3; ++q) {
            int Jq = g.wy[3 * J + q];
            s += g.Rx[3 * i + p] * g.Ry[3 * j + q] * W[((size_t)K * g.ny + Jq) * g.nx + Ip];
        }
    }
    Ws[((size_t)K * g.mz * g.Ny + j) * g.Nx + i] = s;
}

// Stage Z balance: thread per coarse cell; writes the full-area inner-plane W.
// MZ > 0: the refinement factor in z known at compile time (the loop unrolls
// and every load is issued before the running balance); 0: any factor.
template <typename P, int MZ = 0>
__global__ void k_column_balance(Grid<P> g, const P* __restrict__ U, const P* __restrict__ V,
                                 const P* __restrict__ W, P* __restrict__ scrW)
{
    size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    size_t n = (size_t)g.nz * g.ny * g.nx;
    if (t >= n) return;
    int I = (int)(t % g.nx);
    int J = (int)((t / g.nx) % g.ny);
    int K = (int)(t / ((size_t)g.nx * g.ny));
    int Ie = g.walls ? I + 1 : (I + 1) % g.nx;
    int Jn = g.walls ? J + 1 : (J + 1) % g.ny;
    P F = W[((size_t)(K + 1) * g.ny + J) * g.nx + I] * g.DX * g.DY;
    const int mz = MZ > 0 ? MZ : g.mz;
#pragma unroll
    for (int c = mz - 1; c >= 1; --c) {
        int k = K * mz + c;
        P uw = 0, ue = 0, vs = 0, vn = 0;
        for (int q = 0; q < 3; ++q) {
            P r = g.Rz[3 * k + q];
            int Kq = g.wz[3 * K + q];
            uw += r * U[((size_t)Kq * g.ny + J) * g.cux + I];
            ue += r * U[((size_t)Kq * g.ny + J) * g.cux + Ie];
            vs += r * V[((size_t)Kq * g.cvy + J) * g.nx + I];
            vn += r * V[((size_t)Kq * g.cvy + Jn) * g.nx + I];
        }
        F = F + (ue - uw) * g.DY * g.dz[k] + (vn - vs) * g.DX * g.dz[k];
        scrW[((size_t)k * g.ny + J) * g.nx + I] = F / (g.DX * g.DY);
    }
}

// Stage Z split: thread per dense face on an inner z-plane.
template <typename P>
__global__ void k_split_w(Grid<P> g, const P* __restrict__ scrW, P* __restrict__ Ws)
{
    size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    size_t planes = (size_t)g.nz * (g.mz - 1);
    size_t n = planes * g.Ny * g.Nx;
    if (t >= n) return;
    int i = (int)(t % g.Nx);
    int j = (int)((t / g.Nx) % g.Ny);
    int kk = (int)(t / ((size_t)g.Nx * g.Ny));
    int k = (kk / (g.mz - 1)) * g.mz + kk % (g.mz - 1) + 1;
    int I = i / g.mx, J = j / g.my;
    P s = P(0);
    for (int p = 0; p < 3; ++p) {
        int Ip = g.wx[3 * I + p];
        for (int q = 0; q < 3; ++q) {
            int Jq = g.wy[3 * J + q];
            s += g.Rx[3 * i + p] * g.Ry[3 * j + q] * scrW[((size_t)k * g.ny + Jq) * g.nx + Ip];
        }
    }
    Ws[((size_t)k * g.Ny + j) * g.Nx + i] = s;
}

// Stage Y balance: thread per (I, J, dense layer k); writes the full-width
// inner-row V.
template <typename P>
__global__ void k_row_balance(Grid<P> g, const P* __restrict__ Us, const P* __restrict__ Vs,
                              const P* __restrict__ Ws, P* __restrict__ scrV)
{
    size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    size_t n = (size_t)g.Nz * g.ny * g.nx;
    if (t >= n) return;
    int I = (int)(t % g.nx);
    int J = (int)((t / g.nx) % g.ny);
    int k = (int)(t / ((size_t)g.nx * g.ny));
    int Ie = g.walls ? I + 1 : (I + 1) % g.nx;
    P dzk = g.dz[k];
    P G = 0;
    for (int a = 0; a < g.mx; ++a) G += Vs[((size_t)k * g.vfy + (size_t)J * g.my) * g.Nx + I * g.mx + a] * g.dx;
    G *= dzk;
    for (int b = 0; b < g.my - 1; ++b) {
        int j = J * g.my + b;
        P uw = Us[((size_t)k * g.Ny + j) * g.ufx + (size_t)I * g.mx];
        P ue = Us[((size_t)k * g.Ny + j) * g.ufx + (size_t)Ie * g.mx];
        P wb = 0, wt = 0;
        for (int a = 0; a < g.mx; ++a) {
            wb += Ws[((size_t)k * g.Ny + j) * g.Nx + I * g.mx + a] * g.dx;
            wt += Ws[((size_t)(k + 1) * g.Ny + j) * g.Nx + I * g.mx + a] * g.dx;
        }
        G = G - (ue - uw) * g.dy * dzk - (wt - wb) * g.dy;
        scrV[((size_t)k * g.vfy + j + 1) * g.nx + I] = G / (g.DX * dzk);
    }
}

// Stage Y split: thread per dense face on an inner y-row.
template <typename P>
__global__ void k_split_v(Grid<P> g, const P* __restrict__ scrV, P* __restrict__ Vs)
{
    size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    size_t rows = (size_t)g.ny * (g.my - 1);
    size_t n = (size_t)g.Nz * rows * g.Nx;
    if (t >= n) return;
    int i = (int)(t % g.Nx);
    int jj = (int)((t / g.Nx) % rows);
    int k = (int)(t / ((size_t)g.Nx * rows));
    int j = (jj / (g.my - 1)) * g.my + jj % (g.my - 1) + 1;
    int I = i / g.mx;
    P s = P(0);
    for (int p = 0; p < 3; ++p) s += g.Rx[3 * i + p] * scrV[((size_t)k * g.vfy + j) * g.nx + g.wx[3 * I + p]];
    Vs[((size_t)k * g.vfy + j) * g.Nx + i] = s;
}

// Stage X: thread per (I, dense row j, dense layer k).
template <typename P>
__global__ void k_stage_x(Grid<P> g, P* __restrict__ Us, const P* __restrict__ Vs, const P* __restrict__ Ws)
{
    size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    size_t n = (size_t)g.Nz * g.Ny * g.nx;
    if (t >= n) return;
    int I = (int)(t % g.nx);
    int j = (int)((t / g.nx) % g.Ny);
    int k = (int)(t / ((size_t)g.nx * g.Ny));
    int jn = g.walls ? j + 1 : (j + 1) % g.Ny;
    P dzk = g.dz[k];
    size_t urow = ((size_t)k * g.Ny + j) * g.ufx;
    P H = Us[urow + (size_t)I * g.mx] * g.dy * dzk;
    for (int a = 0; a < g.mx - 1; ++a) {
        int i = I * g.mx + a;
        H = H - (Vs[((size_t)k * g.vfy + jn) * g.Nx + i] - Vs[((size_t)k * g.vfy + j) * g.Nx + i]) * g.dx * dzk
              - (Ws[((size_t)(k + 1) * g.Ny + j) * g.Nx + i] - Ws[((size_t)k * g.Ny + j) * g.Nx + i]) * g.dx * g.dy;
        Us[urow + i + 1] = H / (g.dy * dzk);
    }
}

// ------------------------------------------------------------- axis by axis
// The stages reordered so that every value is split along one axis at a time, at
// the coarse resolution of the axes still to come (the tensor product of the R
// matrices, and the balances, are linear):
//   UZ, VZ  R_z of U and V                             [Nz][ny][nx]
//   WC      full-area W on every dense plane            [Nz+1][ny][nx]
//   UO, WY  R_y of UZ and WC                           [Nz][Ny][nx]
//   VR      full-width V: VZ on the coarse rows, the row balance between them
//   dense   R_x of WY and VR, the cell balance for U from UO
// which takes about 10 operations per dense cell at M = 2 (1.5 for each R_x or
// R_y split, see split) where the nine-point products of the in-place chain take
// about 60; in FP64 that is what bounds it.  Runs over groups of coarse slabs so
// that the intermediates stay within kRefineWork bytes.
// Measured in FP64, coarse 128 x 128 x 96 at M = 2 (256 x 256 x 192 dense cells):
// 334 us for the refinement and 338 us with the dense faces given out as well;
// 1311 and 1414 us in place.

constexpr size_t kRefineWork = (size_t)256 << 20;

// Split of one coarse cell's value along an axis: the dense values b < m of the
// window values c0, c1, c2 with the R rows r (rows sum to one, so a row is a
// combination of two differences).  SYM: m = 2 on a uniform axis with every window
// centred on its cell (periodic), whose rows are (1, 8, -1) / 8 and (-1, 8, 1) / 8;
// known at compile time, or both forms would be computed.
template <bool SYM, typename Out>
__device__ __forceinline__ void split(double c0, double c1, double c2, const double* __restrict__ r, int m, Out out)
{
    if constexpr (SYM) {
        const double d = 0.125 * (c0 - c2);
        out(0, c1 + d);
        out(1, c1 - d);
        return;
    }
    const double d0 = c0 - c1, d2 = c2 - c1;
#pragma unroll
    for (int b = 0; b < m; ++b) out(b, c1 + r[3 * b] * d0 + r[3 * b + 2] * d2);
}

struct Refine {
    Grid<double> g;
    const double *U, *V, *W;         // coarse faces
    double *UZ, *VZ, *WC, *UO, *WY, *VR;   // of the group's slabs K0 .. K1 - 1
    double *Us, *Vs, *Ws;            // dense faces
    double *Ue, *Ve, *We;            // a second copy of them, or NULL
    unsigned* vmax;                  // largest magnitudes of the components, or NULL
    int K0, K1;
    int layers;                      // of a block of k_dense
    double iDX, iDY, dydX, dxdy;     // 1 / DX, 1 / DY, dy / DX, dx / dy
};

template <typename N>
__global__ void __launch_bounds__(kThreads) k_z_split(const Refine A)
{
    const Grid<double>& g = A.g;
    const N nu = (N)(A.K1 - A.K0) * g.ny * g.cux, nv = (N)(A.K1 - A.K0) * g.cvy * g.nx;
    for (N t = (N)blockIdx.x * blockDim.x + threadIdx.x; t < nu + nv; t += (N)gridDim.x * blockDim.x) {
        const bool u = t < nu;
        const N plane = u ? (N)g.ny * g.cux : (N)g.cvy * g.nx, e = u ? t : t - nu;
        const int q = (int)(e / plane), K = A.K0 + q;
        const double* src = (u ? A.U : A.V) + e % plane;
        double* dst = (u ? A.UZ : A.VZ) + (size_t)q * g.mz * plane + e % plane;
        if (g.mz == 1) {
            dst[0] = src[(size_t)K * plane];
            continue;
        }
        const int* w = g.wz + 3 * K;
        split<false>(src[(size_t)w[0] * plane], src[(size_t)w[1] * plane], src[(size_t)w[2] * plane],
                     g.Rz + 3 * (size_t)K * g.mz, g.mz, [&](int b, double v) { dst[(size_t)b * plane] = v; });
    }
}

template <typename N>
__global__ void __launch_bounds__(kThreads) k_slab_balance(const Refine A)
{
    const Grid<double>& g = A.g;
    const N plane = (N)g.ny * g.nx, n = (N)(A.K1 - A.K0) * plane;
    for (N t = (N)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (N)gridDim.x * blockDim.x) {
        const int q = (int)(t / plane), K = A.K0 + q;
        const int J = (int)((t % plane) / g.nx), I = (int)(t % g.nx);
        const int Ie = g.walls ? I + 1 : (I + 1 == g.nx ? 0 : I + 1), Jn = g.walls ? J + 1 : (J + 1 == g.ny ? 0 : J + 1);
        double F = A.W[(size_t)(K + 1) * plane + (t % plane)];
        double* wc = A.WC + (size_t)q * g.mz * plane + t % plane;
        if (K == A.K1 - 1) wc[(size_t)g.mz * plane] = F;
        for (int c = g.mz - 1; c >= 1; --c) {
            const size_t k = (size_t)q * g.mz + c;
            const double* u = A.UZ + (k * g.ny + J) * g.cux;
            const double* v = A.VZ + k * g.cvy * g.nx + I;
            F += g.dz[K * g.mz + c] * ((u[Ie] - u[I]) * A.iDX + (v[(size_t)Jn * g.nx] - v[(size_t)J * g.nx]) * A.iDY);
            wc[(size_t)c * plane] = F;
        }
        wc[0] = A.W[(size_t)K * plane + (t % plane)];
    }
}

// R_y of UZ (rows of cux) and WC (rows of nx): thread per (plane, coarse row, column).
template <typename N, bool SYM>
__global__ void __launch_bounds__(kThreads) k_y_split(const Refine A)
{
    const Grid<double>& g = A.g;
    const int L = (A.K1 - A.K0) * g.mz;
    const N nu = (N)L * g.ny * g.cux, nw = (N)(L + 1) * g.ny * g.nx;
    for (N t = (N)blockIdx.x * blockDim.x + threadIdx.x; t < nu + nw; t += (N)gridDim.x * blockDim.x) {
        const bool u = t < nu;
        const int row = u ? g.cux : g.nx;
        const N e = u ? t : t - nu, er = e / row;
        const int I = (int)(e - er * row), k = (int)(er / g.ny), J = (int)(er - (N)k * g.ny);
        const double* src = (u ? A.UZ : A.WC) + (size_t)k * g.ny * row + I;
        double* dst = (u ? A.UO : A.WY) + ((size_t)k * g.Ny + (size_t)J * g.my) * row + I;
        if (g.my == 1) {
            dst[0] = src[(size_t)J * row];
            continue;
        }
        const int* w = g.wy + 3 * J;
        split<SYM>(src[(size_t)w[0] * row], src[(size_t)w[1] * row], src[(size_t)w[2] * row], g.Ry + 3 * (size_t)J * g.my,
                   g.my, [&](int b, double v) { dst[(size_t)b * row] = v; });
    }
}

template <typename N>
__global__ void __launch_bounds__(kThreads) k_row_v(const Refine A)
{
    const Grid<double>& g = A.g;
    const int L = (A.K1 - A.K0) * g.mz;
    const N n = (N)L * g.cvy * g.nx;
    for (N t = (N)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (N)gridDim.x * blockDim.x) {
        const N tr = t / g.nx;
        const int I = (int)(t - tr * g.nx), k = (int)(tr / g.cvy), J = (int)(tr - (N)k * g.cvy);
        double v = A.VZ[t];
        double* dst = A.VR + ((size_t)k * g.vfy + (size_t)J * g.my) * g.nx + I;
        dst[0] = v;
        if (J == g.ny) continue;                           // the north wall's faces
        const int Ie = g.walls ? I + 1 : (I + 1 == g.nx ? 0 : I + 1);
        const double dydz = g.dy * g.inv_dz[A.K0 * g.mz + k];
        for (int b = 0; b < g.my - 1; ++b) {
            const size_t r = (size_t)k * g.Ny + (size_t)J * g.my + b;
            const double* u = A.UO + r * g.cux;
            const double* w = A.WY + r * g.nx + I;
            v = v - (u[Ie] - u[I]) * A.dydX - (w[(size_t)g.Ny * g.nx] - w[0]) * dydz;
            dst[(size_t)(b + 1) * g.nx] = v;
        }
    }
}

// The dense faces: a block takes 32 coarse columns and 8 dense rows through a
// chunk of layers, a warp a row (the ninth one the V faces north of the tile).  The
// splits of V on this layer and of W on the planes below and above meet in shared
// memory, where U's cell balance reads them and whole rows are written from.
constexpr int kDenseRows = 8, kDenseLayers = 8;
// MX: the refinement in x where known at compile time (2, 4), else 0; SYM: see split.
template <int MX, bool SYM>
__global__ void __launch_bounds__(32 * (kDenseRows + 1)) k_dense(const Refine A)
{
    const Grid<double>& g = A.g;
    const int mx = MX ? MX : g.mx;
    extern __shared__ __align__(16) unsigned char dsm[];
    const int row = 32 * mx, lane = threadIdx.x & 31, r = threadIdx.x >> 5;
    double* const wv = reinterpret_cast<double*>(dsm);     // [2][8][row]
    double* const vv = wv + 2 * kDenseRows * row;          // [2][9][row]
    double* const uv = vv + 2 * (kDenseRows + 1) * row;    // [8][row]
    const int ntx = (g.nx + 31) / 32, bx = blockIdx.x % ntx;
    const int I = bx * 32 + lane, j = (blockIdx.x / ntx) * kDenseRows + r;
    const int i0 = bx * row, ni = min(row, g.Nx - i0);
    const int L = (A.K1 - A.K0) * g.mz, l0 = blockIdx.y * A.layers, l1 = min(l0 + A.layers, L);
    const bool col = I < g.nx, own = r < kDenseRows && j < g.Ny;
    const bool vrow = col && j <= g.Ny;
    const int jv = (!g.walls && j == g.Ny) ? 0 : j;
    const int w0 = col ? g.wx[3 * I] : 0, w1 = col ? g.wx[3 * I + 1] : 0, w2 = col ? g.wx[3 * I + 2] : 0;
    const double* const rx = g.Rx + 3 * (size_t)(col ? I : 0) * mx;
    unsigned mu = 0, mv = 0, mw = 0;
    auto mag = [](double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; };
    // the window of this thread's column in a coarse row, and its split along x into a
    // shared row
    auto window = [&](const double* src, double (&c)[3]) {
        c[1] = src[mx == 1 ? I : w1];
        if (mx > 1) {
            c[0] = src[w0];
            c[2] = src[w2];
        }
    };
    auto xsplit = [&](const double (&c)[3], double* dst) {
        if (mx == 1) dst[lane] = c[1];
        else split<SYM>(c[0], c[1], c[2], rx, mx, [&](int b, double v) { dst[lane * mx + b] = v; });
    };
    // a shared row to a dense one (and its copy), n values
    auto put = [&](const double* src, double* a, double* b, size_t at, int n, unsigned& m) {
#pragma unroll
        for (int q = 0; q < mx; ++q) {
            const int e = lane + 32 * q;
            if (e >= n) break;
            const double v = src[e];
            m = max(m, mag(v));
            a[at + e] = v;
            if (b) b[at + e] = v;
        }
    };
    auto wrow = [&](int l) { return wv + ((l & 1) * kDenseRows + r) * row; };
    auto vface = [&](int l, int q) { return vv + ((l & 1) * (kDenseRows + 1) + q) * row; };
    const size_t k00 = (size_t)A.K0 * g.mz;
    // what a layer splits is loaded a layer ahead
    double cv[3], cw[3], cu = 0.0;
    auto ahead = [&](int l) {
        if (vrow) window(A.VR + ((size_t)l * g.vfy + jv) * g.nx, cv);
        if (own && col) {
            window(A.WY + ((size_t)(l + 1) * g.Ny + j) * g.nx, cw);
            cu = A.UO[((size_t)l * g.Ny + j) * g.cux + I];
        }
    };
    if (own) {
        if (col) {
            window(A.WY + ((size_t)l0 * g.Ny + j) * g.nx, cw);
            xsplit(cw, wrow(l0));
        }
        __syncwarp();
        if (k00 + l0 == 0) put(wrow(l0), A.Ws, A.We, (size_t)j * g.Nx + i0, ni, mw);
    }
    if (l0 < l1) ahead(l0);
    for (int l = l0; l < l1; ++l) {
        const size_t k = k00 + l;
        double h = cu;
        if (vrow) xsplit(cv, vface(l, r));
        if (own && col) xsplit(cw, wrow(l + 1));
        if (l + 1 < l1) ahead(l + 1);
        __syncthreads();
        if (r < kDenseRows && j < g.vfy) put(vface(l, r), A.Vs, A.Ve, (k * g.vfy + j) * g.Nx + i0, ni, mv);
        // walls: the north wall's faces where they lie just beyond the tile
        if (g.walls && r == kDenseRows && j == g.Ny) put(vface(l, r), A.Vs, A.Ve, (k * g.vfy + j) * g.Nx + i0, ni, mv);
        if (!own) continue;
        put(wrow(l + 1), A.Ws, A.We, ((k + 1) * g.Ny + j) * g.Nx + i0, ni, mw);
        double* const u = uv + r * row;
        if (col) {
            const double dxdz = g.dx * g.inv_dz[k];
            const double *vs = vface(l, r), *vn = vface(l, r + 1), *wb = wrow(l), *wt = wrow(l + 1);
#pragma unroll
            for (int a = 0; a < mx; ++a) {
                const int e = lane * mx + a;
                u[e] = h;
                if (a == mx - 1) break;
                h = h - (vn[e] - vs[e]) * A.dxdy - (wt[e] - wb[e]) * dxdz;
            }
        }
        __syncwarp();
        const size_t at = (k * g.Ny + j) * g.ufx + i0;
        put(u, A.Us, A.Ue, at, ni, mu);
        if (g.walls && I == g.nx - 1) {                    // the east wall's face
            const double v = A.UO[((size_t)l * g.Ny + j) * g.cux + g.nx];
            mu = max(mu, mag(v));
            A.Us[at + ni] = v;
            if (A.Ue) A.Ue[at + ni] = v;
        }
    }
    if (A.vmax) {
        const unsigned m[3] = {__reduce_max_sync(0xffffffffu, mu), __reduce_max_sync(0xffffffffu, mv),
                               __reduce_max_sync(0xffffffffu, mw)};
        if (lane == 0)
            for (int c = 0; c < 3; ++c)
                if (m[c]) atomicMax(A.vmax + c, m[c]);
    }
}

// Values of the intermediates of one coarse slab (refine_work) and how many slabs
// go together.
size_t slab_values(const Grid<double>& g, size_t (&n)[6], int slabs)
{
    const size_t L = (size_t)slabs * g.mz;
    n[0] = L * g.ny * g.cux;
    n[1] = L * g.cvy * g.nx;
    n[2] = (L + 1) * g.ny * g.nx;
    n[3] = L * g.Ny * g.cux;
    n[4] = (L + 1) * g.Ny * g.nx;
    n[5] = L * g.vfy * g.nx;
    size_t s = 0;
    for (size_t& q : n) s += q = (q + 31) / 32 * 32;
    return s;
}
// The stages at coarse x resolution of S slabs (L layers).
template <typename N>
void launch_coarse(const Refine& A, size_t S, size_t L, cudaStream_t st)
{
    const Grid<double>& g = A.g;
    auto grid = [](size_t threads) { return (unsigned)std::min<size_t>((threads + kThreads - 1) / kThreads, 152 * 64); };
    k_z_split<N><<<grid(S * ((size_t)g.ny * g.cux + (size_t)g.cvy * g.nx)), kThreads, 0, st>>>(A);
    k_slab_balance<N><<<grid(S * g.ny * g.nx), kThreads, 0, st>>>(A);
    const unsigned gy = grid(L * g.ny * ((size_t)g.cux + g.nx));
    if (g.my == 2 && !g.walls) k_y_split<N, true><<<gy, kThreads, 0, st>>>(A);
    else k_y_split<N, false><<<gy, kThreads, 0, st>>>(A);
    k_row_v<N><<<grid(L * g.cvy * g.nx), kThreads, 0, st>>>(A);
}

}  // namespace

int refine_slabs(const Grid<double>& g)
{
    size_t n[6];
    int s = g.nz;
    // (and at most 65535 chunks of layers in a launch)
    while (s > 1 && (slab_values(g, n, s) * sizeof(double) > kRefineWork || (size_t)s * g.mz > 65535u * kDenseLayers))
        s = (s + 1) / 2;
    return s;
}

size_t refine_work(const Grid<double>& g, int slabs)
{
    size_t n[6];
    return slab_values(g, n, slabs) * sizeof(double);
}

cudaError_t launch_refine(const Grid<double>& g, const double* U, const double* V, const double* W, double* const out[3], double* const copy[3],
                          unsigned* vmax, double* work, int slabs, cudaStream_t st)
{
    Refine A;
    A.g = g;
    A.U = U; A.V = V; A.W = W;
    A.Us = out[0]; A.Vs = out[1]; A.Ws = out[2];
    A.Ue = copy ? copy[0] : nullptr;
    A.Ve = copy ? copy[1] : nullptr;
    A.We = copy ? copy[2] : nullptr;
    A.vmax = vmax;
    A.iDX = 1.0 / g.DX;
    A.iDY = 1.0 / g.DY;
    A.dydX = g.dy / g.DX;
    A.dxdy = g.dx / g.dy;
    cudaError_t e = cudaSuccess;
    if (vmax) e = cudaMemsetAsync(vmax, 0, 3 * sizeof(unsigned), st);
    const int form = g.mx == 2 ? (g.walls ? 1 : 2) : (g.mx == 4 ? 3 : 0);
    void (*const forms[4])(const Refine) = {k_dense<0, false>, k_dense<2, false>, k_dense<2, true>, k_dense<4, false>};
    void (*const dense)(const Refine) = forms[form];
    const int smem = (5 * kDenseRows + 2) * 32 * g.mx * (int)sizeof(double);
    static unsigned long long done[4];                     // one bit per device, for each form (mx <= 8: 84 KB in FP64)
    if (e == cudaSuccess)
        e = smem_optin(reinterpret_cast<const void*>(dense), (5 * kDenseRows + 2) * 32 * 8 * (int)sizeof(double),
                       &done[form]);
    if (e != cudaSuccess) return e;
    size_t n[6];
    slab_values(g, n, slabs);
    double** const part[6] = {&A.UZ, &A.VZ, &A.WC, &A.UO, &A.WY, &A.VR};
    for (int q = 0; q < 6; ++q) {
        *part[q] = work;
        work += n[q];
    }
    for (A.K0 = 0; A.K0 < g.nz; A.K0 = A.K1) {
        A.K1 = std::min(A.K0 + slabs, g.nz);
        const size_t S = A.K1 - A.K0, L = S * g.mz;
        // 32-bit indexes unless a slab is enormous
        if (slab_values(g, n, (int)S) < (1ull << 31)) launch_coarse<unsigned>(A, S, L, st);
        else launch_coarse<size_t>(A, S, L, st);
        // eight layers of a column per block (one more W plane split), fewer where that
        // would leave SMs without four blocks
        const size_t tiles = (size_t)((g.nx + 31) / 32) * ((g.Ny + kDenseRows - 1) / kDenseRows);
        A.layers = kDenseLayers;
        while (A.layers > 1 && tiles * ((L + A.layers - 1) / A.layers) < 4 * 152) A.layers /= 2;
        const dim3 grd((unsigned)tiles, (unsigned)((L + A.layers - 1) / A.layers));
        dense<<<grd, 32 * (kDenseRows + 1), smem, st>>>(A);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return e;
}

template <typename P>
cudaError_t launch_refine_in_place(const Grid<P>& g, const P* U, const P* V, const P* W, P* Us, P* Vs, P* Ws, P* scrW,
                                   P* scrV, cudaStream_t st)
{
    size_t n;
    n = (size_t)g.Nz * g.Ny * g.cux;
    k_outer_u<P><<<blocks_for(n), kThreads, 0, st>>>(g, U, Us);
    n = (size_t)g.Nz * g.cvy * g.Nx;
    k_outer_v<P><<<blocks_for(n), kThreads, 0, st>>>(g, V, Vs);
    n = (size_t)(g.nz + 1) * g.Ny * g.Nx;
    k_outer_w<P><<<blocks_for(n), kThreads, 0, st>>>(g, W, Ws);
    if (g.mz > 1) {
        n = (size_t)g.nz * g.ny * g.nx;
        k_column_balance<P><<<blocks_for(n), kThreads, 0, st>>>(g, U, V, W, scrW);
        n = (size_t)g.nz * (g.mz - 1) * g.Ny * g.Nx;
        k_split_w<P><<<blocks_for(n), kThreads, 0, st>>>(g, scrW, Ws);
    }
    if (g.my > 1) {
        n = (size_t)g.Nz * g.ny * g.nx;
        k_row_balance<P><<<blocks_for(n), kThreads, 0, st>>>(g, Us, Vs, Ws, scrV);
        n = (size_t)g.Nz * g.ny * (g.my - 1) * g.Nx;
        k_split_v<P><<<blocks_for(n), kThreads, 0, st>>>(g, scrV, Vs);
    }
    if (g.mx > 1) {
        n = (size_t)g.Nz * g.Ny * g.nx;
        k_stage_x<P><<<blocks_for(n), kThreads, 0, st>>>(g, Us, Vs, Ws);
    }
    return cudaGetLastError();
}

template cudaError_t launch_refine_in_place<double>(const Grid<double>&, const double*, const double*, const double*,
                                                    double*, double*, double*, double*, double*, cudaStream_t);
template cudaError_t launch_refine_in_place<float>(const Grid<float>&, const float*, const float*, const float*, float*,
                                                   float*, float*, float*, float*, cudaStream_t);

// Stage Z slab balance alone (full-area W on the inner planes), for the
// split-x fused path.
template <typename P>
cudaError_t launch_column_balance(const Grid<P>& g, const P* U, const P* V, const P* W, P* scrW, cudaStream_t st)
{
    if (g.mz > 1) {
        const size_t n = (size_t)g.nz * g.ny * g.nx;
        if (g.mz == 4) k_column_balance<P, 4><<<blocks_for(n), kThreads, 0, st>>>(g, U, V, W, scrW);
        else if (g.mz == 2) k_column_balance<P, 2><<<blocks_for(n), kThreads, 0, st>>>(g, U, V, W, scrW);
        else k_column_balance<P><<<blocks_for(n), kThreads, 0, st>>>(g, U, V, W, scrW);
    }
    return cudaGetLastError();
}
template cudaError_t launch_column_balance<float>(const Grid<float>&, const float*, const float*, const float*,
                                                  float*, cudaStream_t);

}  // namespace mr
