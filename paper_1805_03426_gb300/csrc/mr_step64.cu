// The FP64 stored-velocity step (Eq. 5, second-order faces, one velocity
// level) in 64-bit fixed point on the integer pipes (mr_fix.cuh): periodic or
// walled sides, explicit or half-implicit vertical diffusion.
//
// A warp marches a column of 30 x 3 cells through a chunk of layers.  Its 32
// lanes hold the 30 columns and one neighbour on each side, so that x
// neighbours and the fluxes of shared x faces are shuffles; the bands of three
// rows lie end to end, so that a warp may hold the end of one and the start of
// the next (band_span); the rows of T^s and
// T^{s-1} on the current plane, the plane below of T^{s-1} and the flux through
// the bottom faces stay in registers from layer to layer.  What a layer reads
// is copied into shared memory one layer ahead (cp.async, 8 bytes a lane: any
// row length and offset).  Per layer a warp decodes each scalar value once (its
// rows of the next plane, the two rows beyond the tile on this one) and each
// face velocity once, forms every face flux once,
//   F = u (T_a + T_b)  (x, y),   F = 2 w (w_lo T_a + w_hi T_b)  (z),
// and accumulates  sum rates x (flux differences, diffusion neighbours)  in one
// wide integer, which the FP64 pipe then scales and adds to T^{s-1}.
//
// Measured on 256 x 256 x 192 cells (coarse 128 x 128 x 96): 0.210 ms per step,
// 2.9 TB/s on the 48 B/cell of the method; 0.597 ms with one thread per cell and
// 25 FP64 operations per cell, which ran the FP64 pipe at 88 %.  365 instructions
// per cell (of a warp, times 32) issue at 0.59 per clock and scheduler; integer
// multiply-adds and the integer ALU share the time, so what bounds it is the
// decoding (14 instructions a value, 6.7 values a cell) and the 46 multiply-adds.
// Rows: 3 per warp 0.214 ms, 4 (12 instead of 16 warps per SM) 0.225, 2 (two
// of four decoded rows are halo) 0.231, 1 0.274.
//
// Scales.  E is the largest exponent among the scalar values that the warp's
// layer reads (its rows on planes k-1, k, k+1 and the rows beyond the tile);
// values become 60-bit integers relative to it.  The face velocities are 62-bit
// integers relative to the largest one of their component in the domain (vmax,
// found when they were refined): what that rounds off is multiplied by the
// local scalar, so it is small beside the local result wherever u is small.
// The rates (1/(2 dx), kappa/dx^2, ...) are scaled so that their sum, weighted
// by those velocities, is below 2^62 (eR).  Every sum of integers is exact
// and the products' errors are about 2^-58 of (CFL number x largest scalar).
// That is below FP64's own rounding of a result as long as the result is not
// much smaller than the largest value around it, so a layer in which the
// values around some lane's rows are all below 2^-kSpan of the warp's largest
// (and not all zero), or which holds an infinity, a NaN or only values near the
// underflow limit, is stepped in FP64 arithmetic instead (22 operations per cell:
// a field that falls off by many decades from cell to cell everywhere runs at
// 0.65 ms, 0.74 to 0.78 on walled or implicit grids, one of zeros and ones at
// 0.29 ms).  So is every layer where gdt 2^eR
// exceeds 2^kMaxRate = 64: a stable explicit step's rates are below 16 (2^eR is up
// to four times their sum), and beyond the limit the products' error, 2^-58 of
// them, would pass FP64's rounding -- a single face velocity far above all others
// with a time step that follows the others, or implicit vertical diffusion over
// layers much thinner than the time step needs.
// So a result is as accurate as FP64 arithmetic's relative to the largest values
// around its cell, not to its own value where that is much smaller; and as decoding
// and products round down, stepping -T gives the negatives to rounding only (an ulp
// of the largest value; exactly odd rounding would cost 10 % of a step).
#include <math.h>

#include "mr_fix.cuh"
#include "mr_internal.cuh"

namespace mr {
namespace {

using namespace fix;

constexpr int kWarps = 4;            // warps per block (independent of each other)
constexpr int kCols = 30;            // columns a warp writes
constexpr int kRows = 3;             // rows a warp writes
constexpr int kBlocks = 4;           // resident blocks per SM
constexpr int kStart = 3;            // a chunk's start, in layers
constexpr int kSpan = 6;             // binades below the warp's largest value that a lane may lie
constexpr int kMaxChunk = 32;        // layers per chunk
constexpr int kMaxRate = 6;          // binades that the step's rates gdt 2^eR may reach
// exponent fields of scales: what is smaller or larger (but zero) is left to
// FP64 arithmetic, so that no power of two below leaves the normal range
constexpr int kFieldLo = 1023 - 300, kFieldHi = 1023 + 300;

// The constants of the layers of a block's chunk, scaled by 2^(62 - eR).
struct LayerK {
    Bal hz, cdn, cup, ndiag;         // 2 S_W / dz_k, cdn, cup, minus the sum of all neighbours' rates
    Bal wlo, whi;                    // weights of the layer's top face, times 2^62
};

// And what a layer in FP64 arithmetic takes: 1 / dz, the vertical rates, the diagonal,
// the weights of the top face.
struct LayerP {
    double iz, cdn, cup, ndiag, wlo, whi;
};

struct Args {
    Grid<double> g;
    const double *U, *V, *W, *Tm1, *T;
    double* out;
    double a, b, gdt;
    double zs, plate;                // explicit share of the vertical diffusion, plate value / share
    const unsigned* vmax;
    int kc;
};


constexpr int stage_rows(int R) { return 5 * R + 5; }

// z-face flux 2 T_f w from the values below and above (60-bit), their weights
// and w (62-bit)
__device__ __forceinline__ long long zflux(Bal tb, Bal tt, Bal wlo, Bal whi, Bal w)
{
    Acc p{0, 0};
    mac(p, wlo, tb);
    mac(p, whi, tt);
    return mul(bal((p.H << 3) + (p.M >> 29)), w);
}

// DIFF: the diffusion of layers in FP64 arithmetic by differences (as k_step_stored has
// it), or folded (as k_step_periodic has it: the periodic explicit form).
template <int R, bool WALLS, bool DIFF, bool LF>
__global__ void __launch_bounds__(32 * kWarps, kBlocks) k_step_fix(const Args A)
{
    after_previous();
    let_next();
    const Grid<double>& g = A.g;
    __shared__ LayerK sk[kMaxChunk];
    __shared__ LayerP sp[kMaxChunk];
    __shared__ Bal sc[4];                                 // 4 S_U hx, 4 S_V hy, kx2, ky2
    const int k0 = blockIdx.y * A.kc, k1 = min(k0 + A.kc, g.Nz);
    const int lane = threadIdx.x & 31;
    // scales of the velocity components and the rates (the lanes of a warp share
    // the layers, to spare the FP64 pipe)
    const int EU = max((int)(A.vmax[0] >> 20), kFieldLo), EV = max((int)(A.vmax[1] >> 20), kFieldLo),
              EW = max((int)(A.vmax[2] >> 20), kFieldLo);
    bool usable = EU <= kFieldHi && EV <= kFieldHi && EW <= kFieldHi;
    int eR;
    {
        unsigned m = 0;                                   // positive values are ordered like their high words
        for (int k = k0 + lane; k < k1; k += 32)
            m = max(m, (unsigned)__double2hiint(2.0 * g.inv_dz[k] * pow2(EW - 1022) + 2.0 * A.zs * (g.cdn[k] + g.cup[k])));
        m = __reduce_max_sync(0xffffffffu, m);
        const double r = __hiloint2double((int)m + 1, 0) + 4.0 * (g.hx * pow2(EU - 1022) + g.hy * pow2(EV - 1022)) +
                         4.0 * (g.kx2 + g.ky2);
        eR = exponent(r);                                 // 2^eR > r
        usable = usable && eR > -400 && eR < 400 && exponent(A.gdt) + eR <= kMaxRate;
    }
    for (int q = threadIdx.x - 64; q >= 0 && q < k1 - k0; q += blockDim.x) {   // (other warps' lanes than below)
        const int k = k0 + q;
        const double cdn = A.zs * g.cdn[k], cup = A.zs * g.cup[k];
        sp[q] = LayerP{g.inv_dz[k], cdn, cup, -2.0 * (g.kx2 + g.ky2) - cdn - cup, g.wlo[k + 1], g.whi[k + 1]};
    }
    if (usable) {
        for (int q = threadIdx.x; q < k1 - k0; q += blockDim.x) {
            const int k = k0 + q;
            const double p = pow2(62 - eR);
            // the diagonal is minus the sum of the neighbours' integers, so that the
            // diffusion of a constant is zero exactly
            const long long kx = __double2ll_rn(g.kx2 * p), ky = __double2ll_rn(g.ky2 * p);
            const long long dn = __double2ll_rn(A.zs * g.cdn[k] * p), up = __double2ll_rn(A.zs * g.cup[k] * p);
            LayerK L;
            L.hz = fixed(2.0 * g.inv_dz[k] * pow2(EW - 1022 + 62 - eR));
            L.cdn = bal(dn);
            L.cup = bal(up);
            L.ndiag = bal(-(2 * (kx + ky) + dn + up));
            L.wlo = fixed(g.wlo[k + 1] * 0x1p62);
            L.whi = fixed(g.whi[k + 1] * 0x1p62);
            sk[q] = L;
        }
        if (threadIdx.x == 32 * (kWarps - 1)) {
            sc[0] = fixed(g.hx * pow2(EU - 1020 + 62 - eR));
            sc[1] = fixed(g.hy * pow2(EV - 1020 + 62 - eR));
            sc[2] = fixed(g.kx2 * pow2(62 - eR));
            sc[3] = fixed(g.ky2 * pow2(62 - eR));
        }
    }
    __syncthreads();

    // the warp's part of the line of all bands of R rows (band_span)
    const int wid = blockIdx.x * kWarps + (threadIdx.x >> 5), span = band_span(g.Nx), bands = (g.Ny + R - 1) / R;
    if (wid * kCols >= (bands - 1) * span + g.Nx) return;          // whole warps; no barrier below
    const int at0 = wid * kCols + lane, band = min(at0 / span, bands - 1), i = at0 - band * span - 1, j0 = band * R;
    const bool mine = lane >= 1 && lane <= kCols && i >= 0 && i < g.Nx;
    const int ic = WALLS ? min(max(i, 0), g.Nx - 1) : (i + g.Nx) % g.Nx;
    const bool xin = !WALLS || (i > 0 && i < g.Nx);       // the face west of column i carries a flux
    // byte offsets in a plane (below 2^32: step_fix_fits): rows j0-1 .. j0+R; U rows; V faces j0 .. j0+R
    unsigned ro[R + 2], uo[R], vo[R + 1];
#pragma unroll
    for (int r = 0; r < R + 2; ++r) {
        const int j = j0 - 1 + r;
        ro[r] = 8u * (unsigned)((WALLS ? min(max(j, 0), g.Ny - 1) : (j + g.Ny) % g.Ny) * g.Nx + ic);
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
        uo[r] = WALLS ? 8u * (unsigned)(min(j0 + r, g.Ny - 1) * g.ufx + min(max(i, 0), g.Nx)) : ro[r + 1];
#pragma unroll
    for (int f = 0; f <= R; ++f) vo[f] = WALLS ? 8u * (unsigned)(min(j0 + f, g.Ny) * g.Nx + ic) : ro[f + 1];
    const size_t plane = (size_t)g.Nx * g.Ny, uplane = (size_t)g.Ny * g.ufx, vplane = (size_t)g.vfy * g.Nx;
    const double pl = g.dirichlet ? A.plate : 0.0;         // (below; minus this above)

    // A warp's own staging area: what layer k reads, copied one layer ahead.
    // Rows of 32 doubles: T^s and T^{s-1} of the tile's rows on plane k + 1, the
    // rows south and north of it of both on plane k, U, V faces, W on plane k + 1.
    constexpr int kT = 0, kD = R, kH = 2 * R, kU = 2 * R + 4, kV = 3 * R + 4, kW = 4 * R + 5;
    extern __shared__ double stage_all[];
    double* stage = stage_all + (size_t)(threadIdx.x >> 5) * 2 * stage_rows(R) * 32 + lane;
    auto fetch = [&](int k) {
        double* s = stage + (k & 1) * stage_rows(R) * 32;
        const double* pt = A.T + (size_t)k * plane;
        const double* pd = A.Tm1 + (size_t)k * plane;
        const double *ptn = pt + plane, *pdn = pd + plane;
        if (k + 1 < g.Nz) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                copy8(s + (kT + r) * 32, at(ptn, ro[r + 1]));
                copy8(s + (kD + r) * 32, at(pdn, ro[r + 1]));
            }
        }
        copy8(s + (kH + 0) * 32, at(pt, ro[0]));
        copy8(s + (kH + 1) * 32, at(pt, ro[R + 1]));
        copy8(s + (kH + 2) * 32, at(pd, ro[0]));
        copy8(s + (kH + 3) * 32, at(pd, ro[R + 1]));
        const double* pu = A.U + (size_t)k * uplane;
        const double* pv = A.V + (size_t)k * vplane;
        const double* pw = A.W + (size_t)(k + 1) * plane;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            copy8(s + (kU + r) * 32, at(pu, uo[r]));
            copy8(s + (kW + r) * 32, at(pw, ro[r + 1]));
        }
#pragma unroll
        for (int f = 0; f <= R; ++f) copy8(s + (kV + f) * 32, at(pv, vo[f]));
    };

    // state at layer k: T^s and T^{s-1} of the rows on plane k, T^{s-1} on plane
    // k - 1, the flux through the bottom faces (fixed point, scale E), T^{s-1} on
    // plane k as it is, and the lane's largest magnitudes on planes k - 1 and k
    long long t[R], d[R], fb[R];
    Bal db[R];
    double xd[R];
    unsigned mB = 0, mC = 0;
    int E = 0;
    bool primed = false, carried = false;                 // fb: fixed point at scale E; FP64 (after a plain layer)
    double gs = 0.0;
    fetch(k0);
    copy_commit();
    {
        const double* pt = A.T + (size_t)k0 * plane;
        const double* pd = A.Tm1 + (size_t)k0 * plane;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            xd[r] = *at(pd, ro[r + 1]);
            mC = max(mC, max(mag(*at(pt, ro[r + 1])), mag(xd[r])));
            if (k0 > 0) mB = max(mB, max(mag(*at(pt - plane, ro[r + 1])), mag(*at(pd - plane, ro[r + 1]))));
        }
        if (k0 == 0) mB = mag(pl);
    }
    for (int k = k0; k < k1; ++k) {
        const bool top = k == g.Nz - 1;
        const double* pt = A.T + (size_t)k * plane;
        const double* pd = A.Tm1 + (size_t)k * plane;
        const double* s = stage + (k & 1) * stage_rows(R) * 32;
        __syncwarp();                                     // every lane is done with the other half
        if (k + 1 < k1) fetch(k + 1);
        copy_commit();
        copy_wait<1>();                                   // this layer's copies (a lane reads only its own)
        double rt[R], rd[R];
        unsigned ml = max(mB, mC), mN = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            rt[r] = top ? 0.0 : s[(kT + r) * 32];
            rd[r] = top ? -pl : s[(kD + r) * 32];
            mN = max(mN, max(mag(rt[r]), mag(rd[r])));
        }
        const double hs = s[(kH + 0) * 32], hn = s[(kH + 1) * 32], es = s[(kH + 2) * 32], en = s[(kH + 3) * 32];
        ml = max(max(ml, mN), max(max(mag(hs), mag(hn)), max(mag(es), mag(en))));
        const unsigned mw = __reduce_max_sync(0xffffffffu, ml);
        int e = (int)(mw >> 20);
        bool plain = !usable || e > kFieldHi || (mw != 0 && e < kFieldLo) ||
                     __any_sync(0xffffffffu, ml != 0 && (int)(ml >> 20) + kSpan < e);
        if (!plain) {
            e = max(e, kFieldLo);
            if (!primed || e > E || e < E - 1) {
                // (re)start at this layer with the scale e
                E = e;
                primed = true;
                gs = A.gdt * pow2(E + eR - 1080);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    t[r] = dec<60>(*at(pt, ro[r + 1]), E);
                    d[r] = dec<60>(xd[r], E);
                    db[r] = bal(dec<60>(k > 0 ? *at(pd - plane, ro[r + 1]) : pl, E));
                    fb[r] = 0;
                    if (k > 0) {
                        fb[r] = zflux(bal(dec<60>(*at(pt - plane, ro[r + 1]), E)), bal(t[r]), fixed(g.wlo[k] * 0x1p62),
                                      fixed(g.whi[k] * 0x1p62), bal(dec<62>(*at(A.W + (size_t)k * plane, ro[r + 1]), EW)));
                    }
                }
            }
            plain = !ordinary(gs);
        }
        if (plain) {
            // FP64 arithmetic with the same shared fluxes; the bottom faces' are
            // carried from a layer below that was stepped in the same way
            const LayerP& L = sp[k - k0];
            double xt[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                xt[r] = *at(pt, ro[r + 1]);
                if (primed || !carried) {
                    double f = 0.0;
                    if (k > 0)
                        f = *at(A.W + (size_t)k * plane, ro[r + 1]) *
                            (g.wlo[k] * *at(pt - plane, ro[r + 1]) + g.whi[k] * xt[r]);
                    fb[r] = __double_as_longlong(f);
                }
            }
            primed = false;
            carried = true;
            // ds: T^{s-1} of the row to the south (DIFF: the difference from it)
            double fs = s[kV * 32] * (hs + xt[0]), ds = DIFF ? xd[0] - es : es;
            if (WALLS && j0 == 0) fs = 0.0;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                double fw = s[(kU + r) * 32] * (__shfl_up_sync(0xffffffffu, xt[r], 1) + xt[r]);
                if (WALLS && !xin) fw = 0.0;
                const double fe = __shfl_down_sync(0xffffffffu, fw, 1);
                double dx;                                // the two x neighbours (DIFF: the second difference)
                if constexpr (DIFF) {
                    dx = xd[r] - __shfl_up_sync(0xffffffffu, xd[r], 1);
                    dx = __shfl_down_sync(0xffffffffu, dx, 1) - dx;
                } else {
                    dx = __shfl_up_sync(0xffffffffu, xd[r], 1) + __shfl_down_sync(0xffffffffu, xd[r], 1);
                }
                const double tn = r + 1 < R ? xt[r + 1 < R ? r + 1 : r] : hn, dn = r + 1 < R ? xd[r + 1 < R ? r + 1 : r] : en;
                double fn = s[(kV + r + 1) * 32] * (xt[r] + tn);
                if (WALLS && j0 + r + 1 >= g.Ny) fn = 0.0;
                const double ft = top ? 0.0 : s[(kW + r) * 32] * (L.wlo * xt[r] + L.whi * rt[r]);
                const double below = k > 0 ? *at(pd - plane, ro[r + 1]) : pl;
                double sum;
                if constexpr (DIFF) {
                    const double dd = dn - xd[r];
                    sum = g.kx2 * dx + g.ky2 * (dd - ds) + L.cup * (rd[r] - xd[r]) - L.cdn * (xd[r] - below);
                    ds = dd;
                } else {
                    sum = g.kx2 * dx + g.ky2 * (ds + dn) + L.cdn * below + L.cup * rd[r] + L.ndiag * xd[r];
                    ds = xd[r];
                }
                sum = fma(L.iz, __longlong_as_double(fb[r]) - ft, fma(g.hy, fs - fn, fma(g.hx, fw - fe, sum)));
                if (mine && j0 + r < g.Ny)
                    *const_cast<double*>(at(A.out + (size_t)k * plane, ro[r + 1])) =
                        LF ? fma(A.gdt, sum, xd[r]) : fma(A.gdt, sum, A.a * xd[r] + A.b * xt[r]);
                fs = fn;
                fb[r] = __double_as_longlong(ft);
            }
        } else {
            carried = false;
            const LayerK& L = sk[k - k0];
            // the row south of the tile, and the flux through its first south face
            const long long ths = dec<60>(hs, E), thn = dec<60>(hn, E);
            long long ds = dec<60>(es, E);
            long long fs = mul(bal(ths + t[0]), bal(dec<62>(s[kV * 32], EV)));
            if (WALLS && j0 == 0) fs = 0;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const long long tt = dec<60>(rt[r], E), dt = dec<60>(rd[r], E);
                // x: the west face's flux, the east one from the next lane
                long long fw = mul(bal(__shfl_up_sync(0xffffffffu, t[r], 1) + t[r]), bal(dec<62>(s[(kU + r) * 32], EU)));
                if (WALLS && !xin) fw = 0;
                const long long fe = __shfl_down_sync(0xffffffffu, fw, 1);
                const long long dx = __shfl_up_sync(0xffffffffu, d[r], 1) + __shfl_down_sync(0xffffffffu, d[r], 1);
                const long long tn = r + 1 < R ? t[r + 1 < R ? r + 1 : r] : thn;
                const long long dn = r + 1 < R ? d[r + 1 < R ? r + 1 : r] : dec<60>(en, E);
                long long fn = mul(bal(t[r] + tn), bal(dec<62>(s[(kV + r + 1) * 32], EV)));
                if (WALLS && j0 + r + 1 >= g.Ny) fn = 0;
                const long long ft = top ? 0 : zflux(bal(t[r]), bal(tt), L.wlo, L.whi, bal(dec<62>(s[(kW + r) * 32], EW)));
                const Bal dc = bal(d[r]);
                Acc a{0, 1ll << 31};                      // rounds the sum
                mac(a, sc[0], bal(fw - fe));
                mac(a, sc[1], bal(fs - fn));
                mac(a, L.hz, bal(fb[r] - ft));
                mac(a, sc[2], bal(dx));
                mac(a, sc[3], bal(ds + dn));
                mac(a, L.cdn, db[r]);
                mac(a, L.cup, bal(dt));
                mac(a, L.ndiag, dc);
                const long long sum = madw((int)(a.M >> 32), 1, a.H);
                if (mine && j0 + r < g.Ny) {
                    double x;
                    if (LF) x = fma(gs, (double)sum, xd[r]);
                    else x = fma(gs, (double)sum, A.a * xd[r] + A.b * *at(pt, ro[r + 1]));
                    *const_cast<double*>(at(A.out + (size_t)k * plane, ro[r + 1])) = x;
                }
                // on to the next row; t, d of this one become the plane above
                fs = fn;
                ds = d[r];
                fb[r] = ft;
                db[r] = dc;
                t[r] = tt;
                d[r] = dt;
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) xd[r] = rd[r];
        mB = mC;
        mC = mN;
    }
}

template <int R>
cudaError_t launch_r(Args& A, bool lf, cudaStream_t st)
{
    const Grid<double>& g = A.g;
    const int form = g.walls ? 2 : (A.zs != 1.0 ? 1 : 0);  // walled; periodic implicit; periodic explicit
    void (*const forms[6])(const Args) = {k_step_fix<R, false, false, false>, k_step_fix<R, false, false, true>,
                                          k_step_fix<R, false, true, false>,  k_step_fix<R, false, true, true>,
                                          k_step_fix<R, true, true, false>,   k_step_fix<R, true, true, true>};
    void (*const k)(const Args) = forms[2 * form + lf];
    constexpr int smem = kWarps * 2 * stage_rows(R) * 32 * (int)sizeof(double);
    static unsigned long long done[6];                    // one bit per device, for each form
    cudaError_t e = smem_optin(reinterpret_cast<const void*>(k), smem, &done[2 * form + lf]);
    if (e != cudaSuccess) return e;
    // The chunks of layers: as many as give the shortest run, the rounds of
    // resident blocks times the layers of a chunk, each chunk's start counted as
    // kStart layers.
    const long long line = (long long)((g.Ny + R - 1) / R - 1) * band_span(g.Nx) + g.Nx;
    const long long blocks = (line + kCols * kWarps - 1) / (kCols * kWarps);
    const long long slots = 152LL * kBlocks;
    double best = 1e300;
    for (int n = (g.Nz + kMaxChunk - 1) / kMaxChunk; n <= g.Nz; ++n) {
        const int kc = (g.Nz + n - 1) / n;
        const double cost = (double)((blocks * ((g.Nz + kc - 1) / kc) + slots - 1) / slots) * (kc + kStart);
        if (cost < best * 0.999) {
            best = cost;
            A.kc = kc;
        }
    }
    const dim3 grd((unsigned)blocks, (unsigned)((g.Nz + A.kc - 1) / A.kc));
    return launch_after(k, grd, 32 * kWarps, smem, st, A);
}

}  // namespace

// Grids it takes: 32-bit byte offsets inside a plane, second-order faces, and at
// least 196,608 cells.  On small grids too few warps march too long a chain, and one
// thread per cell in FP64 arithmetic (mr_step.cu) is as fast or faster.  us per step
// here and there, M = 2, steps back to back:
//   cells      periodic        walled          implicit z (either)
//   32,768     5.5    3.1      5.7    4.9      12.3   12.3
//   69,120     7.2    6.8      7.0   10.7      14.4   18.5
//   110,592   10.4   10.3     10.4   13.8      16.4   22.6
//   153,088   10.5   10.3     10.5   13.8      18.5   22.6
//   196,608   14.9   12.4     14.9   21.9      20.4   28.7
//   317,440   15.2   21.5     15.0   34.9      24.6   47.2
// The line is where periodic explicit grids cross for good, and it is one for all
// forms; walled and implicit grids would gain from about 50,000 cells on.
bool step_fix_fits(const Grid<double>& g)
{
    const size_t row = (size_t)(g.ufx > g.Nx ? g.ufx : g.Nx), rows = (size_t)(g.vfy > g.Ny ? g.vfy : g.Ny);
    return row * rows < (1ull << 29) && !g.order4 && (size_t)g.Nx * g.Ny * g.Nz >= 196608;
}

cudaError_t launch_step_fix(const Grid<double>& g, const double* Us, const double* Vs, const double* Ws,
                            const double* Tm1, const double* T, double* Tp1, StepCoef c, bool implz,
                            const unsigned* vmax, cudaStream_t st)
{
    Args A;
    A.g = g;
    A.U = Us; A.V = Vs; A.W = Ws; A.Tm1 = Tm1; A.T = T; A.out = Tp1;
    A.a = c.a; A.b = c.b; A.gdt = c.gdt;
    A.zs = implz ? 0.5 : 1.0;
    A.plate = implz ? 1.0 : 0.5;
    A.vmax = vmax;
    return launch_r<kRows>(A, c.a == 1.0 && c.b == 0.0, st);
}

}  // namespace mr
