// One FP64 backward step of the adjoint (mr_adjoint.cu: k_adj_step) with the
// adjoint's advection and diffusion in 64-bit fixed point on the integer pipes
// (mr_fix.cuh; the forward's counterpart and the reasons for the layout are in
// mr_step64.cu) and the face gradients in FP64.
//
// Per cell  mu^s += b M + gdt C^T M,  mu^{s-1} = direct + a M + gdt D^T M  with
// M = mu^{s+1}:
//   C^T M = hx (u_w d_w + u_e d_e) + hy (v_s d_s + v_n d_n)
//           + (w_hi w_b d_b + w_lo' w_t d_t) / dz
//   D^T M = kx2 (d_e - d_w) + ky2 (d_n - d_s) + cup d_t - cdn d_b
// d being the differences of M across the faces (M is zero beyond the plates, and
// mirrored at side walls).  Each product u d is formed once per face.  M is a 59-bit
// integer relative to the largest value the warp's layer reads (so that the sums
// below stay under 2^63).  The face gradients gU += c (T_w + T_c) d_w, ... keep
// their FP64 arithmetic, differences of M included: they are sums over a run that
// the coarse gradients cancel to 1e-4 of themselves, so that a product error
// relative to the warp's largest M would show there.  That leaves 26 FP64 instructions
// per cell (23 and 2.6 conversions), which is what bounds it: the FP64 pipes are 80 %
// busy while it runs.  128 x 128 x 96 cells 82 us per step, 130 us in FP64 arithmetic
// throughout.  Rows x blocks per SM on the 40-step gradient: 2 x 4 8.6 ms, 3 x 3 8.6,
// 2 x 3 8.9, 1 x 6 9.6, 2 x 5 (spills) 9.6, before the layers' gradient factors moved
// to shared memory and comparisons to integers (2 x 4: 7.3).
// Layers of very uneven, infinite or NaN values are done in FP64 arithmetic.
#include "mr_fix.cuh"
#include "mr_internal.cuh"

namespace mr {
namespace {

using namespace fix;

constexpr int kWarps = 4;            // warps per block (independent of each other)
constexpr int kCols = 30;            // columns a warp writes
constexpr int kRows = 2;             // rows a warp writes
constexpr int kBlocks = 4;           // resident blocks per SM
constexpr int kStart = 3;            // a chunk's start, in layers
constexpr int kSpan = 6;             // binades below the warp's largest value that a lane may lie
constexpr int kMaxChunk = 32;        // layers per chunk
constexpr int kMaxRate = 7;          // binades that the step's rates gdt 2^eR may reach (mr_step64.cu; a stable step: 2^7)
constexpr int kFieldLo = 1023 - 300, kFieldHi = 1023 + 300;   // exponent fields of scales

// The constants of the layers of a block's chunk, scaled by 2^(62 - eR), and the
// factors of their face gradients.
struct LayerK {
    Bal zb, zt, cup, ncdn;           // 4 S_W w_hi / dz (bottom face), 4 S_W w_lo / dz (top face), cup, -cdn
};
struct LayerG {
    double ex, ey, lo, hi;           // gdt dy dz / 2, gdt dx dz / 2, gdt dx dy times the bottom face's weights
};

struct Args {
    Grid<double> g;
    const double *U, *V, *W, *T, *Tprev, *Mn;
    double *Mc, *Mp, *gU, *gV, *gW;
    double s_nu, s_var, mean_prev, a, b, gdt;
    double cx, cy, cz;               // face-gradient factors: gdt dy / 2, gdt dx / 2 (per dz_k), gdt dx dy
    const unsigned* vmax;
    int kc;
    bool has_b, has_var;             // b, s_var other than 0
};

constexpr int stage_rows(int R) { return 9 * R + 4; }

template <int R, bool WALLS, bool EULER>
__global__ void __launch_bounds__(32 * kWarps, kBlocks) k_adj_fix(const Args A)
{
    after_previous();
    let_next();
    const Grid<double>& g = A.g;
    __shared__ LayerK sk[kMaxChunk];
    __shared__ LayerG sg[kMaxChunk];
    __shared__ Bal sc[4];                                 // 4 S_U hx, 4 S_V hy, kx2, ky2
    const int k0 = blockIdx.y * A.kc, k1 = min(k0 + A.kc, g.Nz);
    const int lane = threadIdx.x & 31;
    const int EU = max((int)(A.vmax[0] >> 20), kFieldLo), EV = max((int)(A.vmax[1] >> 20), kFieldLo),
              EW = max((int)(A.vmax[2] >> 20), kFieldLo);
    bool usable = EU <= kFieldHi && EV <= kFieldHi && EW <= kFieldHi;
    int eR;
    {
        unsigned m = 0;                                   // positive values are ordered like their high words
        for (int k = k0 + lane; k < k1; k += 32)
            m = max(m, (unsigned)__double2hiint(8.0 * g.inv_dz[k] * pow2(EW - 1022) + 2.0 * (g.cdn[k] + g.cup[k])));
        m = __reduce_max_sync(0xffffffffu, m);
        const double r = __hiloint2double((int)m + 1, 0) + 4.0 * (g.hx * pow2(EU - 1022) + g.hy * pow2(EV - 1022)) +
                         4.0 * (g.kx2 + g.ky2);
        eR = exponent(r);                                 // 2^eR > r
        usable = usable && eR > -400 && eR < 400 && exponent(A.gdt) + eR <= kMaxRate;
    }
    for (int q = threadIdx.x; q < k1 - k0; q += blockDim.x) {
        const int k = k0 + q;
        sg[q] = LayerG{A.cx * g.dz[k], A.cy * g.dz[k], A.cz * g.wlo[k], A.cz * g.whi[k]};
    }
    if (usable) {
        for (int q = threadIdx.x; q < k1 - k0; q += blockDim.x) {
            const int k = k0 + q;
            const double p = pow2(62 - eR), z = g.inv_dz[k] * pow2(EW - 1020 + 62 - eR);
            sk[q] = LayerK{fixed(g.whi[k] * z), fixed(g.wlo[k + 1] * z), fixed(g.cup[k] * p), fixed(-(g.cdn[k] * p))};
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
    // byte offsets in a plane: rows j0-1 .. j0+R; U rows; V faces j0 .. j0+R
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

    // A warp's staging area, filled one layer ahead: M of the rows on plane k + 1, the
    // rows beyond the tile of M (both) and T (south) and T's rows on plane k, U, V
    // faces, W on plane k + 1, the three face gradients and mu^s.
    constexpr int kM = 0, kH = R, kT = R + 2, kS = 2 * R + 2, kU = 2 * R + 3, kV = 3 * R + 3, kW = 4 * R + 4, kGU = 5 * R + 4,
                  kGV = 6 * R + 4, kGW = 7 * R + 4, kMC = 8 * R + 4;
    extern __shared__ double stage_all[];
    double* stage = stage_all + (size_t)(threadIdx.x >> 5) * 2 * stage_rows(R) * 32 + lane;
    auto fetch = [&](int k) {
        double* s = stage + (k & 1) * stage_rows(R) * 32;
        const double *pm = A.Mn + (size_t)k * plane, *pmn = pm + plane, *pt = A.T + (size_t)k * plane;
        if (k + 1 < g.Nz) {
#pragma unroll
            for (int r = 0; r < R; ++r) copy8(s + (kM + r) * 32, at(pmn, ro[r + 1]));
        }
        copy8(s + (kH + 0) * 32, at(pm, ro[0]));
        copy8(s + (kH + 1) * 32, at(pm, ro[R + 1]));
        copy8(s + kS * 32, at(pt, ro[0]));
        const double *pu = A.U + (size_t)k * uplane, *pv = A.V + (size_t)k * vplane, *pw = A.W + (size_t)(k + 1) * plane;
        const double *qu = A.gU + (size_t)k * uplane, *qv = A.gV + (size_t)k * vplane, *qw = A.gW + (size_t)k * plane,
                     *qm = A.Mc + (size_t)k * plane;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            copy8(s + (kT + r) * 32, at(pt, ro[r + 1]));
            copy8(s + (kU + r) * 32, at(pu, uo[r]));
            copy8(s + (kW + r) * 32, at(pw, ro[r + 1]));
            copy8(s + (kGU + r) * 32, at(qu, uo[r]));
            copy8(s + (kGV + r) * 32, at(qv, vo[r]));
            copy8(s + (kGW + r) * 32, at(qw, ro[r + 1]));
            copy8(s + (kMC + r) * 32, at(qm, ro[r + 1]));
        }
#pragma unroll
        for (int f = 0; f <= R; ++f) copy8(s + (kV + f) * 32, at(pv, vo[f]));
    };

    // state at layer k: M of the rows on plane k, its difference and product w d across
    // the bottom faces (fixed point, scale E), M on planes k and k - 1 and T on plane
    // k - 1 as they are, and the lane's largest magnitudes on planes k - 1 and k
    long long m[R], db[R], qb[R];
    double xm[R], xb[R], tb[R];
    unsigned mB = 0, mC = 0;
    int E = 0;
    bool primed = false;
    double gs = 0.0;
    fetch(k0);
    copy_commit();
    {
        const double *pm = A.Mn + (size_t)k0 * plane, *pt = A.T + (size_t)k0 * plane;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            xm[r] = *at(pm, ro[r + 1]);
            xb[r] = k0 > 0 ? *at(pm - plane, ro[r + 1]) : 0.0;
            tb[r] = k0 > 0 ? *at(pt - plane, ro[r + 1]) : 0.0;
            mC = max(mC, mag(xm[r]));
            mB = max(mB, mag(xb[r]));
        }
    }
    for (int k = k0; k < k1; ++k) {
        const bool top = k == g.Nz - 1;
        const double* s = stage + (k & 1) * stage_rows(R) * 32;
        copy_wait<0>();                                   // this layer's copies, and no later ones yet
        __syncwarp();                                     // every lane's: T is read across lanes, and the other half is free
        if (k + 1 < k1) fetch(k + 1);
        copy_commit();
        double rm[R];
        unsigned mN = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            rm[r] = top ? 0.0 : s[(kM + r) * 32];
            mN = max(mN, mag(rm[r]));
        }
        const double hs = s[(kH + 0) * 32], hn = s[(kH + 1) * 32];
        const unsigned ml = max(max(max(mB, mC), mN), max(mag(hs), mag(hn)));
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
                gs = A.gdt * pow2(E + eR - 1079);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    m[r] = dec<59>(xm[r], E);
                    db[r] = m[r] - (k > 0 ? dec<59>(xb[r], E) : 0);
                    qb[r] = k > 0 ? mul(bal(db[r]), bal(dec<62>(*at(A.W + (size_t)k * plane, ro[r + 1]), EW))) : 0;
                }
            }
            plain = !ordinary(gs);
        }
        if (plain) primed = false;
        // the sums C^T M and D^T M of the rows, in FP64 or in units of gs / gdt
        double ct[R], dt_[R];
        if (plain) {
            const double* pw = A.W + (size_t)k * plane;
            double ds = xm[0] - hs, fs = s[kV * 32] * ds;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const double dw = xm[r] - __shfl_up_sync(0xffffffffu, xm[r], 1), fw = s[(kU + r) * 32] * dw;
                const double de = __shfl_down_sync(0xffffffffu, dw, 1), fe = __shfl_down_sync(0xffffffffu, fw, 1);
                const double dn = (r + 1 < R ? xm[r + 1 < R ? r + 1 : r] : hn) - xm[r], fn = s[(kV + r + 1) * 32] * dn;
                const double d0 = xm[r] - xb[r], d1 = rm[r] - xm[r];
                double z = 0.0;
                if (k > 0) z = (*at(pw, ro[r + 1]) * g.whi[k]) * d0;
                if (!top) z += (s[(kW + r) * 32] * g.wlo[k + 1]) * d1;
                ct[r] = g.hx * (fw + fe) + g.hy * (fs + fn) + g.inv_dz[k] * z;
                dt_[r] = g.kx2 * (de - dw) + g.ky2 * (dn - ds) + g.cup[k] * d1 - g.cdn[k] * d0;
                ds = dn;
                fs = fn;
            }
        } else {
            const LayerK& L = sk[k - k0];
            const long long mnh = dec<59>(hn, E);
            long long ds = m[0] - dec<59>(hs, E), fs = mul(bal(ds), bal(dec<62>(s[kV * 32], EV)));
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const long long dw = m[r] - __shfl_up_sync(0xffffffffu, m[r], 1);
                const long long fw = mul(bal(dw), bal(dec<62>(s[(kU + r) * 32], EU)));
                const long long de = __shfl_down_sync(0xffffffffu, dw, 1), fe = __shfl_down_sync(0xffffffffu, fw, 1);
                const long long dn = (r + 1 < R ? m[r + 1 < R ? r + 1 : r] : mnh) - m[r];
                const long long fn = mul(bal(dn), bal(dec<62>(s[(kV + r + 1) * 32], EV)));
                const long long mt = top ? 0 : dec<59>(rm[r], E), d1 = mt - m[r];
                const Bal d1b = bal(d1);
                const long long qt = top ? 0 : mul(d1b, bal(dec<62>(s[(kW + r) * 32], EW)));
                Acc c{0, 1ll << 31}, d{0, 1ll << 31};     // round the sums
                mac(c, sc[0], bal(fw + fe));
                mac(c, sc[1], bal(fs + fn));
                mac(c, L.zb, bal(qb[r]));
                mac(c, L.zt, bal(qt));
                mac(d, sc[2], bal(de - dw));
                mac(d, sc[3], bal(dn - ds));
                mac(d, L.cup, d1b);
                mac(d, L.ncdn, bal(db[r]));
                const long long cs = madw((int)(c.M >> 32), 1, c.H), dsum = madw((int)(d.M >> 32), 1, d.H);
                if (EULER) {
                    ct[r] = (double)(cs + dsum);
                    dt_[r] = 0.0;
                } else {
                    ct[r] = (double)cs;
                    dt_[r] = (double)dsum;
                }
                ds = dn;
                fs = fn;
                db[r] = d1;
                qb[r] = qt;
                m[r] = mt;
            }
        }
        // the new levels, and the gradients of the west, south and bottom faces (FP64)
        const double f = plain ? A.gdt : gs;
        const LayerG& G = sg[k - k0];
        double south = hs, tsouth = s[kS * 32];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const double tc = s[(kT + r) * 32];
            const double west = __shfl_up_sync(0xffffffffu, xm[r], 1), tw = __shfl_up_sync(0xffffffffu, tc, 1);
            if (mine && j0 + r < g.Ny) {
                double c = s[(kMC + r) * 32];
                if (EULER) {
                    c += xm[r];
                    if (plain) c = fma(f, dt_[r], c);
                } else {
                    if (A.has_b) c = fma(A.b, xm[r], c);
                    double d = k == 0 ? A.s_nu : 0.0;
                    if (A.has_var) d += A.s_var * (*at(A.Tprev + (size_t)k * plane, ro[r + 1]) - A.mean_prev);
                    *const_cast<double*>(at(A.Mp + (size_t)k * plane, ro[r + 1])) = fma(f, dt_[r], fma(A.a, xm[r], d));
                }
                *const_cast<double*>(at(A.Mc + (size_t)k * plane, ro[r + 1])) = fma(f, ct[r], c);
                *const_cast<double*>(at(A.gU + (size_t)k * uplane, uo[r])) = fma(G.ex * (tw + tc), xm[r] - west, s[(kGU + r) * 32]);
                *const_cast<double*>(at(A.gV + (size_t)k * vplane, vo[r])) =
                    fma(G.ey * (tsouth + tc), xm[r] - south, s[(kGV + r) * 32]);
                if (k > 0)
                    *const_cast<double*>(at(A.gW + (size_t)k * plane, ro[r + 1])) =
                        fma(fma(G.lo, tb[r], G.hi * tc), xm[r] - xb[r], s[(kGW + r) * 32]);
            }
            south = xm[r];
            tsouth = tc;
            tb[r] = tc;
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            xb[r] = xm[r];
            xm[r] = rm[r];
        }
        mB = mC;
        mC = mN;
    }
}

}  // namespace

// Plane offsets below 2^32 bytes, and enough cells to fill the chip: gradients of 40
// steps, this kernel against k_adj_step_periodic: 32,768 cells 1.31 and 1.17 ms,
// 110,592 2.10 and 2.43, 196,608 2.54 and 2.60, 262,144 2.62 and 2.81, 512,000 3.49
// and 4.37.
bool adj_fix_fits(const Grid<double>& g)
{
    const size_t row = (size_t)(g.ufx > g.Nx ? g.ufx : g.Nx), rows = (size_t)(g.vfy > g.Ny ? g.vfy : g.Ny);
    return row * rows < (1ull << 29) && !g.order4 && (size_t)g.Nx * g.Ny * g.Nz >= 98304;
}

cudaError_t launch_adj_fix(const Grid<double>& g, const double* Us, const double* Vs, const double* Ws, const double* T,
                           const double* Tprev, const double* Mn, double* Mc, double* Mp, double s_nu, double s_var,
                           double mean_prev, double* gU, double* gV, double* gW, StepCoef c, bool euler,
                           const unsigned* vmax, cudaStream_t st)
{
    constexpr int R = kRows;
    Args A;
    A.g = g;
    A.U = Us; A.V = Vs; A.W = Ws; A.T = T; A.Tprev = Tprev; A.Mn = Mn;
    A.Mc = Mc; A.Mp = Mp; A.gU = gU; A.gV = gV; A.gW = gW;
    A.s_nu = s_nu; A.s_var = s_var; A.mean_prev = mean_prev;
    A.a = c.a; A.b = c.b; A.gdt = c.gdt;
    A.cx = 0.5 * c.gdt * g.dy;
    A.cy = 0.5 * c.gdt * g.dx;
    A.cz = c.gdt * (g.dx * g.dy);
    A.vmax = vmax;
    A.has_b = c.b != 0.0;
    A.has_var = s_var != 0.0;
    void (*const k)(const Args) = g.walls ? (euler ? k_adj_fix<R, true, true> : k_adj_fix<R, true, false>)
                                          : (euler ? k_adj_fix<R, false, true> : k_adj_fix<R, false, false>);
    constexpr int smem = kWarps * 2 * stage_rows(R) * 32 * (int)sizeof(double);
    static unsigned long long done[4];                    // one bit per device, for each form
    cudaError_t e = smem_optin(reinterpret_cast<const void*>(k), smem, &done[2 * (g.walls != 0) + euler]);
    if (e != cudaSuccess) return e;
    // the chunks of layers that give the shortest run (as in the forward step)
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

}  // namespace mr
