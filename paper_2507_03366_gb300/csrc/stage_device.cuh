// stage_device.cuh -- the parts of one SSP-RK3 stage (Eq. 58) of the EULBFS
// explicit step that both stage kernels are built from: the ring of derived
// rows, boundary rows, mu_c, the face fluxes, the cell update, and the waits
// between the work items of a launch.
//
// The face computation is written in the face frame (n, t): an x-face has
// n = x, t = y and a y-face n = y, t = x (D2Q9 is symmetric under the swap).
// With dt_s = 0.5 the surrounding points x_f - e_a dt_s of a face are the two
// cell centres (e_n = +-1, e_t = 0), the two cells' extrapolations half a cell
// along t (e_n = +-1, e_t = +-1) and three points on the face itself (e_n = 0),
// which take the mean of the two one-sided reconstructions (Eq. 54, R7).
#pragma once
#include "device_common.cuh"

namespace eulbfs {

namespace {

constexpr int RW = kStripX + 2 * kHalo;   // ring columns: strip plus halo (37)
constexpr int RING = 16;                  // ring rows (power of two)

// Two fields of a cell side by side, read and written with one 8-byte
// (FP64: 16-byte) shared-memory access.
template <class R> struct Pair;
template <> struct Pair<float> { using T = float2; };
template <> struct Pair<double> { using T = double2; };
template <class R> using P2 = typename Pair<R>::T;


// Derived fields of the ring rows (row r in slot r & 15), paired by the
// places that read them together: every face point needs (u, v), (rho, C)
// and (T, C_p); p is needed at every point and mu_c at the cell and outer
// n-neighbours; lambda and mu only at the face.
template <class R>
struct Ring {
    P2<R> uv[RING][RW];       // u, v
    P2<R> rc[RING][RW];       // rho, C
    P2<R> tc[RING][RW];       // T, C_p
    P2<R> pm[RING][RW];       // p, mu_c
    P2<R> lm[RING][RW];       // lambda, mu
    R fl[RING][RW];           // F_l
};

// What both stage kernels keep in shared memory.
template <class R>
struct Core {
    Ring<R> P;
    // face fluxes in pairs (F_h, F_p), (F_mx, F_my), (F_C, u_n): y-faces in a
    // ring of face rows, x-faces of the current rows
    P2<R> YF[3][RING][32];
    P2<R> XF[3][kChunk][32];
    Consts<R> K;
    R inv_rc[RW];    // axisymmetric domains: 1 / r of the ring columns' cells
    R rw[sizeof(R) == 8 ? RW : 1];   // and the radius of their left faces (FP64: conversions are slow)
};

// The radius of the left face of ring column cc (column gx of the domain).
__device__ __forceinline__ float left_radius(const Core<float>&, int, int gx) { return (float)gx; }
__device__ __forceinline__ double left_radius(const Core<double>& S, int cc, int) { return S.rw[cc]; }

// 1 / r of the strip's ring columns (used by mu_c; every CTA thread calls it
// before the barrier that ends the item's first load phase).
template <class R, bool AXI>
__device__ __forceinline__ void column_radii(Core<R>& S, int x0) {
    if (AXI && threadIdx.x < RW) {
        const R rw = (R)(x0 + (int)threadIdx.x - kHalo);
        S.inv_rc[threadIdx.x] = wdiv(R(1), rw + R(0.5));
        if (sizeof(R) == 8) S.rw[threadIdx.x] = rw;
    }
}

__device__ __forceinline__ int slot(int r) { return r & (RING - 1); }

// Position g of a launch's item sequence: its stage (counted over the
// launch: 3 k + s for Runge-Kutta stage s of the launch's step k) and work item.
__device__ __forceinline__ int2 stage_item(const StageLaunch& a, int g) {
    if (a.stages == 1) return make_int2(a.stage, g);
    const int st = g / a.nitems;
    return make_int2(st, g - st * a.nitems);
}

__device__ __forceinline__ int ld_acquire(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Step 1: rows [r0, r0 + nrows) of the strip (all RW columns).
template <class R>
__device__ __forceinline__ void store_prim(Core<R>& S, int s, int cc, const Prim<R>& q) {
    S.P.uv[s][cc] = P2<R>{q.u, q.v};
    S.P.rc[s][cc] = P2<R>{q.rho, q.C};
    S.P.tc[s][cc] = P2<R>{q.T, q.cp};
    S.P.pm[s][cc].x = q.p;     // mu_c follows in step 2
    S.P.lm[s][cc] = P2<R>{q.lam, q.mu};
    S.P.fl[s][cc] = q.Fl;
}

// NTH: threads of the CTA.
template <class R, int NTH>
__device__ __forceinline__ void load_rows(Core<R>& S, const R* in, int x0, int r0, int nrows) {
    const Consts<R>& K = S.K;
    const int total = nrows * RW;
    if (x0 >= kHalo && x0 + kStripX + kHalo <= K.nx && r0 >= -K.hlo && r0 + nrows <= K.ny + K.hhi) {
        // every cell of these rows is inside the domain (or a slab's halo):
        // no boundary mapping
        const long long base = (long long)r0 * K.nx + (x0 - kHalo) + K.off;
        for (int idx = threadIdx.x; idx < total; idx += NTH) {
            const int rr = idx / RW, cc = idx - rr * RW;
            const SV<R> w = load_state(in, K.plane, base + (long long)rr * K.nx + cc);
            store_prim(S, slot(r0 + rr), cc, derive(K, w));
        }
        return;
    }
    for (int idx = threadIdx.x; idx < total; idx += NTH) {
        const int rr = idx / RW, cc = idx - rr * RW;
        const int gy = r0 + rr, gx = x0 + cc - kHalo;
        int sx, kx, sdx, sy, ky, sdy;
        map_axis(gx, K.nx, K.per_x, XLO, sx, kx, sdx);
        map_row(K, gy, sy, ky, sdy);
        const SV<R> w = load_state(in, K.plane, (long long)sy * K.nx + sx + K.off);
        Prim<R> q = derive(K, w);
        // x sides first, then y (corners); an x ghost takes the wetting of its
        // (interior) row, a y ghost that of its column
        if (kx) apply_ghost(K, sdx, kx, true, wall_wetting(K, in, sdx, sy), q);
        if (ky) apply_ghost(K, sdy, ky, false, wall_wetting(K, in, sdy, gx), q);
        store_prim(S, slot(gy), cc, q);
    }
}

// mu_c = 2 beta C (C-1)(2C-1) - kappa lap C (reading R5) at ring offset s0
// with the y-neighbours at sN, sS.  The Laplacian is the 5-point one, or in an
// axisymmetric domain the conservative (1/r) d/dr (r dC/dr) + d2C/dz2 with
// faces at r = rw and rw + 1.
template <class R, bool AXI>
__device__ __forceinline__ R chem_potential_of(const Consts<R>& K, R c, R ce, R cw, R cn, R cs, R rw, R inv_rc) {
    R lap;
    if (AXI) {
        const R re = rw + R(1);
        lap = fma(fma(re, ce - c, -(rw * (c - cw))), inv_rc, fma(R(-2), c, cn + cs));
    } else {
        lap = fma(R(-4), c, ce + cw + cn + cs);
    }
    const Q4<R> cc = ld4(K.cellc2);   // 2 beta, kappa
    // (explicit FMAs: every place that inlines this has to round alike)
    return fma(-cc.y, lap, cc.x * c * (c - R(1)) * fma(R(2), c, R(-1)));
}

template <class R, bool AXI>
__device__ __forceinline__ R chem_potential(const Core<R>& S, int cc, int sc, int sN, int sS, int x0) {
    const P2<R>* RC = &S.P.rc[0][0];
    return chem_potential_of<R, AXI>(S.K, RC[sc].y, RC[sc + 1].y, RC[sc - 1].y, RC[sN].y, RC[sS].y,
                                     AXI ? left_radius(S, cc, x0 + cc - kHalo) : R(0), AXI ? S.inv_rc[cc] : R(0));
}

// True if mu_c of rows [r0, r0 + nrows) of the strip involves no wall ghost
// (the in-place Laplacian of muc_rows' first branch applies to all of them).
template <class R>
__device__ __forceinline__ bool muc_in_place(const Consts<R>& K, int x0, int r0, int nrows) {
    const int rlo = K.hlo ? 1 - K.hlo : 0, rhi = K.hhi ? K.ny + K.hhi - 1 : K.ny;
    return x0 >= kHalo - 1 && x0 + (RW - 2) - (kHalo - 1) <= K.nx && r0 >= rlo && r0 + nrows <= rhi;
}

// Step 2: mu_c for rows [r0, r0 + nrows), columns 1 .. RW-2.  A wall ghost
// (layer 1 or 2) evaluates mu_c at its mirror cell, which equals mirroring
// the interior value; deeper layers are never read by a face of the strip
// and get 0.
template <class R, bool AXI, int NTH>
__device__ __forceinline__ void muc_rows(Core<R>& S, int x0, int r0, int nrows) {
    const Consts<R>& K = S.K;
    constexpr int NC = RW - 2;
    const int total = nrows * NC;
    // a slab's halo rows take mu_c in place, except the outermost (never read)
    const int rlo = K.hlo ? 1 - K.hlo : 0, rhi = K.hhi ? K.ny + K.hhi - 1 : K.ny;
    if ((K.per_x || (x0 >= kHalo - 1 && x0 + NC - (kHalo - 1) <= K.nx)) &&
        (K.per_y || (r0 >= rlo && r0 + nrows <= rhi))) {
        // no wall ghost among these cells: the Laplacian in place
        for (int idx = threadIdx.x; idx < total; idx += NTH) {
            const int rr = idx / NC, cc = 1 + idx - rr * NC;
            const int gy = r0 + rr;
            const int s0 = slot(gy) * RW + cc;
            S.P.pm[slot(gy)][cc].y =
                chem_potential<R, AXI>(S, cc, s0, slot(gy + 1) * RW + cc, slot(gy - 1) * RW + cc, x0);
        }
        return;
    }
    for (int idx = threadIdx.x; idx < total; idx += NTH) {
        const int rr = idx / NC, cc = 1 + idx - rr * NC;
        const int gy = r0 + rr, gx = x0 + cc - kHalo;
        int mc = cc, my = gy, deep = 0;
        if (!K.per_x) {
            if (gx < 0) { const int k = -gx; mc = cc + 2 * k - 1; deep |= k > 2; }
            else if (gx >= K.nx) { const int k = gx - K.nx + 1; mc = cc - (2 * k - 1); deep |= k > 2; }
        }
        if (gy < 0 && K.hlo) {
            deep |= gy < rlo;
        } else if (gy >= K.ny && K.hhi) {
            deep |= gy >= rhi;
        } else if (!K.per_y) {
            if (gy < 0) { const int k = -gy; my = gy + 2 * k - 1; deep |= k > 2; }
            else if (gy >= K.ny) { const int k = gy - K.ny + 1; my = gy - (2 * k - 1); deep |= k > 2; }
        }
        R mu = R(0);
        if (!deep)
            mu = chem_potential<R, AXI>(S, mc, slot(my) * RW + mc, slot(my + 1) * RW + mc, slot(my - 1) * RW + mc, x0);
        S.P.pm[slot(gy)][cc].y = mu;
    }
}

// The 9 surrounding-point values of one field of a face (Eq. 54, R7), given
// the ring offsets of the L and R cells, their outer n-neighbours and their
// t-neighbours.
struct FaceIdx { int L, R, LL, RR, Lp, Lm, Rp, Rm; };

template <class R>
struct FaceFlux { R Fh, Fp, Fmn, Fmt, Fc, un; };

// Reconstruction pieces of one field: the cell values l, r, eight times the
// face value f8 (the face value is the mean of the two one-sided
// reconstructions l + (r - ll)/4 and r - (rr - l)/4, i.e. 5/8 (l + r) -
// 1/8 (ll + rr); powers of two are left to the constants it meets) and the
// central t-differences dtl, dtr of the two cells (half-cell t-step = dt / 4).
template <class R>
struct Rec { R l, r, f8, dtl, dtr; };

template <class R>
__device__ __forceinline__ R face_value8(R l, R r, R ll, R rr) {
    return fma(R(5), l + r, -(ll + rr));
}

template <class R>
__device__ __forceinline__ Rec<R> rec_of(R l, R r, R ll, R rr, R lp, R lm, R rp, R rm) {
    Rec<R> z;
    z.l = l;
    z.r = r;
    z.f8 = face_value8(l, r, ll, rr);
    z.dtl = lp - lm;
    z.dtr = rp - rm;
    return z;
}

// The reconstruction pieces of both fields of a pair.
template <class R>
__device__ __forceinline__ void rec2(const P2<R>* f, const FaceIdx& x, Rec<R>& a, Rec<R>& b) {
    const P2<R> l = f[x.L], r = f[x.R], ll = f[x.LL], rr = f[x.RR];
    const P2<R> lp = f[x.Lp], lm = f[x.Lm], rp = f[x.Rp], rm = f[x.Rm];
    a = rec_of(l.x, r.x, ll.x, rr.x, lp.x, lm.x, rp.x, rm.x);
    b = rec_of(l.y, r.y, ll.y, rr.y, lp.y, lm.y, rp.y, rm.y);
}

// Eight times the face values of both fields of a pair (cells L, R and their outer
// n-neighbours).
template <class R>
__device__ __forceinline__ void face_value8_2(const P2<R>* f, const FaceIdx& x, R& a, R& b) {
    const P2<R> l = f[x.L], r = f[x.R], ll = f[x.LL], rr = f[x.RR];
    a = face_value8(l.x, r.x, ll.x, rr.x);
    b = face_value8(l.y, r.y, ll.y, rr.y);
}

// What one side column of a face adds to its moments: the points
// x_f - e_a dt_s with e_n = SN (+1: the L cell, points 1, 5, 8; -1: the R cell,
// points 3, 6, 7).  The column's centre point (e_t = 0) takes the cell values;
// its t-points (e_t = +1 / -1) the cell value minus / plus a quarter d of the
// central t-difference.  With q = e.u + 3/2 (e.u)^2 - 1/2 u^2 (cs^2 = 1/3):
//   centre:   q0 = SN u_n + u_n^2 - u_t^2 / 2
//   t-points: q = e.u (1 + e.u) + e_n e_t u_n u_t, where with
//             A = SN u_n - d u_t, B = u_t - SN d u_n:  e.u = A + B and A - B,
// so that the two t-points' half sum and half difference of q are
//   hq = A + A^2 + B^2 - SN (u_n d u_t + d u_n u_t)
//   hd = B (1 + 2 A) + SN (u_n u_t + d u_n d u_t),
// and the half sum / difference of (f - / + df) q are f hq - df hd and
// f hd - df hq.  The weights of the centre (1/9) and the t-points (1/36, in pairs
// 1/18) then meet as V = 2 q0 + hq = 18 sum w q.  Per side, scaled:
//   X = rho V - d rho hd         18 x its part of sum f, of +- sum e_n f
//   F = rho hd - d rho hq        18 x its part of sum e_t f
//   G = C (2 SN u_n + A) - d C B    6 x its part of sum g, of +- sum e_n g
//   H = C_p T V + d C_p d T hq - (C_p d T + d C_p T) hd    6 x its part of +- sum e_n h
// The parts linear in p, mu_c and T stay out of them, so that the flux takes
// their differences across the face exactly.
// Folding the weights into V and so into X, G and H takes a face from about 237
// to 191 FP operations besides its division (against the t-points one by one and
// each moment from its own sums).  us per step: FP64, bound by its pipe, 16
// domains 6460 -> 5760, 256^2 348 -> 316; FP32C, bound by issue, the benchmark's 64
// domains (6.80 M cells) 1023 -> 977, 16 domains 260 -> 251, 512^2 63.6 -> 60.9.
// Constants like 1/6 are a biased 3e-8 in FP32: none stands on an undivided flux
// of mass, enthalpy or phase, or on the normal momentum flux.  The tangential
// momentum flux carries that of its 1/24, as it would that of cs^2 = 1/3.
template <class R>
struct SideTerms { R X, V, hd, F, G, H; };

template <class R, int SN>
__device__ __forceinline__ SideTerms<R> side_terms(R un, R ut, R rho, R C, R T, R cp, R dun, R dut, R drho, R dC,
                                                   R dT, R dcp) {
    constexpr R sg = SN > 0 ? R(1) : R(-1);
    const R sun = SN > 0 ? un : -un;
    const R A = fma(R(-0.25), dut, sun), B = fma(R(-0.25) * sg, dun, ut);
    const R hq = fma(R(-0.25) * sg, fma(dun, ut, un * dut), fma(B, B, fma(A, A, A)));
    SideTerms<R> s;
    s.hd = fma(R(1.0 / 16.0) * sg, dun * dut, fma(sun, ut, fma(R(2), A, R(1)) * B));
    s.V = fma(R(2), fma(un, un, fma(R(-0.5) * ut, ut, sun)), hq);
    const R dr = R(0.25) * drho;
    s.X = fma(rho, s.V, -(dr * s.hd));
    s.F = fma(rho, s.hd, -(dr * hq));
    s.G = fma(C, fma(R(2) * sg, un, A), -((R(0.25) * dC) * B));
    const R c4 = R(0.25) * dcp, t4 = R(0.25) * dT;
    s.H = fma(-fma(c4, T, cp * t4), s.hd, fma(c4 * t4, hq, (cp * T) * s.V));
    return s;
}

// Sec. 2.5 steps (2)-(4) and Eq. 53 for one face.
//
// The face equilibria enter only through their closed moments (C_p T u_n,
// cs^2 (p + rho u_n^2), cs^2 rho u_n u_t, C u_n; Eq. 11 and the moments of
// Eq. 29, 42).  The sums over the surrounding points x_f - e_a dt_s go by
// columns of equal e_n: the two side columns (side_terms) and the face column
// e_n = 0.  The parts linear in one reconstructed field have closed forms,
// because the reconstruction is linear (the t-offsets cancel in pairs):
//   sum w p = 2/3 p_0 + (p_L + p_R)/6          sum e_n w p = (p_L - p_R)/6
//   sum e_t w p = -(dp_L + dp_R)/24             sum e_n e_t w p = (dp_R - dp_L)/72
//   sum_{e_n != 0} w p = (p_L + p_R)/6
//   mu_c part of sum g = Q ((mu_L + mu_R)/2 - mu_0), of sum e_n g = Q (mu_L - mu_R)/2
//   C_ref T part of sum e_n h = C_ref (T_L - T_R)/6
// (dp = central t-difference).  Face-column values and t-steps are all carried
// times eight (f8, and the sum of the two cells' t-differences), so its terms
// come times 64 and, with rho, 512; the constants below undo that.
//
// Axisymmetric domains (reading R24): the face pressure is advanced with the
// axisymmetric mass source -rho cs^2 u_r / r as well, streamed with weight
// w_a over dt_s.  Of the fluxes only the normal momentum flux changes, by
// cs^2 dt_s (-rho_f cs^2 u_r / r) = -rho_f u_r / (18 r) with the face values;
// inv_r = 1 / r of the face (0 on the axis, where the face area is zero).
//
// The moments of the surrounding equilibria, scaled as above: 18 sum e_n f, 18 sum
// e_t f, 18 p_f, C_f, 6 sum e_n g; T_L - T_R and 6 x the rest of sum e_n h; and of
// f^eq-m the sum of V and the difference of hd of the two sides, p_L + p_R and
// 8 dt_f (dp_R - dp_L) / 2.
template <class R>
struct Moments { R mn, mt, pf, Cf, gn, dT, hn, V, hd, ps, dp; };

// From the moments to the fluxes; Cref6 = C_ref / 6, rho8, cpT64: 8 x rho and 64 x C_p T of the
// face, ir = 1 / rho8, th, tf: tau_h - 1/2 and tau_f - 1/2.
template <class R>
__device__ __forceinline__ FaceFlux<R> close_flux(const Consts<R>& K, const Moments<R>& m, R Cref6, R rho8, R cpT64, R ir,
                                                  R th, R tf) {
    // rho_f cs^2 u_f = sum e f^eq (Eq. 56)
    const R i43 = fma(R(1.0 / 3.0), ir, ir);              // 4/3 ir (a rounded 4/3 would bias every advective flux by 3e-8 in FP32)
    const R un = m.mn * i43, ut = m.mt * i43;
    const R ru = rho8 * un;                               // 8 rho_f u_n
    FaceFlux<R> F;
    // h* = (1.5 - tau) h^eq(x_f) + (tau - 0.5) h^eq(x_f - e dt_s) (Eq. 13, 16)
    const R fh = R(1.0 / 64.0) * (cpT64 * un);
    F.Fh = fma(th, fma(Cref6, m.dT, fma(R(1.0 / 6.0), m.hn, -fh)), fh);
    F.Fp = R(1.0 / 18.0) * m.mn;                          // sum e_n f^eq(x_f) = rho_f cs^2 u_n,f
    // f* = (1.5 - tau_f) f^eq(x_f) + (tau_f - 0.5) f^eq-m (Eq. 35, 37 with R3)
    const R nn = fma(R(2.25), ru * un, m.pf);             // 54 cs^2 (p_f + rho_f u_n^2)
    F.Fmn = R(1.0 / 54.0) * fma(tf, fma(R(0.375), rho8 * m.V, R(9) * m.ps) - nn, nn);
    const R nt = ru * ut;                                 // 24 cs^2 rho_f u_n u_t
    F.Fmt = R(1.0 / 24.0) * fma(tf, fma(R(1.0 / 6.0), fma(rho8, m.hd, m.dp), -nt), nt);
    F.Fc = fma(K.facet[0], m.Cf * un, K.facet[1] * m.gn);            // Eq. 44, 46
    F.un = un;
    return F;
}

template <class R, bool AXI, class Src>
__device__ __forceinline__ FaceFlux<R> face_math(const Consts<R>& K, const Src& src, R inv_r) {
    const Q4<R> fc = ld4(K.facek);   // 3 Q, 3 Q / 4, C_ref / 6, 6 / C_ref
    Rec<R> n, t, rho, C, T, cp, p, muc;
    src.vel(n, t);               // normal and tangential velocity
    src.rc(rho, C);
    src.tc(T, cp);
    const SideTerms<R> L = side_terms<R, 1>(n.l, t.l, rho.l, C.l, T.l, cp.l, n.dtl, t.dtl, rho.dtl, C.dtl, T.dtl,
                                            cp.dtl);
    const SideTerms<R> S = side_terms<R, -1>(n.r, t.r, rho.r, C.r, T.r, cp.r, n.dtr, t.dtr, rho.dtr, C.dtr, T.dtr,
                                             cp.dtr);

    // face column (e_n = 0): point 0 at the face value, points 2 (e_t = +1) and
    // 4 (e_t = -1) shifted by the mean t-step st = (dt_L + dt_R) / 8; there
    // q = e_t u_t + u_t^2 - u_n^2 / 2 and at point 0 q = -u^2 / 2.  hs, hd: half
    // sum and half difference of q at 2 and 4, times 64
    const R sn = n.dtl + n.dtr, st = t.dtl + t.dtr, sr = rho.dtl + rho.dtr, sc = C.dtl + C.dtr;
    const R a = n.f8 * n.f8, b = t.f8 * t.f8;
    const R hs = fma(R(-0.5), fma(sn, sn, a), fma(R(-8), st, fma(st, st, b)));
    const R hd = fma(n.f8, sn, fma(R(-2), st, R(8)) * t.f8);
    const R G0 = fma(rho.f8, hs - (a + b), -(sr * hd));   // 512 x (half the sum of rho q at 2 and 4, less rho u^2 of point 0)
    const R Gt = fma(rho.f8, hd, -(sr * hs));             // 512 x half the difference of rho q
    const R cc = fma(C.f8, st, sc * t.f8);                // -32 x the sum of C e.u at 2 and 4

    // Eq. 56 and the moments of the surrounding equilibria
    src.pm(p, muc);
    R lam8, mu8;
    src.lm(lam8, mu8);
    const R ps = p.l + p.r;
    const R mn = fma(R(3), p.l - p.r, L.X - S.X);                                                // 18 sum e_n f
    const R pf = fma(R(1.5), p.f8, fma(R(3), ps, fma(R(1.0 / 128.0), G0, L.X + S.X)));           // 18 p_f
    const R mt = fma(R(-0.75), p.dtl + p.dtr, fma(R(1.0 / 128.0), Gt, L.F + S.F));               // 18 sum e_t f
    const R Cf = fma(R(1.0 / 6.0), fma(R(-1.0 / 16.0), cc, fma(fc.y, fma(R(4), muc.l + muc.r, -muc.f8), L.G + S.G)),
                     R(0.125) * C.f8);                                                           // C_f
    const R gn = fma(fc.x, muc.l - muc.r, L.G - S.G);                                            // 6 sum e_n g
    const R ir = wdiv(R(1), rho.f8);
    const Moments<R> m{mn, mt, pf, Cf, gn, T.l - T.r, L.H - S.H, L.V + S.V, L.hd - S.hd, ps, R(2) * (p.dtr - p.dtl)};
    // tau - 1/2 from the face properties (R9): lambda / (rho C_ref cs^2 dt_s), mu / (rho cs^2 dt_s)
    FaceFlux<R> F = close_flux(K, m, fc.z, rho.f8, cp.f8 * T.f8, ir, fc.w * (lam8 * ir), R(6) * (mu8 * ir));
    if (AXI) F.Fmn = fma(R(-1.0 / 1152.0) * rho.f8, src.radial(n.f8, t.f8) * inv_r, F.Fmn);
    return F;
}

// The pieces of one face from the ring, in the working precision.
template <class R>
struct RingFace {
    const Ring<R>& P;
    const FaceIdx& x;
    bool normal_x, normal_is_r;
    __device__ __forceinline__ void vel(Rec<R>& n, Rec<R>& t) const {
        Rec<R> ru, rv;
        rec2(&P.uv[0][0], x, ru, rv);
        n = normal_x ? ru : rv;
        t = normal_x ? rv : ru;
    }
    __device__ __forceinline__ void rc(Rec<R>& a, Rec<R>& b) const { rec2(&P.rc[0][0], x, a, b); }
    __device__ __forceinline__ void tc(Rec<R>& a, Rec<R>& b) const { rec2(&P.tc[0][0], x, a, b); }
    __device__ __forceinline__ void pm(Rec<R>& a, Rec<R>& b) const { rec2(&P.pm[0][0], x, a, b); }
    __device__ __forceinline__ void lm(R& a, R& b) const { face_value8_2(&P.lm[0][0], x, a, b); }
    __device__ __forceinline__ R radial(R n0, R t0) const { return normal_is_r ? n0 : t0; }
};

template <class R, bool AXI>
__device__ __forceinline__ FaceFlux<R> face_flux(const Consts<R>& K, const Ring<R>& P, const FaceIdx& x, bool normal_x,
                                                 bool normal_is_r, R inv_r) {
    const RingFace<R> src{P, x, normal_x, normal_is_r};
    return face_math<R, AXI>(K, src, inv_r);
}


// ---------------------------------------------------------------------------
// General streaming steps (reading R26): h, f and g take their surrounding
// points at x_f - e_a dt_h, dt_f, dt_g.  A side point then lies inside its
// cell at distance a = 1/2 - dt from the centre along n and dt along t, so
// its value is f' -/+ (dt/2) d_t f with f' = f + a g_n (g_n the central
// n-slope of that cell); the face points move by -/+ (dt/4)(d_t f_L + d_t f_R).
// The linear parts keep their closed forms with f' for f and dt/12, dt/36 in
// the t-moments, and the side columns the terms of side_terms, each
// distribution's on its own points.  Used only when some step differs from
// 1/2; face_math above is this with a = 0, dt = 1/2.
// ---------------------------------------------------------------------------
// The pieces of one field: cell values, twice their n-slopes, eight times the
// face value, and the t-differences.
template <class R>
struct RecN { R l, r, gl, gr, f8, dtl, dtr; };

template <class R>
__device__ __forceinline__ RecN<R> recn_of(R l, R r, R ll, R rr, R lp, R lm, R rp, R rm) {
    return RecN<R>{l, r, r - ll, rr - l, face_value8(l, r, ll, rr), lp - lm, rp - rm};
}

template <class R>
__device__ __forceinline__ void recn2(const P2<R>* f, const FaceIdx& x, RecN<R>& a, RecN<R>& b) {
    const P2<R> l = f[x.L], r = f[x.R], ll = f[x.LL], rr = f[x.RR];
    const P2<R> lp = f[x.Lp], lm = f[x.Lm], rp = f[x.Rp], rm = f[x.Rm];
    a = recn_of(l.x, r.x, ll.x, rr.x, lp.x, lm.x, rp.x, rm.x);
    b = recn_of(l.y, r.y, ll.y, rr.y, lp.y, lm.y, rp.y, rm.y);
}

// One distribution's points: h = (1/2 - dt) / 2 of the normal offset (applied to
// twice the slopes), b = dt / 2 of the tangential one.
template <class R>
struct Points { R h, b; };
template <class R>
__device__ __forceinline__ Points<R> points_of(R dt) { return Points<R>{fma(R(-0.5), dt, R(0.25)), R(0.5) * dt}; }

// The value at the centre of a side column, and its t-points' offset.
template <class R, int SN>
__device__ __forceinline__ R centre(const RecN<R>& z, const Points<R>& p) {
    return SN > 0 ? fma(p.h, z.gl, z.l) : fma(-p.h, z.gr, z.r);
}
template <class R, int SN>
__device__ __forceinline__ R offset(const RecN<R>& z, const Points<R>& p) { return p.b * (SN > 0 ? z.dtl : z.dtr); }

// A, B, hq, hd and V of side_terms at one distribution's points.
template <class R, int SN>
struct Quad {
    R un, ut, sun, dn, dt, A, B;
    __device__ __forceinline__ Quad(const RecN<R>& Un, const RecN<R>& Ut, const Points<R>& p) {
        un = centre<R, SN>(Un, p);
        ut = centre<R, SN>(Ut, p);
        sun = SN > 0 ? un : -un;
        dn = offset<R, SN>(Un, p);
        dt = offset<R, SN>(Ut, p);
        A = sun - dt;
        B = SN > 0 ? ut - dn : ut + dn;
    }
    __device__ __forceinline__ R hq() const {
        const R x = fma(dn, ut, un * dt);
        return fma(B, B, fma(A, A, A)) - (SN > 0 ? x : -x);
    }
    __device__ __forceinline__ R hd() const {
        return fma(SN > 0 ? dn : -dn, dt, fma(sun, ut, fma(R(2), A, R(1)) * B));
    }
    __device__ __forceinline__ R V(R hq_) const { return fma(R(2), fma(un, un, fma(R(-0.5) * ut, ut, sun)), hq_); }
};

template <class R>
struct ColF { R X, V, hd, F; };

template <class R, int SN>
__device__ __forceinline__ ColF<R> col_f(const RecN<R>& Un, const RecN<R>& Ut, const RecN<R>& Rho, const Points<R>& p) {
    const Quad<R, SN> q(Un, Ut, p);
    const R rho = centre<R, SN>(Rho, p), dr = offset<R, SN>(Rho, p), hq = q.hq();
    ColF<R> s;
    s.hd = q.hd();
    s.V = q.V(hq);
    s.X = fma(rho, s.V, -(dr * s.hd));
    s.F = fma(rho, s.hd, -(dr * hq));
    return s;
}

template <class R, int SN>
__device__ __forceinline__ R col_g(const RecN<R>& Un, const RecN<R>& Ut, const RecN<R>& C, const Points<R>& p) {
    const Quad<R, SN> q(Un, Ut, p);
    return fma(centre<R, SN>(C, p), fma(R(2), q.sun, q.A), -(offset<R, SN>(C, p) * q.B));
}

template <class R, int SN>
__device__ __forceinline__ R col_h(const RecN<R>& Un, const RecN<R>& Ut, const RecN<R>& T, const RecN<R>& cp,
                                   const Points<R>& p) {
    const Quad<R, SN> q(Un, Ut, p);
    const R t = centre<R, SN>(T, p), c = centre<R, SN>(cp, p), dT = offset<R, SN>(T, p), dc = offset<R, SN>(cp, p);
    const R hq = q.hq();
    return fma(-fma(dc, t, c * dT), q.hd(), fma(dc * dT, hq, (c * t) * q.V(hq)));
}

template <class R, bool AXI>
__device__ __forceinline__ FaceFlux<R> face_flux_gen(const Consts<R>& K, const Ring<R>& P, const FaceIdx& x,
                                                     bool normal_x, bool normal_is_r, R inv_r) {
    const Points<R> pf_ = points_of(K.dtf), pg_ = points_of(K.dtg), ph_ = points_of(K.dth);
    RecN<R> Un, Ut;
    recn2(&P.uv[0][0], x, Un, Ut);
    if (!normal_x) { const RecN<R> t = Un; Un = Ut; Ut = t; }
    const R Sn = Un.dtl + Un.dtr, St = Ut.dtl + Ut.dtr;
    Moments<R> m;
    // h: points at dt_h (only e_n != 0 points carry C_p T q into the flux)
    RecN<R> T, cp;
    recn2(&P.tc[0][0], x, T, cp);
    m.hn = col_h<R, 1>(Un, Ut, T, cp, ph_) - col_h<R, -1>(Un, Ut, T, cp, ph_);
    m.dT = centre<R, 1>(T, ph_) - centre<R, -1>(T, ph_);
    RecN<R> Rho, Cc;
    recn2(&P.rc[0][0], x, Rho, Cc);
    const R rho8 = Rho.f8;
    // g: points at dt_g
    R cf;
    {
        const R L = col_g<R, 1>(Un, Ut, Cc, pg_), S = col_g<R, -1>(Un, Ut, Cc, pg_);
        const R w = R(4) * pg_.b;
        cf = fma(R(-1.0 / 16.0) * w, fma(Cc.f8, St, (Cc.dtl + Cc.dtr) * Ut.f8), L + S);
        m.gn = L - S;
    }
    // f: points at dt_f; the face column as in face_math, its steps 8 (dt/4)(dt_L + dt_R)
    {
        const ColF<R> L = col_f<R, 1>(Un, Ut, Rho, pf_), S = col_f<R, -1>(Un, Ut, Rho, pf_);
        const R w = R(4) * pf_.b;
        const R sn = w * Sn, st = w * St, sr = w * (Rho.dtl + Rho.dtr);
        const R a = Un.f8 * Un.f8, b = Ut.f8 * Ut.f8;
        const R hs = fma(R(-0.5), fma(sn, sn, a), fma(R(-8), st, fma(st, st, b)));
        const R hd = fma(Un.f8, sn, fma(R(-2), st, R(8)) * Ut.f8);
        const R G0 = fma(rho8, hs - (a + b), -(sr * hd)), Gt = fma(rho8, hd, -(sr * hs));
        m.mn = L.X - S.X;
        m.pf = fma(R(1.0 / 128.0), G0, L.X + S.X);
        m.mt = fma(R(1.0 / 128.0), Gt, L.F + S.F);
        m.V = L.V + S.V;
        m.hd = L.hd - S.hd;
    }
    RecN<R> p, mu;
    recn2(&P.pm[0][0], x, p, mu);
    R lam8, mu8;
    face_value8_2(&P.lm[0][0], x, lam8, mu8);
    const Q4<R> fc = ld4(K.facek);   // 3 Q, 3 Q / 4, C_ref / 6, 6 / C_ref
    const R pl = centre<R, 1>(p, pf_), pr = centre<R, -1>(p, pf_);
    const R ml = centre<R, 1>(mu, pg_), mr = centre<R, -1>(mu, pg_);
    m.ps = pl + pr;
    m.mn = fma(R(3), pl - pr, m.mn);
    m.pf = fma(R(1.5), p.f8, fma(R(3), m.ps, m.pf));
    m.mt = fma(R(-3) * pf_.b, p.dtl + p.dtr, m.mt);
    m.dp = (R(8) * pf_.b) * (p.dtr - p.dtl);
    m.Cf = fma(R(1.0 / 6.0), fma(fc.y, fma(R(4), ml + mr, -mu.f8), cf), R(0.125) * Cc.f8);
    m.gn = fma(fc.x, ml - mr, m.gn);
    const R ir = wdiv(R(1), rho8);
    FaceFlux<R> F = close_flux(K, m, fc.z, rho8, cp.f8 * T.f8, ir, K.th_coef * (lam8 * ir), K.tf_coef * (mu8 * ir));
    if (AXI) F.Fmn = fma(R(-1.0 / 576.0) * K.dtf * rho8, (normal_is_r ? Un.f8 : Ut.f8) * inv_r, F.Fmn);
    return F;
}

// Step 3, x-faces of ring row r: lane l computes the face between columns
// l+2 and l+3 (cells x0+l-1 and x0+l), at x = x0 + l.  In an axisymmetric
// domain the stored fluxes are multiplied by the face area r_f = x0 + l.
template <class R, bool AXI, bool GEN>
__device__ __forceinline__ void x_face(Core<R>& S, int x0, int r, int row_in_chunk, int lane, R inv_rf) {
    FaceIdx x;
    const int cL = lane + 2;
    x.L = slot(r) * RW + cL;
    x.R = x.L + 1;
    x.LL = x.L - 1;
    x.RR = x.L + 2;
    x.Lp = slot(r + 1) * RW + cL;
    x.Lm = slot(r - 1) * RW + cL;
    x.Rp = x.Lp + 1;
    x.Rm = x.Lm + 1;
    const R rf = AXI ? left_radius(S, lane + kHalo, x0 + lane) : R(1);
    FaceFlux<R> F = GEN ? face_flux_gen<R, AXI>(S.K, S.P, x, true, true, inv_rf)
                        : face_flux<R, AXI>(S.K, S.P, x, true, true, inv_rf);
    if (AXI) {
        F.Fh *= rf; F.Fp *= rf; F.Fmn *= rf; F.Fmt *= rf; F.Fc *= rf; F.un *= rf;
    }
    S.XF[0][row_in_chunk][lane] = P2<R>{F.Fh, F.Fp};
    S.XF[1][row_in_chunk][lane] = P2<R>{F.Fmn, F.Fmt};   // x-, y-momentum
    S.XF[2][row_in_chunk][lane] = P2<R>{F.Fc, F.un};
}

// Step 3, y-faces of face row r (between rows r-1 and r), lane l < 31 at
// column l+3 (cell x0 + l, radius x0 + l + 1/2 in an axisymmetric domain).
template <class R, bool AXI, bool GEN>
__device__ __forceinline__ void y_face(Core<R>& S, int r, int lane, R inv_r) {
    FaceIdx x;
    const int c = lane + kHalo;
    x.L = slot(r - 1) * RW + c;
    x.R = slot(r) * RW + c;
    x.LL = slot(r - 2) * RW + c;
    x.RR = slot(r + 1) * RW + c;
    x.Lp = x.L + 1;
    x.Lm = x.L - 1;
    x.Rp = x.R + 1;
    x.Rm = x.R - 1;
    const FaceFlux<R> F = GEN ? face_flux_gen<R, AXI>(S.K, S.P, x, false, false, inv_r)
                              : face_flux<R, AXI>(S.K, S.P, x, false, false, inv_r);
    const int s = slot(r);
    S.YF[0][s][lane] = P2<R>{F.Fh, F.Fp};
    S.YF[1][s][lane] = P2<R>{F.Fmt, F.Fmn};   // x-, y-momentum
    S.YF[2][s][lane] = P2<R>{F.Fc, F.un};
}

// The cell update's inputs besides the ring and the fluxes, straight from
// global memory: W^n, the stage's input W^s and F_s^{n-1} (stage 0) or
// dF_s/dt of the step.
template <class R>
struct GlobalCell {
    const Consts<R>& K;
    int stage;
    long long c;
    __device__ __forceinline__ R frac() const {
        return ld_l2(reinterpret_cast<const R*>(stage == 0 ? K.Fsp : K.dFs) + c);
    }
    __device__ __forceinline__ SV<R> wn() const { return load_state(reinterpret_cast<const R*>(K.st[0]), K.plane, c); }
    __device__ __forceinline__ SV<R> ws() const {
        return load_state(reinterpret_cast<const R*>(K.st[stage]), K.plane, c);
    }
};

// Step 4 for the cell (r, x0 + lane), plane index c.
template <class R, bool AXI, class Cell>
__device__ __forceinline__ void cell_update(Core<R>& S, const Cell& in, int stage, long long c, int r,
                                            int row_in_chunk, int lane, R irc, int* flag) {
    const Consts<R>& K = S.K;
    const int q = slot(r) * RW + lane + kHalo;
    const int qn = slot(r + 1) * RW + lane + kHalo, qs = slot(r - 1) * RW + lane + kHalo;
    const int sr = slot(r), sn = slot(r + 1);
    // Eq. 52; axisymmetric: the x-face fluxes carry their areas r_f, divided
    // here by the cell volume r_i = gx + 1/2 (per radian); irc = 1 / r_i
    R Rk[5], divu;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const P2<R> e = S.XF[k][row_in_chunk][lane + 1], w = S.XF[k][row_in_chunk][lane];
        const P2<R> n = S.YF[k][sn][lane], so = S.YF[k][sr][lane];
        const R dx0 = e.x - w.x, dx1 = e.y - w.y;
        const R d0 = -((AXI ? dx0 * irc : dx0) + (n.x - so.x));
        const R d1 = (AXI ? dx1 * irc : dx1) + (n.y - so.y);
        Rk[2 * k] = d0;
        if (k < 2) Rk[2 * k + 1] = -d1;
        else divu = d1;
    }
    const R divF1 = -Rk[1];   // div(rho cs^2 u), the pressure-flux divergence

    const Ring<R>& P = S.P;
    const P2<R> tc = (&P.tc[0][0])[q], rc = (&P.rc[0][0])[q], uv = (&P.uv[0][0])[q];
    const R T = tc.x, Cp = tc.y, rho = rc.x, C = rc.y, u = uv.x, v = uv.y;
    const R Fl = (&P.fl[0][0])[q];
    const P2<R>* RC = &P.rc[0][0];
    const P2<R>* PM = &P.pm[0][0];
    // twice the central slopes of rho and mu_c
    const R drx = RC[q + 1].x - RC[q - 1].x, dry = RC[qn].x - RC[qs].x;
    const R dmx = PM[q + 1].y - PM[q - 1].y, dmy = PM[qn].y - PM[qs].y;
    const Q4<R> cc = ld4(K.cellc);   // kv, g_x, g_y, 1 / dt
    R dfs;
    if (stage == 0) {   // reading R14: lagged dF_s/dt, fixed over the step
        const R Fs = R(1) - Fl;
        dfs = (Fs - in.frac()) * cc.w;
        reinterpret_cast<R*>(K.dFs)[c] = dfs;
        reinterpret_cast<R*>(K.Fsp)[c] = Fs;
    } else {
        dfs = in.frac();
    }
    const R cs2 = R(1.0 / 3.0);
    const R rD = rho * (solid_gate(K, C) * dfs);
    const R hFC = R(0.5) * (Fl * C);
    Rk[0] = fma(Cp * T, divu, Rk[0]);                                                       // Eq. 51 row 1
    Rk[1] = fma(R(1.0 / 6.0), fma(u, drx, v * dry), fma(cs2 * cc.x, rD, Rk[1]));            // row 2
    Rk[2] = fma(cs2, fma(rho, cc.y, -fma(hFC, dmx, u * rD)), Rk[2]);                        // row 3 (R13)
    Rk[3] = fma(cs2, fma(rho, cc.z, -fma(hFC, dmy, v * rD)), Rk[3]);                        // row 4
    Rk[4] = fma(C * cc.x, dfs, Rk[4]);                                                      // row 5 (R12: Eq. 40 / 47)
    const Q4<R> c2 = ld4(K.cellc2);   // dt, dt_f in z, w
    if (AXI)   // hoop stress Pi_thetatheta / r with the pressure advanced over dt_s (reading R24)
        Rk[2] = fma(cs2 * irc, fma(R(-2) * irc, (&P.lm[0][0])[q].y * u, fma(-c2.w, divF1, PM[q].x)), Rk[2]);

    // stage 0 reads W^n as its input: one load serves both
    const SV<R> wn = in.wn();
    const SV<R> ws = stage == 0 ? wn : in.ws();
    SV<R> o;
    if constexpr (sizeof(R) == 8) {
        // Eq. 58 as written (stage 0 without its products by 1 and 0); explicit
        // FMAs, so that both kernels round alike
        if (stage == 0) {
            o.Hh = fma(c2.z, Rk[0], wn.Hh);
            o.p = fma(c2.z, Rk[1], wn.p);
            o.mx = fma(c2.z, Rk[2], wn.mx);
            o.my = fma(c2.z, Rk[3], wn.my);
            o.Ch = fma(c2.z, Rk[4], wn.Ch);
        } else {
            const R A = stage == 1 ? R(0.75) : R(1.0 / 3.0);
            const R B = stage == 1 ? R(0.25) : R(2.0 / 3.0);
            const R Cd = B * c2.z;
            o.Hh = fma(Cd, Rk[0], fma(A, wn.Hh, B * ws.Hh));
            o.p = fma(Cd, Rk[1], fma(A, wn.p, B * ws.p));
            o.mx = fma(Cd, Rk[2], fma(A, wn.mx, B * ws.mx));
            o.my = fma(Cd, Rk[3], fma(A, wn.my, B * ws.my));
            o.Ch = fma(Cd, Rk[4], fma(A, wn.Ch, B * ws.Ch));
        }
        o.Hl = R(0);
        o.Cl = R(0);
    } else {
        // Eq. 58 as W^n + increment (stage 0: dt R alone, 14 operations fewer; us per
        // step of 64 domains (7.23 M cells) 1006 -> 994, 512^2 53.2 -> 52.7); H and C kept as
        // compensated pairs.  TwoSum for the sum and the renormalisation keeps
        // every pair canonical.
        R dH, dC;
        if (stage == 0) {
            dH = mul_rn(c2.z, Rk[0]);
            dC = mul_rn(c2.z, Rk[4]);
            o.p = fma(c2.z, Rk[1], wn.p);
            o.mx = fma(c2.z, Rk[2], wn.mx);
            o.my = fma(c2.z, Rk[3], wn.my);
        } else {
            const R B = stage == 1 ? R(0.25) : R(2.0 / 3.0);
            const R Cd = B * c2.z;
            dH = fma(Cd, Rk[0], B * ((ws.Hh - wn.Hh) + (ws.Hl - wn.Hl)));
            dC = fma(Cd, Rk[4], B * ((ws.Ch - wn.Ch) + (ws.Cl - wn.Cl)));
            o.p = wn.p + fma(Cd, Rk[1], B * (ws.p - wn.p));
            o.mx = wn.mx + fma(Cd, Rk[2], B * (ws.mx - wn.mx));
            o.my = wn.my + fma(Cd, Rk[3], B * (ws.my - wn.my));
        }
        R s1, e1;
        two_sum(wn.Hh, dH, s1, e1);
        two_sum(s1, wn.Hl + e1, o.Hh, o.Hl);
        two_sum(wn.Ch, dC, s1, e1);
        two_sum(s1, wn.Cl + e1, o.Ch, o.Cl);
    }
    if (K.zsv) {   // reading R15: no motion of the solid part
        R Tn, Fln;
        const R Cn = pair_sum(o.Ch, o.Cl);
        invert_enthalpy(K, o.Hh, o.Hl, clamp01(Cn), Tn, Fln);
        const R keep = R(1) - solid_gate(K, Cn) * (R(1) - Fln);
        o.mx *= keep;
        o.my *= keep;
    }
    if (!(is_finite(o.Hh) && is_finite(o.p) && is_finite(o.mx) && is_finite(o.my) && is_finite(o.Ch))) {
        atomicOr(flag, 1);      // solver-wide
        atomicOr(K.flag, 1);    // this domain
    }
    store_state(reinterpret_cast<R*>(K.st[stage == 2 ? 0 : stage + 1]), K.plane, c, o);
}

}  // namespace

}  // namespace eulbfs
