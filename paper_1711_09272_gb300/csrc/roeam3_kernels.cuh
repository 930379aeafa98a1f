// roeam3_kernels.cuh — the 3D Roe-AM path: Cartesian grids, first-order faces, up to three
// passive scalars (the complete form of Eq. 85, the 9-face detector of Eq. 96), fused with the
// residual and the SSP-RK3 stage update like the 2D kernels.
//
// Decomposition: a CTA takes a rectangle of cells of the (x, y) plane with one halo position around it
// and marches along z over a segment of planes (see stage3_march for FP32, stage3_phases for FP64).
#pragma once

#include <algorithm>

#include "roeam_kernels.cuh"
#include "roeam3_internal.h"

namespace roeam {

// Primitive and derived values of one cell: c2 = gamma p / rho, H total enthalpy,
// sr = sqrt(rho), Mq = |q| / c, scalars k.
template <typename T, int NS> struct C3 {
    T r, u, v, w, p, c2, H, sr, Mq;
    T k[NS > 0 ? NS : 1];
};

template <typename T, int NS>
__device__ __forceinline__ void derive3(C3<T, NS> &c, T ri, const GridCoef3<T> &K)   // ri = 1 / rho
{
    c.c2 = K.g * c.p * ri;
    const T q2 = c.u * c.u + c.v * c.v + c.w * c.w;
    c.H = vfma(c.c2, K.gm1i, T(0.5) * q2);
    c.sr = sqrt1(c.r);
    c.Mq = sqrt0(q2 * rcp(c.c2));
}

// One side of a face in the face frame: normal velocity un, tangential ut, uw. V is the
// working precision, or V2 for two faces evaluated together in packed FP32.
template <typename V, int NS> struct FS3 {
    V r, un, ut, uw, p, c2, H, sr, Mq;
    V k[NS > 0 ? NS : 1];
};

template <typename T, int NS>
__device__ __forceinline__ FS3<T, NS> side3(const C3<T, NS> &c, int axis)
{
    FS3<T, NS> s;
    s.r = c.r; s.p = c.p; s.c2 = c.c2; s.H = c.H; s.sr = c.sr; s.Mq = c.Mq;
    if (axis == 0) { s.un = c.u; s.ut = c.v; s.uw = c.w; }
    else if (axis == 1) { s.un = c.v; s.ut = c.u; s.uw = c.w; }
    else { s.un = c.w; s.ut = c.u; s.uw = c.v; }
#pragma unroll
    for (int q = 0; q < NS; ++q) s.k[q] = c.k[q];
    return s;
}

// The sides of an x-face (component x) and a y-face (component y) packed together.
template <int NS>
__device__ __forceinline__ FS3<V2, NS> side3_xy(const C3<float, NS> &cx, const C3<float, NS> &cy)
{
    FS3<V2, NS> s;
    s.r = mk2(cx.r, cy.r); s.p = mk2(cx.p, cy.p); s.c2 = mk2(cx.c2, cy.c2); s.H = mk2(cx.H, cy.H);
    s.sr = mk2(cx.sr, cy.sr); s.Mq = mk2(cx.Mq, cy.Mq);
    s.un = mk2(cx.u, cy.v); s.ut = mk2(cx.v, cy.u); s.uw = mk2(cx.w, cy.w);
#pragma unroll
    for (int q = 0; q < NS; ++q) s.k[q] = mk2(cx.k[q], cy.k[q]);
    return s;
}

// Twice the Roe-AM flux per unit area in the face frame (mass, normal momentum, the two
// tangential momenta, energy, scalars): Section 6.2 term by term as in roeam_flux2, with the
// w rows and Eq. 85's scalar rows; the rotated-Riemann estimate of Eqs. 103-109 in 3D
// (n2 the unit part of n perpendicular to n1, so |a2 U2| = |U - a1 U1|).
template <typename V, typename S, int NS>
__device__ __forceinline__ void roeam_flux3(const FS3<V, NS> &L, const FS3<V, NS> &R, V s1, const GridCoef3<S> &K,
                                            int eps1, int xi_form, V F[5 + NS])
{
    const V zero = splat<V>(0), one = splat<V>(1), half = splat<V>(S(0.5));

    const V w = rcp(L.sr + R.sr);
    const V wl = L.sr * w, wr = R.sr * w;
    const V rh = L.sr * R.sr;
    const V Hh = vfma(wl, L.H, wr * R.H);
    const V du = R.un - L.un, dv = R.ut - L.ut, dw = R.uw - L.uw;
    const V uh = vfma(wr, du, L.un), vh = vfma(wr, dv, L.ut), wh = vfma(wr, dw, L.uw);   // (wl + wr = 1)
    const V dq2 = vfma(du, du, vfma(dv, dv, dw * dw));
    const V c2h = vfma(splat<V>(K.hgm1) * wl * wr, dq2, vfma(wl, L.c2, wr * R.c2));
    const V chi = rsq(c2h);
    const V ch = c2h * chi;
    const V aU = vabs(uh);

    const V M = half * (L.Mq + R.Mq);
    const V Mb = aU * chi;
    const V fM = fmach(M), fMb = fmach(Mb);
    const V fM8 = pow8(fM), fMb8 = pow8(fMb);
    const V dp = R.p - L.p;

    const V br = bracket4(aU, ch);
    const V Up = vmx(vfma(fMb * br, vmx(du, zero), aU), zero);   // du <= 0 leaves |U|

    const V xfh = xi_form ? half : vfma(splat<V>(S(-0.5)), fMb8, half);   // [1 - f^8(Mbar)] / 2
    V xi = vmx(vfma(xfh, du, vabs(vfma(half, du, L.un))), zero);
    if (eps1) {
        const V dq = sqrt0(dq2);
        const auto big = ge(dq, splat<V>(K.rr_thr));
        const V dqi = rcp(sel(big, dq, one));
        const V n1x = sel(big, du * dqi, one);
        const V U1 = sel(big, vfma(du, uh, vfma(dv, vh, dw * wh)) * dqi, uh);
        const V frr = vabs(n1x * U1) + vabs(vfma(-n1x, U1, uh));
        xi = vmx(xi, (one - fMb8) * fM8 * vmn(splat<V>(K.eps2) * ch, frr));
    }

    const V mn = vmn(Up, ch);
    const V smc = vcopysign(mn, uh) * chi;
    const V pp = vfma(smc, dp, vfma(s1, fM, one - s1) * vmx(ch - Up, zero) * rh * du);
    const V th = vmn(vmx(splat<V>(K.mr2), M * M), one);
    const V om = one - th;
    const V nh = vnabs(half * om * uh);   // (as in roeam_flux2)
    const V Z = c2h * th;
    const V X = vfma(nh, nh, Z);
    const V rX = rsq(X);
    const V ct = X * rX;
    const V term = vfma(nh, rX * vmn(aU + nh, ct), vfma(om, Up, vmx(ct - Up, zero)));
    const V nA = s1 * (fM8 - one) * term * dp * rcp(Z);   // -rho delta U_p
    const V ns = splat<V>(S(-0.5)) * smc;   // (-delta U_u = ns du)

    // Eq. 85 per side (as in roeam_flux2): rho_side (U_side +- xi - dUu) times the side's
    // (1, U, V, W, H, k), plus the pressure and delta U_p terms.
    const V gL = L.r * (L.un + vfma(ns, du, xi)), gR = R.r * vfma(ns, du, R.un - xi);
    F[0] = (gL + gR) + nA;
    F[1] = vfma(gL, L.un, vfma(gR, R.un, vfma(nA, uh, L.p + R.p) - pp));
    F[2] = vfma(gL, L.ut, vfma(gR, R.ut, nA * vh));
    F[3] = vfma(gL, L.uw, vfma(gR, R.uw, nA * wh));
    F[4] = vfma(gL, L.H, vfma(gR, R.H, nA * Hh));
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        const V kh = vfma(wl, L.k[s], wr * R.k[s]);
        F[5 + s] = vfma(gL, L.k[s], vfma(gR, R.k[s], nA * kh));
    }
}

template <typename T> __device__ __forceinline__ T min9(T a, T b, T c, T d, T e, T f, T g, T h, T i)
{
    return fmn3(fmn3(a, b, c), fmn3(d, e, f), fmn3(g, h, i));   // (positive ratios, never NaN)
}

// Velocity, |q|^2 and pressure of a conserved 3D state, with explicit rounding (the stage
// epilogue's positivity check and the time-step rate share them).
template <typename T> struct Prims3 { T ri, u, v, w, q2, p; };
template <typename T>
__device__ __forceinline__ Prims3<T> cell_prims3(T r, T ru, T rv, T rw, T rE, const GridCoef3<T> &K)
{
    Prims3<T> s;
    s.ri = rcp(r);
    s.u = rmul(ru, s.ri); s.v = rmul(rv, s.ri); s.w = rmul(rw, s.ri);
    s.q2 = radd(radd(rmul(s.u, s.u), rmul(s.v, s.v)), rmul(s.w, s.w));
    s.p = rmul(K.gm1, rsub(rE, rmul(rmul(T(0.5), r), s.q2)));
    return s;
}

// Time-step rate of one 3D cell (the 2D rule with three directions; theta shared).
template <typename T>
__device__ __forceinline__ T cell_rate3(const Prims3<T> &s, const GridCoef3<T> &K)
{
    const T c2 = rmul(rmul(K.g, s.p), s.ri);
    const T c = sqrt0(c2);
    const T th = vmin(vmax(K.mr2, rmul(s.q2, rcp(c2))), T(1));
    T wx = c, wy = c, wz = c;
    if (th < T(1)) {
        const T om = rsub(T(1), th), ith = rcp(th);
        const T a = rmul(rmul(T(4), c2), th), o2 = rmul(om, om);
        wx = vmax(c, rmul(rmul(T(0.5), sqrt0(radd(a, rmul(o2, rmul(s.u, s.u))))), ith));
        wy = vmax(c, rmul(rmul(T(0.5), sqrt0(radd(a, rmul(o2, rmul(s.v, s.v))))), ith));
        wz = vmax(c, rmul(rmul(T(0.5), sqrt0(radd(a, rmul(o2, rmul(s.w, s.w))))), ith));
    }
    return radd(radd(rmul(radd(vabs(s.u), wx), K.idx), rmul(radd(vabs(s.v), wy), K.idy)),
                rmul(radd(vabs(s.w), wz), K.idz));
}

// After a stage: non-positive or non-finite states raise the status; with `rate` the cell's time-step
// rate raises m.
template <typename T, int NV>
__device__ __forceinline__ void check_cell3(const T (&out)[NV], bool rate, const GridCoef3<T> &K, unsigned *status, T &m)
{
    // p > 0 without the division: 2 rho (rho E) > |rho q|^2; a cell that fails it (rare: also products
    // beyond the FP32 range) is decided by its pressure
    const T e2 = T(2) * out[0] * out[4];
    const T m2 = out[1] * out[1] + out[2] * out[2] + out[3] * out[3];
    if (rate || !(out[0] > T(0)) || !(e2 > m2)) {
        const Prims3<T> cp = cell_prims3(out[0], out[1], out[2], out[3], out[4], K);
        if (!(out[0] > T(0)) || !(cp.p > T(0))) {
            const bool fin = isfinite((double)out[0]) && isfinite((double)cp.p);
            atomicOr(status, fin ? ST_NONPOSITIVE : ST_NONFINITE);
        } else if (rate) {
            m = vmax(m, cell_rate3(cp, K));
        }
    }
}

// A cell's values in memory: four together, then the rest (tail3<NV>() values: the fifth variable and
// the scalars), as quads and tails of the state buffers and of shared memory.
template <int N, typename T> __device__ __forceinline__ void ld_tail(const T *p, T q[N])
{
    if constexpr (N == 1) q[0] = p[0];
    else if constexpr (N == 2 && sizeof(T) == 4) { const float2 v = *reinterpret_cast<const float2 *>(p); q[0] = v.x; q[1] = v.y; }
    else if constexpr (N == 2) { const double2 v = *reinterpret_cast<const double2 *>(p); q[0] = v.x; q[1] = v.y; }
    else ld_own(p, q);
}
template <int N, typename T> __device__ __forceinline__ void st_tail(T *p, const T q[N])
{
    if constexpr (N == 1) p[0] = q[0];
    else if constexpr (N == 2 && sizeof(T) == 4) *reinterpret_cast<float2 *>(p) = make_float2(q[0], q[1]);
    else if constexpr (N == 2) *reinterpret_cast<double2 *>(p) = make_double2(q[0], q[1]);
    else st_cell(p, q);
}
template <int N, typename T> __device__ __forceinline__ void copy_tail(unsigned dst, const T *src)
{
    constexpr int B = N * (int)sizeof(T);
    if constexpr (B >= 16) {
        cp16(dst, src);
        if constexpr (B == 32) cp16(dst + 16, src + 2);
    } else {
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(B) : "memory");
    }
}

// FP64: bound by the FP64 pipe, so every face is evaluated once per CTA and no lane idles while another
// evaluates one. Raw planes k - 1 to k + 2 in shared memory (asynchronous copies run ahead), primitives
// and derived quantities of planes k and k + 1, their Eq. 97 ratios, the fluxes of plane k; per plane
// three phases, a block barrier after each: update of plane k - 1 and primitives of plane k + 1 (each
// thread its own positions), ratios of plane k + 1, fluxes through the west and south faces of plane k
// and the face above it, one list for all threads. 720 FP64 operations per cell where the marching
// layout of FP32 took 1700 (8-row tiles, halo rows, segments of 4 planes): 64^3 with two scalars
// 3306 -> 1252 us a step, 128^3 16.9 -> 9.3 ms.
template <typename T, int NS> __device__ __forceinline__ void stage3_phases(const StageArgs3<T> &a)
{
    // Everything of one position lies in one record of shared memory, so that a thread addresses a cell
    // and its neighbours by one base and constants (in separate arrays per quantity the address
    // arithmetic was a third of the instructions). Words of a record: raw quads of planes k & 3, U^n, west
    // and south flux, z-flux (slot k & 1: the face below plane k), primitives r u v w and p c2 H sr
    // (slot k & 1), then the tails of the same (Mq and the scalars for the primitives) and the Eq. 97
    // ratios of the west, south and lower face (slot k & 1).
    constexpr int NV = 5 + NS, TW = tail3(NV), REC = rec3(NV);
    constexpr int oQ = 0, oN = 16, oF = 24, oZ = 32, oW = 40, oE = 48, oQT = 56, oNT = oQT + 4 * TW, oFT = oNT + 2 * TW,
                  oZT = oFT + 2 * TW, oX = oZT + 2 * TW, oP = oX + 2 * TW;
    constexpr int MP = 2;   // positions per thread
    pdl_trigger();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ T red[threads3<T>() / 32];

    const int4 unit = __ldg(a.units + blockIdx.x);
    const int g = a.ngrids == 1 ? 0 : unit.x;
    const int x0 = unit.y & 0xffff, w = unit.y >> 16, y0 = unit.z & 0xffff, h = unit.z >> 16;
    const int k0 = unit.w & 0xffff, k1 = (int)((unsigned)unit.w >> 16);
    const GridDev3 &G = a.grids[g];
    const GridCoef3<T> K = a.coef[g];
    const int ni = G.ni, nj = G.nj, nk = G.nk, pitch = G.pitch;
    const int bcB = G.bc[4], bcT = G.bc[5];
    const int eps1 = G.eps1, xi_form = G.xi_form;
    const bool use_s1 = G.use_s1 != 0;
    const int W = w + 2, NP = W * (h + 2);   // positions: (c, r) is cell (x0 - 1 + c, y0 - 1 + r)
    const int tid = threadIdx.x, nt = blockDim.x;
    T *const S = reinterpret_cast<T *>(smem_raw);
    const int WR = W * REC;                  // from a record to the one in the next row

    // this thread's positions: source column in the plane, kinds (bit 0 x wall, 1 y wall, 2 inflow, 3 own cell)
    int xy[MP], kind[MP];
    const unsigned mW = 0xffffffffu / (unsigned)W + 1u;
#pragma unroll
    for (int m = 0; m < MP; ++m) {
        const int q = tid + m * nt, r = (int)__umulhi((unsigned)q, mW), c = q - r * W;
        int kx, ky;
        const int is = resolve_index(x0 - 1 + c, ni, G.bc[0], G.bc[1], kx), js = resolve_index(y0 - 1 + r, nj, G.bc[2], G.bc[3], ky);
        xy[m] = js * pitch + is;
        kind[m] = (kx == 1) | (ky == 1) << 1 | (kx == 2 || ky == 2) << 2 | (c >= 1 && c <= w && r >= 1 && r <= h) << 3;
        if (q >= NP) kind[m] = -1;
    }
    const bool stage_mode = a.mode == MODE_STAGE;
    const bool combine = stage_mode && a.alpha != T(0);
    const T hx = T(0.5) * K.idx, hy = T(0.5) * K.idy, hz = T(0.5) * K.idz;
    const long long row = (long long)nj * pitch;   // cells per plane
    const T *const src = a.src + G.off, *const un = a.un + G.off;
    T *const dst = a.dst + G.off;
    const long long tails = 4 * G.vol;             // the grid's tails follow its quads
    const unsigned sm = (unsigned)__cvta_generic_to_shared(S) + (unsigned)(tid * REC * (int)sizeof(T));
    const unsigned sm_step = (unsigned)(nt * REC * (int)sizeof(T));
    pdl_wait();
    if (a.rate_zero && blockIdx.x == 0)
        for (int q = tid; q < a.ngrids; q += nt) a.rate_zero[q] = 0ull;
    T dt = T(0);
    if (stage_mode) dt = a.dt_fixed_t > T(0) ? a.dt_fixed_t : a.cfl_t / rate_at<T>(a.rate_rd + g);

    // starts the copies of plane k (to k1 at most) and, in the same group, of U^n of plane k - 2
    auto issue = [&](int k) {
        int kz;
        const long long base = (long long)resolve_index(k, nk, bcB, bcT, kz) * row;
        const int slot = k & 3, m2 = k - 2;
        const bool plane = k <= k1, combined = combine && m2 >= k0 && m2 < k1;
#pragma unroll
        for (int m = 0; m < MP; ++m) {
            if (kind[m] < 0) continue;
            const unsigned rec = sm + m * sm_step;
            if (plane) {
                const long long c = base + xy[m];
                copy_cell(rec + (unsigned)((oQ + 4 * slot) * (int)sizeof(T)), src + 4 * c);
                copy_tail<TW>(rec + (unsigned)((oQT + TW * slot) * (int)sizeof(T)), src + tails + TW * c);
            }
            if (combined && (kind[m] & 8)) {
                const long long o = (long long)m2 * row + xy[m];
                copy_cell(rec + (unsigned)((oN + 4 * (m2 & 1)) * (int)sizeof(T)), un + 4 * o);
                copy_tail<TW>(rec + (unsigned)((oNT + TW * (m2 & 1)) * (int)sizeof(T)), un + tails + TW * o);
            }
        }
        copies_commit();
    };
    // primitives of this thread's positions of plane k
    auto prims = [&](int k) {
        int kz;
        resolve_index(k, nk, bcB, bcT, kz);
        const int s4 = k & 3, s2 = k & 1;
#pragma unroll 1
        for (int m = 0; m < MP; ++m) {
            const int kd = m == 0 ? kind[0] : kind[1];
            if (kd < 0) continue;
            T *const rec = S + (tid + m * nt) * REC;
            C3<T, NS> c;
            T v[4], t[TW];
            ld_own(rec + oQ + 4 * s4, v);
            ld_tail<TW>(rec + oQT + TW * s4, t);
            T ri = rcp(v[0]);
            c.r = v[0];
            c.u = v[1] * ri; c.v = v[2] * ri; c.w = v[3] * ri;
            c.p = K.gm1 * (t[0] - T(0.5) * c.r * (c.u * c.u + c.v * c.v + c.w * c.w));
#pragma unroll
            for (int s = 0; s < NS; ++s) c.k[s] = t[1 + s] * ri;
            if (kd & 1) c.u = -c.u;
            if (kd & 2) c.v = -c.v;
            if (kz == 1) c.w = -c.w;
            if ((kd & 4) || kz == 2) {
                c.r = K.inflow[0]; c.u = K.inflow[1]; c.v = K.inflow[2]; c.w = K.inflow[3]; c.p = K.inflow[4];
#pragma unroll
                for (int s = 0; s < NS; ++s) c.k[s] = K.inflow[5 + s];
                ri = rcp(c.r);
            }
            derive3(c, ri, K);
            const T a0[4] = {c.r, c.u, c.v, c.w}, a1[4] = {c.p, c.c2, c.H, c.sr};
            T a2[4] = {c.Mq, T(0), T(0), T(0)};
#pragma unroll
            for (int s = 0; s < NS; ++s) a2[1 + s] = c.k[s];
            st_cell(rec + oW + 4 * s2, a0);
            st_cell(rec + oE + 4 * s2, a1);
            st_tail<TW>(rec + oX + TW * s2, a2);
        }
    };
    auto cell = [&](int s2, const T *rec, C3<T, NS> &c) {
        T v[4], t[TW];
        ld_own(rec + oW + 4 * s2, v);
        c.r = v[0]; c.u = v[1]; c.v = v[2]; c.w = v[3];
        ld_own(rec + oE + 4 * s2, v);
        c.p = v[0]; c.c2 = v[1]; c.H = v[2]; c.sr = v[3];
        ld_tail<TW>(rec + oX + TW * s2, t);
        c.Mq = t[0];
#pragma unroll
        for (int s = 0; s < NS; ++s) c.k[s] = t[1 + s];
    };
    // ratios of plane k; `below`: also those of the faces towards plane k - 1. (Those of the outermost
    // positions towards the outside are not used.)
    auto ratios = [&](int k, bool below) {
        const int s2 = k & 1, o = 3 * s2;
        for (int q = tid; q < NP; q += nt) {
            T *const rec = S + q * REC;
            const T *rw = S + max(q - 1, 0) * REC, *rs = S + max(q - W, 0) * REC;
            const T r = rec[oW + 4 * s2], p = rec[oE + 4 * s2];
            rec[oP + o] = ratio_P(rw[oW + 4 * s2], rw[oE + 4 * s2], r, p);
            rec[oP + o + 1] = ratio_P(rs[oW + 4 * s2], rs[oE + 4 * s2], r, p);
            if (below) rec[oP + o + 2] = ratio_P(rec[oW + 4 * (s2 ^ 1)], rec[oE + 4 * (s2 ^ 1)], r, p);
        }
    };
    // Eq. 96 in 3D: the face and the eight transverse faces of its two cells.
    auto min_x = [&](int s2, const T *rec, const T *north) {
        const int o = oP + 3 * s2, z = oP + 3 * (s2 ^ 1) + 2;
        return min9(rec[o], rec[o + 1 - REC], north[o + 1 - REC], rec[o + 1], north[o + 1], rec[o + 2 - REC], rec[z - REC],
                    rec[o + 2], rec[z]);
    };
    auto min_y = [&](int s2, const T *rec, const T *south) {
        const int o = oP + 3 * s2, z = oP + 3 * (s2 ^ 1) + 2;
        return min9(rec[o + 1], south[o], south[o + REC], rec[o], rec[o + REC], south[o + 2], south[z], rec[o + 2], rec[z]);
    };
    auto min_z = [&](int s2, const T *rec, const T *north) {   // the face below the plane of slot s2
        const int o = oP + 3 * s2, b = oP + 3 * (s2 ^ 1);
        return min9(rec[o + 2], rec[b], rec[b + REC], rec[b + 1], north[b + 1], rec[o], rec[o + REC], rec[o + 1], north[o + 1]);
    };
    // NV values as a quad and a tail
    auto put = [&](T *F4, T *FT, const T F[NV]) {
        st_cell(F4, F);
        T t[TW];
#pragma unroll
        for (int s = 0; s < TW; ++s) t[s] = s < NV - 4 ? F[4 + (s < NV - 4 ? s : 0)] : T(0);
        st_tail<TW>(FT, t);
    };
    auto get = [&](const T *F4, const T *FT, T v[NV]) {
        T t[TW];
        ld_own(F4, v);
        ld_tail<TW>(FT, t);
#pragma unroll
        for (int s = 4; s < NV; ++s) v[s] = t[s - 4];
    };
    const unsigned mw1 = 0xffffffffu / (unsigned)(w + 1) + 1u, mw = 0xffffffffu / (unsigned)w + 1u;
    auto div = [](int q, unsigned m, int n) { return n == 1 ? q : (int)__umulhi((unsigned)q, m); };

    issue(k0 - 1);
    issue(k0);
    issue(k0 + 1);
    copies_wait<2>();
    prims(k0 - 1);
    __syncthreads();
    ratios(k0 - 1, false);

    T my_rate = T(0);
#pragma unroll 1
    for (int k = k0 - 1; k <= k1; ++k) {
        const int sk = k & 1, sn = sk ^ 1;   // slots of planes k and k + 1
        copies_wait<1>();
        // ---- update plane k - 1: R = hx (F_w - F_e) + hy (F_s - F_n) + hz (F_b - F_t) of the doubled fluxes
        if (k > k0) {
#pragma unroll 1
            for (int m = 0; m < MP; ++m) {
                const int kd = m == 0 ? kind[0] : kind[1];
                if (kd < 0 || !(kd & 8)) continue;
                const T *const rec = S + (tid + m * nt) * REC;
                T R[NV], uk[NV], out[NV], fa[NV], fb[NV];
                get(rec + oZ + 4 * sn, rec + oZT + TW * sn, fa);   // (below plane k - 1, below plane k)
                get(rec + oZ + 4 * sk, rec + oZT + TW * sk, fb);
#pragma unroll
                for (int v = 0; v < NV; ++v) R[v] = hz * (fa[v] - fb[v]);
                get(rec + oF + 4, rec + oFT + TW, fa);
                get(rec + WR + oF + 4, rec + WR + oFT + TW, fb);
#pragma unroll
                for (int v = 0; v < NV; ++v) R[v] = vfma(hy, fa[v] - fb[v], R[v]);
                get(rec + oF, rec + oFT, fa);
                get(rec + REC + oF, rec + REC + oFT, fb);
#pragma unroll
                for (int v = 0; v < NV; ++v) R[v] = vfma(hx, fa[v] - fb[v], R[v]);
                const long long o = (long long)(k - 1) * row + (m == 0 ? xy[0] : xy[1]);
                if (stage_mode) {
                    const int q4 = (k - 1) & 3, n2 = (k - 1) & 1;
                    get(rec + oQ + 4 * q4, rec + oQT + TW * q4, uk);
                    if (combine) get(rec + oN + 4 * n2, rec + oNT + TW * n2, fa);
                    else
#pragma unroll
                        for (int v = 0; v < NV; ++v) fa[v] = uk[v];
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        const T upd = vfma(dt, R[v], uk[v]);
                        out[v] = combine ? vfma(a.alpha, fa[v], a.beta * upd) : upd;
                    }
                } else {
#pragma unroll
                    for (int v = 0; v < NV; ++v) out[v] = R[v];
                }
                put(dst + 4 * o, dst + tails + TW * o, out);   // (the state has the same layout)
                if (stage_mode) check_cell3(out, a.want_rate != 0, K, a.status, my_rate);
            }
        }
        if (k == k1) break;
        // ---- primitives of plane k + 1 (into the slot of plane k - 1, whose last reader was two barriers ago),
        //      and the copies of plane k + 3 into the raw slot that the update has just read
        prims(k + 1);
        issue(k + 3);
        __syncthreads();
        ratios(k + 1, true);
        __syncthreads();
        // ---- fluxes: west and south faces of plane k (k >= k0), the face between planes k and k + 1
        const bool xyf = k >= k0;
        const int nz = w * h;
        {
            // one list of single faces: z, then west, then south
            const int nx = (w + 1) * h, all = nz + (xyf ? nx + w * (h + 1) : 0);
#pragma unroll 1
            for (int f = tid; f < all; f += nt) {
                const int axis = f < nz ? 2 : (f < nz + nx ? 0 : 1);
                const int i = axis == 2 ? f : (axis == 0 ? f - nz : f - nz - nx), wd = axis == 0 ? w + 1 : w;
                const int r = div(i, axis == 0 ? mw1 : mw, wd), q = (r + 1) * W + 1 + i - r * wd;
                C3<T, NS> A, B;
                T *const rec = S + q * REC;
                cell(sk, axis == 2 ? rec : rec - (axis == 0 ? REC : WR), A);
                cell(axis == 2 ? sn : sk, rec, B);
                const T s1 = use_s1 ? detector_of(axis == 2 ? min_z(sn, rec, rec + WR)
                                                            : (axis == 0 ? min_x(sk, rec, rec + WR) : min_y(sk, rec, rec - WR)))
                                    : T(1);
                auto face_side = [&](const C3<T, NS> &c) {
                    FS3<T, NS> s = side3(c, 0);
                    s.un = axis == 0 ? c.u : (axis == 1 ? c.v : c.w);
                    s.ut = axis == 0 ? c.v : c.u;
                    s.uw = axis == 2 ? c.v : c.w;
                    return s;
                };
                T G2[NV], F[NV];
                roeam_flux3<T, T, NS>(face_side(A), face_side(B), s1, K, eps1, xi_form, G2);
#pragma unroll
                for (int v = 0; v < NV; ++v) F[v] = G2[v];
                F[1] = axis == 0 ? G2[1] : G2[2];
                F[2] = axis == 0 ? G2[2] : (axis == 1 ? G2[1] : G2[3]);
                F[3] = axis == 2 ? G2[1] : G2[3];
                const int o4 = axis == 2 ? oZ + 4 * sn : (axis == 0 ? oF : oF + 4);
                const int ot = axis == 2 ? oZT + TW * sn : (axis == 0 ? oFT : oFT + TW);
                put(rec + o4, rec + ot, F);
            }
        }
        __syncthreads();
    }
    if (a.want_rate) {
        my_rate = warp_rate_max(my_rate);
        if ((tid & 31) == 0) red[tid >> 5] = my_rate;
        __syncthreads();
        if (tid < 32) {
            my_rate = warp_rate_max(tid < nt / 32 ? red[tid] : T(0));
            if (tid == 0 && my_rate > T(0)) atomicMax(a.rate_wr + g, rate_bits(my_rate));
        }
    }
}

// FP32: lane = column, warp = row of a 32 x 16 tile of positions (one halo position on each side; 30 x 14
// cells). Each thread keeps its cell's primitives for planes k - 1, k, k + 1 in registers, exchanges plane k
// with its x-neighbours by shuffles and with its y-neighbours through shared memory (double-buffered by
// plane parity, one block barrier per plane: the row above's south flux of plane k is read after the
// barrier of plane k + 1), and evaluates the west x-face and south y-face of its cell as a packed pair and
// the bottom z-face alone. Raw planes and U^n arrive by
// asynchronous copies in the thread's own slots of shared memory: with them in registers, a plane per
// variable and an address each, a plane took 37.5 warp instructions per cell at 58 % issue; now 31.4 at
// 67 % (256^3, one scalar: 2603 -> 1938 us a step, 64^3 96 -> 56). Measured and dropped: all work spread
// over the threads in phases as in FP64, faces paired with their neighbours' (30 instructions per cell,
// but 46 % issue between the barriers: 2630 us, though 44 against 71 us on 200 x 2 x 200).
template <int NS> struct March3 {
    static constexpr int NV = 5 + NS, TW = tail3(NV), NC = 9 + NS, FIELDS = NC + 3 + NV, TH = threads3<float>();
};

template <int NS, bool ONE> __device__ __forceinline__ void stage3_march(const StageArgs3<float> &a)
{
    using M = March3<NS>;
    constexpr int NV = M::NV, TW = M::TW, NC = M::NC, TH = M::TH, ROWS = TH / 32;
    pdl_trigger();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float red[ROWS];
    float *const Q = reinterpret_cast<float *>(smem_raw), *const QT = Q + 16 * TH, *const N4 = QT + 4 * TW * TH,
                *const NT = N4 + 8 * TH, *const X = NT + 2 * TW * TH;   // X: exchanged fields [2][FIELDS][TH]
    const int tid = threadIdx.x, lane = tid & 31, wy = tid >> 5;
    const int ts = wy > 0 ? tid - 32 : tid, tn = wy < ROWS - 1 ? tid + 32 : tid;   // clamped neighbour rows
    const int te = lane < 31 ? 1 : 0;
    auto at = [&](int buf, int f, int t) -> float & { return X[(buf * M::FIELDS + f) * TH + t]; };

    const int4 unit = __ldg(a.units + blockIdx.x);
    const int g = a.ngrids == 1 ? 0 : unit.x;
    const int x0 = unit.y & 0xffff, w = unit.y >> 16, y0 = unit.z & 0xffff, h = unit.z >> 16;
    const int k0 = unit.w & 0xffff, k1 = (int)((unsigned)unit.w >> 16);
    const GridDev3 &G = ONE ? a.g0 : a.grids[g];
    const GridCoef3<float> K = ONE ? a.c0 : a.coef[g];
    const int nk = G.nk, pitch = G.pitch, bcB = G.bc[4], bcT = G.bc[5];
    int kx, ky;
    const int isrc = resolve_index(x0 - 1 + lane, G.ni, G.bc[0], G.bc[1], kx);
    const int jsrc = resolve_index(y0 - 1 + wy, G.nj, G.bc[2], G.bc[3], ky);
    const bool inflow_xy = kx == 2 || ky == 2;
    const int xy = jsrc * pitch + isrc;   // (an own cell's own place)
    const bool own = lane >= 1 && lane <= w && wy >= 1 && wy <= h;
    const int eps1 = G.eps1, xi_form = G.xi_form;
    const bool use_s1 = G.use_s1 != 0;
    const bool stage_mode = a.mode == MODE_STAGE;
    const bool combine = stage_mode && a.alpha != 0.f;
    const float hx = 0.5f * K.idx, hy = 0.5f * K.idy, hz = 0.5f * K.idz;
    const long long row = (long long)G.nj * pitch, tails = 4 * G.vol;
    const float *const src = a.src + G.off + 4 * (long long)xy, *const srct = a.src + G.off + tails + TW * (long long)xy;
    const float *const un = a.un + G.off + 4 * (long long)xy, *const unt = a.un + G.off + tails + TW * (long long)xy;
    float *const dst = a.dst + G.off + 4 * (long long)xy, *const dstt = a.dst + G.off + tails + TW * (long long)xy;
    const unsigned sq = (unsigned)__cvta_generic_to_shared(Q + 4 * tid), sqt = (unsigned)__cvta_generic_to_shared(QT + TW * tid);
    const unsigned sn = (unsigned)__cvta_generic_to_shared(N4 + 4 * tid), snt = (unsigned)__cvta_generic_to_shared(NT + TW * tid);
    pdl_wait();
    if (a.rate_zero && blockIdx.x == 0)
        for (int i = tid; i < a.ngrids; i += TH) a.rate_zero[i] = 0ull;
    float dt = 0.f;
    if (stage_mode) dt = a.dt_fixed_t > 0.f ? a.dt_fixed_t : a.cfl_t / rate_at<float>(a.rate_rd + g);

    // starts the copies of plane k (to k1 at most) and, in the same group, of U^n of plane k - 2
    auto issue = [&](int k) {
        if (k <= k1) {
            int kz;
            const long long o = (long long)resolve_index(k, nk, bcB, bcT, kz) * row;
            copy_cell(sq + (k & 3) * (16 * TH), src + 4 * o);
            copy_tail<TW>(sqt + (k & 3) * (4 * TW * TH), srct + TW * o);
        }
        const int m = k - 2;
        if (combine && own && m >= k0 && m < k1) {
            const long long o = (long long)m * row;
            copy_cell(sn + (m & 1) * (16 * TH), un + 4 * o);
            copy_tail<TW>(snt + (m & 1) * (4 * TW * TH), unt + TW * o);
        }
        copies_commit();
    };
    auto raw = [&](const float *B, const float *BT, float v[NV]) {
        float t[TW];
        ld_own(B, v);
        ld_tail<TW>(BT, t);
#pragma unroll
        for (int s = 4; s < NV; ++s) v[s] = t[s - 4];
    };
    auto finish = [&](int k, C3<float, NS> &c) {
        int kz;
        resolve_index(k, nk, bcB, bcT, kz);
        float v[NV];
        raw(Q + 4 * ((k & 3) * TH + tid), QT + TW * ((k & 3) * TH + tid), v);
        float ri = rcp(v[0]);
        c.r = v[0];
        c.u = v[1] * ri; c.v = v[2] * ri; c.w = v[3] * ri;
        c.p = K.gm1 * (v[4] - 0.5f * c.r * (c.u * c.u + c.v * c.v + c.w * c.w));
#pragma unroll
        for (int s = 0; s < NS; ++s) c.k[s] = v[5 + s] * ri;
        if (kx | ky | kz) {
            if (kx == 1) c.u = -c.u;
            if (ky == 1) c.v = -c.v;
            if (kz == 1) c.w = -c.w;
            if (inflow_xy || kz == 2) {
                c.r = K.inflow[0]; c.u = K.inflow[1]; c.v = K.inflow[2]; c.w = K.inflow[3]; c.p = K.inflow[4];
#pragma unroll
                for (int s = 0; s < NS; ++s) c.k[s] = K.inflow[5 + s];
                ri = rcp(c.r);
            }
        }
        derive3(c, ri, K);
    };

    for (int k = k0 - 1; k <= k0 + 2; ++k) issue(k);
    copies_wait<1>();
    // window: planes k - 1 (Wm), k (W0), k + 1 (Wp)
    C3<float, NS> Wm, W0, Wp;
    finish(k0 - 1, Wm);
    finish(k0, W0);
    finish(k0 + 1, Wp);
    // detector values of plane k0 - 1 (x and y faces), for the first z-face
    float Px_m, Pxe_m, Py_m, Pyn_m;
    {
        const int bp = (k0 + 1) & 1;   // (plane k0 writes the other buffer)
        Px_m = ratio_P(shup(Wm.r, 1), shup(Wm.p, 1), Wm.r, Wm.p);
        Pxe_m = shdn(Px_m, 1);
        at(bp, 0, tid) = Wm.r;
        at(bp, 4, tid) = Wm.p;
        __syncthreads();
        Py_m = ratio_P(at(bp, 0, ts), at(bp, 4, ts), Wm.r, Wm.p);
        Pyn_m = ratio_P(Wm.r, Wm.p, at(bp, 0, tn), at(bp, 4, tn));
    }
    float acc[NV];
    float my_rate = 0.f;
    float Pz = ratio_P(Wm.r, Wm.p, W0.r, W0.p);   // bottom z-face of plane k

#pragma unroll 1
    for (int k = k0; k <= k1; ++k) {
        const int b = k & 1;
        // detector values of plane k known to this thread
        const float Px = ratio_P(shup(W0.r, 1), shup(W0.p, 1), W0.r, W0.p);   // west x-face
        const float Pxe = shdn(Px, 1);                                        // east x-face
        const float Pzt = ratio_P(W0.r, W0.p, Wp.r, Wp.p);                    // top z-face

        // exchange plane k with the rows above and below
        at(b, 0, tid) = W0.r; at(b, 1, tid) = W0.u; at(b, 2, tid) = W0.v; at(b, 3, tid) = W0.w; at(b, 4, tid) = W0.p;
        at(b, 5, tid) = W0.c2; at(b, 6, tid) = W0.H; at(b, 7, tid) = W0.sr; at(b, 8, tid) = W0.Mq;
#pragma unroll
        for (int s = 0; s < NS; ++s) at(b, 9 + s, tid) = W0.k[s];
        at(b, NC, tid) = Px;
        at(b, NC + 1, tid) = Pz;
        at(b, NC + 2, tid) = Pzt;
        __syncthreads();
        // the north neighbour's south flux of plane k - 1 (written after the previous barrier)
        if (k > k0) {
#pragma unroll
            for (int v = 0; v < NV; ++v) acc[v] = vfma(-hy, at(b ^ 1, NC + 3 + v, tn), acc[v]);
        }
        C3<float, NS> S;   // the cell below (row j - 1)
        S.r = at(b, 0, ts); S.u = at(b, 1, ts); S.v = at(b, 2, ts); S.w = at(b, 3, ts); S.p = at(b, 4, ts);
        S.c2 = at(b, 5, ts); S.H = at(b, 6, ts); S.sr = at(b, 7, ts); S.Mq = at(b, 8, ts);
#pragma unroll
        for (int s = 0; s < NS; ++s) S.k[s] = at(b, 9 + s, ts);
        const float Py = ratio_P(S.r, S.p, W0.r, W0.p);
        const float Pyn = ratio_P(W0.r, W0.p, at(b, 0, tn), at(b, 4, tn));

        // s1 of the three faces (Eq. 96: the face and the 8 transverse faces of its cells)
        V2 s1 = mk2(1.f, 1.f);
        float s1z = 1.f;
        if (use_s1) {
            const float ax = min9(Px, shup(Py, 1), shup(Pyn, 1), Py, Pyn, shup(Pz, 1), shup(Pzt, 1), Pz, Pzt);
            const float ay = min9(Py, at(b, NC, ts), at(b, NC, ts + te), Px, Pxe, at(b, NC + 1, ts), at(b, NC + 2, ts), Pz, Pzt);
            s1 = detector_of(mk2(ax, ay));
            s1z = detector_of(min9(Pz, Px_m, Pxe_m, Px, Pxe, Py_m, Pyn_m, Py, Pyn));
        }

        // the west and the south face as a pair (the halo rows need none of theirs but the top row's
        // south face; the segment's last plane needs neither)
        float Fw[NV], Fs[NV], Fb[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) Fw[v] = Fs[v] = Fb[v] = 0.f;
        if (wy > 0 && k < k1) {
            C3<float, NS> Wl;   // the cell to the west (lane - 1)
            Wl.r = shup(W0.r, 1); Wl.u = shup(W0.u, 1); Wl.v = shup(W0.v, 1); Wl.w = shup(W0.w, 1);
            Wl.p = shup(W0.p, 1); Wl.c2 = shup(W0.c2, 1); Wl.H = shup(W0.H, 1); Wl.sr = shup(W0.sr, 1);
            Wl.Mq = shup(W0.Mq, 1);
#pragma unroll
            for (int s = 0; s < NS; ++s) Wl.k[s] = shup(W0.k[s], 1);
            V2 G2[NV];
            roeam_flux3<V2, float, NS>(side3_xy(Wl, S), side3_xy(W0, W0), s1, K, eps1, xi_form, G2);
#pragma unroll
            for (int v = 0; v < NV; ++v) { const int o = v == 1 ? 2 : (v == 2 ? 1 : v); Fw[v] = G2[v].v.x; Fs[v] = G2[o].v.y; }
        }
        if (wy > 0 && wy < ROWS - 1) {
            float G2[NV];
            roeam_flux3<float, float, NS>(side3(Wm, 2), side3(W0, 2), s1z, K, eps1, xi_form, G2);
#pragma unroll
            for (int v = 0; v < NV; ++v) { const int o = v == 1 ? 2 : (v == 2 ? 3 : (v == 3 ? 1 : v)); Fb[v] = G2[o]; }
        }

        // this plane's south flux, read by the row below after the next plane's barrier
#pragma unroll
        for (int v = 0; v < NV; ++v) at(b, NC + 3 + v, tid) = Fs[v];

        // finish plane k - 1: R = hx (F_w - F_e) + hy (F_s - F_n) + hz (F_b - F_t) of the doubled fluxes
        if (k > k0 && own) {
            const int m = k - 1;
            const long long o = (long long)m * row;
            float out[NV], t[TW];
#pragma unroll
            for (int v = 0; v < NV; ++v) out[v] = vfma(-hz, Fb[v], acc[v]);
            if (stage_mode) {
                float uk[NV], u0[NV];
                const float *const q4 = Q + 4 * ((m & 3) * TH + tid), *const qt = QT + TW * ((m & 3) * TH + tid);
                raw(q4, qt, uk);
                // (the first stage, alpha = 0 and beta = 1, combines with U^(k) itself)
                raw(combine ? N4 + 4 * ((m & 1) * TH + tid) : q4, combine ? NT + TW * ((m & 1) * TH + tid) : qt, u0);
#pragma unroll
                for (int v = 0; v < NV; ++v) out[v] = vfma(a.alpha, u0[v], a.beta * vfma(dt, out[v], uk[v]));
            }
#pragma unroll
            for (int s = 0; s < TW; ++s) t[s] = s < NV - 4 ? out[4 + (s < NV - 4 ? s : 0)] : 0.f;
            st_cell(dst + 4 * o, out);
            st_tail<TW>(dstt + TW * o, t);
            if (stage_mode) check_cell3(out, a.want_rate != 0, K, a.status, my_rate);
        }
        if (k == k1) break;
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] = vfma(hx, Fw[v] - shdn(Fw[v], 1), vfma(hy, Fs[v], hz * Fb[v]));

        // advance the window: plane k + 2 enters; the raw slot of plane k - 1 takes plane k + 3
        Px_m = Px; Pxe_m = Pxe; Py_m = Py; Pyn_m = Pyn;
        Pz = Pzt;   // the top z-face of plane k is the bottom one of plane k + 1
        Wm = W0;
        W0 = Wp;
        issue(k + 3);
        copies_wait<1>();
        if (k + 2 <= k1) finish(k + 2, Wp);
    }
    if (a.want_rate) {
        my_rate = warp_rate_max(my_rate);
        if (lane == 0) red[wy] = my_rate;
        __syncthreads();
        if (tid < 32) {
            my_rate = warp_rate_max(tid < ROWS ? red[tid] : 0.f);
            if (tid == 0 && my_rate > 0.f) atomicMax(a.rate_wr + g, rate_bits(my_rate));
        }
    }
}

template <typename T, int NS>
__global__ void __launch_bounds__(threads3<T>(), 1) stage3_kernel(const StageArgs3<T> a)
{
    if constexpr (sizeof(T) == 4) stage3_march<NS, false>(a);
    else stage3_phases<T, NS>(a);
}
// FP32 with three scalars, a single grid: its descriptor and constants are kernel arguments, not registers,
// of which this kernel has none to spare (192^3: 1073 -> 931 us a step). With fewer scalars the
// constants as operands change nothing or lose 0.7 %, nor does FP64 gain.
template <int NS>
__global__ void __launch_bounds__(threads3<float>(), 1) stage3_single(const __grid_constant__ StageArgs3<float> a)
{
    stage3_march<NS, true>(a);
}

// Host float64 layout [nv][nk][nj][ni] per grid <-> the state's quads and tails, blockIdx.y = grid; as
// the 2D pack and unpack: IO_PER cells per thread in flight, 32-bit indices, and the pack also takes
// the time-step rate of the state it writes.
template <typename T, int NS>
__global__ void __launch_bounds__(256) pack3_kernel(const GridDev3 *grids, const GridCoef3<T> *coef, int g_lo,
                                                    const double *__restrict__ packed, T *__restrict__ U,
                                                    unsigned long long *rate)
{
    constexpr int NV = 5 + NS, TW = tail3(NV);
    __shared__ T red[8];
    const int g = g_lo + blockIdx.y;
    const GridDev3 &G = grids[g];
    const GridCoef3<T> &K = coef[g];
    const unsigned ni = (unsigned)G.ni, n = ni * (unsigned)G.nj * (unsigned)G.nk, stride = gridDim.x * 256u;
    const double *__restrict__ src = packed + G.poff;
    T *__restrict__ quads = U + G.off, *__restrict__ tails = quads + 4 * G.vol;
    T m = T(0);
    for (unsigned q0 = blockIdx.x * 256u + threadIdx.x; q0 < n; q0 += IO_PER * stride) {
        T v[IO_PER][NV];
#pragma unroll
        for (int e = 0; e < IO_PER; ++e) {
            const unsigned q = q0 + e * stride;
            if (q < n)
#pragma unroll
                for (int k = 0; k < NV; ++k) v[e][k] = T(src[(long long)k * n + q]);
        }
#pragma unroll
        for (int e = 0; e < IO_PER; ++e) {
            const unsigned q = q0 + e * stride;
            if (q >= n) break;
            const unsigned jk = q / ni, i = q - jk * ni;
            const long long c = (long long)jk * G.pitch + i;
            T t[TW];
#pragma unroll
            for (int k = 0; k < TW; ++k) t[k] = k < NV - 4 ? v[e][4 + (k < NV - 4 ? k : 0)] : T(0);
            st_cell(quads + 4 * c, v[e]);
            st_tail<TW>(tails + TW * c, t);
            m = vmax(m, cell_rate3(cell_prims3(v[e][0], v[e][1], v[e][2], v[e][3], v[e][4], K), K));
        }
    }
    m = block_max<256>(m, red);
    if (threadIdx.x == 0 && m > T(0)) atomicMax(rate + g, rate_bits(m));
}

template <typename T, int NS>
__global__ void __launch_bounds__(256) unpack3_kernel(const GridDev3 *grids, int g_lo, const T *__restrict__ U,
                                                      double *__restrict__ packed)
{
    constexpr int NV = 5 + NS, TW = tail3(NV);
    const GridDev3 &G = grids[g_lo + blockIdx.y];
    const unsigned ni = (unsigned)G.ni, n = ni * (unsigned)G.nj * (unsigned)G.nk, stride = gridDim.x * 256u;
    const T *__restrict__ quads = U + G.off, *__restrict__ tails = quads + 4 * G.vol;
    double *__restrict__ dst = packed + G.poff;
    for (unsigned q0 = blockIdx.x * 256u + threadIdx.x; q0 < n; q0 += IO_PER * stride) {
        T v[IO_PER][4], t[IO_PER][TW];
#pragma unroll
        for (int e = 0; e < IO_PER; ++e) {
            const unsigned q = q0 + e * stride;
            if (q < n) {
                const unsigned jk = q / ni, i = q - jk * ni;
                const long long c = (long long)jk * G.pitch + i;
                ld_own(quads + 4 * c, v[e]);
                ld_tail<TW>(tails + TW * c, t[e]);
            }
        }
#pragma unroll
        for (int e = 0; e < IO_PER; ++e) {
            const unsigned q = q0 + e * stride;
            if (q < n) {
#pragma unroll
                for (int k = 0; k < NV; ++k) dst[(long long)k * n + q] = (double)(k < 4 ? v[e][k & 3] : t[e][k < 4 ? 0 : k - 4]);
            }
        }
    }
}

// FP64 block partials of sum V Q over grid g (gridDim.x x MAX_VARS3 doubles).
template <typename T>
__global__ void __launch_bounds__(256) totals3_kernel(const GridDev3 *grids, int g, const T *U, int nv, double *partials)
{
    __shared__ double wred[8][MAX_VARS3];
    const GridDev3 &G = grids[g];
    const long long n = (long long)G.ni * G.nj * G.nk;
    const double V = G.dx * G.dy * G.dz;
    double s[MAX_VARS3];
    for (int v = 0; v < MAX_VARS3; ++v) s[v] = 0.0;
    for (long long q = (long long)blockIdx.x * 256 + threadIdx.x; q < n; q += (long long)gridDim.x * 256) {
        const long long c = (q / G.ni) * G.pitch + q % G.ni;
        const int tw = tail3(nv);
        for (int v = 0; v < nv; ++v)
            s[v] += V * (double)(v < 4 ? U[G.off + 4 * c + v] : U[G.off + 4 * G.vol + tw * c + v - 4]);
    }
    for (int o = 16; o > 0; o >>= 1)
        for (int v = 0; v < MAX_VARS3; ++v) s[v] += __shfl_xor_sync(0xffffffffu, s[v], o);
    if ((threadIdx.x & 31) == 0)
        for (int v = 0; v < MAX_VARS3; ++v) wred[threadIdx.x >> 5][v] = s[v];
    __syncthreads();
    if (threadIdx.x < MAX_VARS3) {
        double r = 0.0;
        for (int w = 0; w < 8; ++w) r += wred[w][threadIdx.x];
        partials[(size_t)blockIdx.x * MAX_VARS3 + threadIdx.x] = r;
    }
}

// ------------------------------------------------------------------ launchers
template <typename T, int NS> struct Stage3Variant {
    static constexpr bool SINGLE = sizeof(T) == 4 && NS == 3;
    static cudaError_t launch(const StageArgs3<T> &a, int threads, size_t smem, cudaStream_t s)
    {
        if constexpr (SINGLE)
            if (a.ngrids == 1) return launch_pdl(stage3_single<NS>, dim3((unsigned)a.nunits), dim3((unsigned)threads), smem, s, a);
        return launch_pdl(stage3_kernel<T, NS>, dim3((unsigned)a.nunits), dim3((unsigned)threads), smem, s, a);
    }
    static cudaError_t prepare()
    {
        if constexpr (SINGLE) {
            const cudaError_t e = cudaFuncSetAttribute(stage3_single<NS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TILE_SMEM_MAX);
            if (e != cudaSuccess) return e;
        }
        return cudaFuncSetAttribute(stage3_kernel<T, NS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TILE_SMEM_MAX);
    }
    static cudaError_t pack(dim3 grid, const GridDev3 *grids, const GridCoef3<T> *coef, int g_lo, const double *packed,
                            T *U, unsigned long long *rate, cudaStream_t s)
    {
        pack3_kernel<T, NS><<<grid, 256, 0, s>>>(grids, coef, g_lo, packed, U, rate);
        return cudaGetLastError();
    }
    static cudaError_t unpack(dim3 grid, const GridDev3 *grids, int g_lo, const T *U, double *packed, cudaStream_t s)
    {
        unpack3_kernel<T, NS><<<grid, 256, 0, s>>>(grids, g_lo, U, packed);
        return cudaGetLastError();
    }
};

#define ROEAM3_DISPATCH(CALL)                                  \
    switch (nscal) {                                           \
    case 0: return Stage3Variant<T, 0>::CALL;                  \
    case 1: return Stage3Variant<T, 1>::CALL;                  \
    case 2: return Stage3Variant<T, 2>::CALL;                  \
    default: return Stage3Variant<T, 3>::CALL;                 \
    }

template <typename T>
cudaError_t Launchers3<T>::stage(const StageArgs3<T> &a, int nscal, int threads, size_t smem, cudaStream_t s)
{
    if (a.nunits <= 0) return cudaSuccess;
    ROEAM3_DISPATCH(launch(a, threads, smem, s))
}

template <typename T> cudaError_t Launchers3<T>::prepare(int nscal) { ROEAM3_DISPATCH(prepare()) }

// IO_PER cells per thread, but a cell per thread as long as that takes no more than two blocks per SM (the
// FP64 rates of four cells in a row keep a few SMs busy while the others idle: loading 16^3 40.7 -> 27.3 us
// in FP64, 18.5 -> 15.3 in FP32, reading it 29.7 -> 27.6).
static inline dim3 io_grid3(long long max_cells, int grids)
{
    const long long full = (max_cells + 256 * IO_PER - 1) / (256 * IO_PER), spread = (max_cells + 255) / 256;
    const long long bx = std::max(full, std::min(spread, 304ll / grids));
    return dim3((unsigned)(bx < 1 ? 1 : (bx > 4096 ? 4096 : bx)), (unsigned)grids);
}

template <typename T>
cudaError_t Launchers3<T>::pack(const GridDev3 *grids, const GridCoef3<T> *coef, int g_lo, int g_hi, int nscal,
                                long long max_cells, const double *packed, T *U, unsigned long long *rate, cudaStream_t s)
{
    if (g_hi <= g_lo) return cudaSuccess;
    ROEAM3_DISPATCH(pack(io_grid3(max_cells, g_hi - g_lo), grids, coef, g_lo, packed, U, rate, s))
}

template <typename T>
cudaError_t Launchers3<T>::unpack(const GridDev3 *grids, int g_lo, int g_hi, int nscal, long long max_cells, const T *U,
                                  double *packed, cudaStream_t s)
{
    if (g_hi <= g_lo) return cudaSuccess;
    ROEAM3_DISPATCH(unpack(io_grid3(max_cells, g_hi - g_lo), grids, g_lo, U, packed, s))
}

template <typename T>
cudaError_t Launchers3<T>::totals(const GridDev3 *grids, int g, const T *U, int nv, double *partials, int nblocks,
                                  cudaStream_t s)
{
    totals3_kernel<T><<<nblocks, 256, 0, s>>>(grids, g, U, nv, partials);
    return cudaGetLastError();
}

}  // namespace roeam
