// wb_sweep_js.cuh -- the Jiang-Shu and WENO-Z flux sweeps (staging, slots and
// eigen-structure of wb_sweep.cuh), for FP64 and FP32.
//
// One interface per thread.  FP64 takes the interface arithmetic below
// (sweep_flux), which counts operations of the FP64 pipe (two per clock and SM
// on this GPU, 87 % busy, everything else hidden behind it): smoothness
// indicators of ten operations and one reciprocal for the two phi_N of a field
// (60 instead of 83 operations), three-operation reciprocals, Alfven rows that act
// on the differences directly.  96^3, x + y + z sweep of a step: 21.3 -> 17.6
// ms; three and four blocks per SM (168 and 128 registers) are no faster.
// FP32 takes the one of wb_sweep.cuh (interface_flux), which packs the U and F
// differences of a stencil step, and here the two sides of phi_N, in the lanes
// of Blackwell's packed FP32 instructions: 1 333 to 1 348 instructions per
// interface (1 454 before), issued on 60 to 62 % of cycles by sixteen warps per
// SM.  256^3, x, y, z sweeps of a step: 2.88 / 2.83 / 3.01 -> 2.71 / 2.77 / 2.79
// ms.  Two interfaces per thread (neighbouring pencils in the two lanes) need
// only 1 107 instructions per interface, but 200 to 255 registers: eight warps
// per SM issue on 41 % of cycles, and with the staging moved to further warps
// (cp.async, registers split between the warps) on 50 %: 3.1 to 3.5 and 2.6 to
// 3.0 ms per axis.
#pragma once
#include "wb_sweep.cuh"

#include <cmath>

namespace wb {
namespace {

// resident blocks per SM the register budget is shaped for
#ifndef WB_SWEEP_BLOCKS_F32
#define WB_SWEEP_BLOCKS_F32 4
#endif
#ifndef WB_SWEEP_BLOCKS_F64
#define WB_SWEEP_BLOCKS_F64 2
#endif
template <class T> constexpr int kMinBlocks = sizeof(T) == 4 ? WB_SWEEP_BLOCKS_F32 : WB_SWEEP_BLOCKS_F64;
// per-thread slots of sweep_flux: back-projection coefficients, then the
// Alfven and entropy projections while the fast/slow group is reconstructed
enum : int { B_ALF = 0, B_ALS, B_AFCF, B_ASCS, B_ASR, B_SSR, B_RAG, kNBackV = 7 };
constexpr int kSlotsV = kNBackV + 24;
template <class T> constexpr int kSlots = sizeof(T) == 4 ? thread_slots(4) : kSlotsV;

// ---- phi_N (Sec. 2.1) ------------------------------------------------------------
// With a, b, c, d four successive differences, the IS_k as printed are quadratic
// forms; completed squares keep them sums of non-negative terms,
//   IS_0 / 16 = (a - 11/8 b)^2 + 39/64 b^2, IS_1 / 16 = (b - 5/8 c)^2 + 39/64 c^2,
//   IS_2 / 16 = (d - 11/8 c)^2 + 39/64 c^2,
// each good to three roundings.  The weights depend on the ratios of the
// eps + IS_k only, so e_k = (eps + IS_k) / 16, ten operations, serve.  (The forms
// multiplied out, a (a - 11/4 b) + 5/2 b^2 and so on, also take ten, but lose
// four bits where a = 11/8 b, and round IS_0 and IS_2 of a symmetric stencil
// differently: WENO-Z divides their difference, then a rounding error, by the
// smallest eps + IS_k.)
template <class V>
__device__ __forceinline__ void smoothness(V a, V b, V c, V d, typename Lanes<V>::S eps16, V& e0, V& e1, V& e2) {
    using S = typename Lanes<V>::S;
    const V eps = splat<V>(eps16), k39 = splat<V>(S(39.0 / 64.0)), k11 = splat<V>(S(-1.375)), k5 = splat<V>(S(-0.625));
    const V sb = vfma(vmul(b, k39), b, eps), sc = vfma(vmul(c, k39), c, eps);
    const V t0 = vfma(b, k11, a), t1 = vfma(c, k5, b), t2 = vfma(c, k11, d);
    e0 = vfma(t0, t0, sb);
    e1 = vfma(t1, t1, sc);
    e2 = vfma(t2, t2, sc);
}

// p = a - 2b + c
template <class V>
__device__ __forceinline__ V second(V a, V b, V c) {
    return vfma(b, splat<V>(typename Lanes<V>::S(-2)), vadd(a, c));
}

// phi_N = (w_0 p + w_2 q / 2) / 3 - q / 12 with p = a - 2b + c, q = b - 2c + d and
// the weights w_k proportional to d_k a_k, d = (1, 6, 3), over the common W = a_0 +
// 6 a_1 + 3 a_2: 12 phi_N W = 4 a_0 p + (3 a_2 - a_0 - 6 a_1) q.  The bracket is
// w_2 - 1/2 of a side with one rounding; taking the two sides' -q / 12 apart
// from their weighted parts instead cancels at jumps (blasts, both precisions:
// 1.4 times the rounding error).
template <class V>
__device__ __forceinline__ V phi_num(V a0, V a1, V a2, V p, V q, V& w) {
    using S = typename Lanes<V>::S;
    const V t = vfma(a1, splat<V>(S(6)), a0);
    w = vfma(a2, splat<V>(S(3)), t);
    return vfma(vfms(a2, splat<V>(S(3)), t), q, vmul(vmul(a0, splat<V>(S(4))), p));
}

// (phi_N(am, bm, cm, dm) - phi_N(ap, bp, cp, dp)) / 2 for Jiang-Shu weights, a_k =
// 1 / e_k^2, taken times (e_0 e_1 e_2)^2.
__device__ __forceinline__ void js_side(double a, double b, double c, double d, double eps16, double& a0, double& a1,
                                        double& a2, double& p, double& q) {
    double e0, e1, e2;
    smoothness<double>(a, b, c, d, eps16, e0, e1, e2);
    const double m0 = e1 * e2, m1 = e0 * e2, m2 = e0 * e1;
    a0 = m0 * m0;
    a1 = m1 * m1;
    a2 = m2 * m2;
    p = second(a, b, c);
    q = second(b, c, d);
}
// FP64: one reciprocal for both sides, of the product of their denominators,
// where neither exceeds 1e130 (the product and its numerators then stay far
// inside the range); else one division each.
__device__ __forceinline__ double half_phi_diff(double am, double bm, double cm, double dm, double ap, double bp,
                                                double cp, double dp, double eps16) {
    double a0m, a1m, a2m, pm, qm, wm, a0p, a1p, a2p, pp, qp, wp;
    js_side(am, bm, cm, dm, eps16, a0m, a1m, a2m, pm, qm);
    js_side(ap, bp, cp, dp, eps16, a0p, a1p, a2p, pp, qp);
    const double nm = phi_num(a0m, a1m, a2m, pm, qm, wm), np = phi_num(a0p, a1p, a2p, pp, qp, wp);
    double r;
    // high words of the (positive) denominators against that of 1e130
    if (max(__double2hiint(wm), __double2hiint(wp)) < 0x5af00000) {
        r = fma(nm, wp, -(np * wm)) * recip_inrange(wm * wp);
    } else {
        double one;
        const double im = 1.0 / wm, ip = 1.0 / wp;
        r = phi_num(a0m * im, a1m * im, a2m * im, pm, qm, one) - phi_num(a0p * ip, a1p * ip, a2p * ip, pp, qp, one);
    }
    return r * (1.0 / 24.0);
}
// FP32: reciprocals of the e_k^2 keep the range (products of them could
// overflow).  12 phi_N of both sides.
__device__ __forceinline__ float2 js_phi12(float2 a, float2 b, float2 c, float2 d, float eps16) {
    float2 e0, e1, e2, w;
    smoothness<float2>(a, b, c, d, eps16, e0, e1, e2);
    const float2 n = phi_num(vrcp(vmul(e0, e0)), vrcp(vmul(e1, e1)), vrcp(vmul(e2, e2)), second(a, b, c),
                             second(b, c, d), w);
    return vmul(n, vrcp(w));
}

// WENO-Z (the alternative Sec. 2.1 names): alpha_k = d_k (1 + tau5 / (eps +
// IS_k)), tau5 = |IS_0 - IS_2|; the ratio is free of the common factor.
template <class V>
__device__ __forceinline__ V z_phi12(V a, V b, V c, V d, typename Lanes<V>::S eps16) {
    V e0, e1, e2, w;
    smoothness<V>(a, b, c, d, eps16, e0, e1, e2);
    const V tau = vabs(vsub(e0, e2)), one = splat<V>(typename Lanes<V>::S(1));
    const V n = phi_num(vfma(tau, vrcp(e0), one), vfma(tau, vrcp(e1), one), vfma(tau, vrcp(e2), one), second(a, b, c),
                        second(b, c, d), w);
    return vmul(n, vrcp(w));
}

// Correction of eq. FWENO for one characteristic field, -phi_N(D+_{i-3/2} ..) +
// phi_N(D-_{i+5/2} ..), from the split differences taken twice over, p_m = 2 D+
// of steps m = 0..3 and n_m = 2 D- of steps m = 1..4 of the stencil: phi_N with
// 4 eps on them, halved (exact).
template <bool Z>
__device__ __forceinline__ double weno_corr(const double (&p)[4], const double (&n)[4]) {
    constexpr double eps16 = 4.0 * 1e-6 / 16.0;
    if constexpr (Z) {
        const double rm = z_phi12<double>(n[3], n[2], n[1], n[0], eps16);
        const double rp = z_phi12<double>(p[0], p[1], p[2], p[3], eps16);
        return (rm - rp) * (1.0 / 24.0);
    } else {
        return half_phi_diff(n[3], n[2], n[1], n[0], p[0], p[1], p[2], p[3], eps16);
    }
}

// Weights of interface_flux (FP32): both sides of a field in one packed pair.
template <bool Z>
struct JsWeights {
    static constexpr bool kSplit = true;
    __device__ __forceinline__ float corr_s(const float (&p)[4], const float (&n)[4]) {
        constexpr float eps16 = 4.0f * 1e-6f / 16.0f;
        // the minus side in lane x, the plus side in lane y
        const float2 a = make_float2(n[3], p[0]), b = make_float2(n[2], p[1]), c = make_float2(n[1], p[2]),
                     d = make_float2(n[0], p[3]);
        const float2 r = Z ? z_phi12<float2>(a, b, c, d, eps16) : js_phi12(a, b, c, d, eps16);
        return (r.x - r.y) * (1.f / 24.f);
    }
};

// ---- one interface in FP64 --------------------------------------------------------------
// Left-vector coefficients (negated where the projection subtracts), the
// speeds and what the back-projection needs.
struct Eig64 {
    double rho, nu, nv1, nv2, nbm, hv2, be1, be2, nbe2;
    double cf, cs, ca;
    double Af, Bf, Cf, Df, As, Bs, Cs, Ds, nEe;
    double nvb;                       // -(be1 v1 + be2 v2)
    double q1, q2, q0, r1, r2;        // Alfven rows: q1 x3 + q2 x2 + q0 x0 +- (r1 x5 + r2 x4)
};

__device__ __forceinline__ void eigen64(double rho, double u, double v1, double v2, double bn, double b1, double b2,
                                        double p, double gamma, double rg1, Eig64& e, double (&back)[kNBackV]) {
    Eig<double> s;
    double bp[kNBack];
    eigen<double>(rho, u, v1, v2, bn, b1, b2, p, gamma, s, bp, 1);
    e.rho = s.rho;
    e.nu = -s.u;
    e.nv1 = -s.v1;
    e.nv2 = -s.v2;
    e.nbm = -s.bm;
    e.hv2 = s.hv2;
    e.be1 = s.be1;
    e.be2 = s.be2;
    e.nbe2 = -s.be2;
    e.cf = s.cf;
    e.cs = s.cs;
    e.ca = s.ca;
    e.Af = s.Af;
    e.Bf = s.Bf;
    e.Cf = s.Cf;
    e.Df = s.Df;
    e.As = s.As;
    e.Bs = s.Bs;
    e.Cs = s.Cs;
    e.Ds = s.Ds;
    e.nEe = -s.Ee;
    e.nvb = -(s.be1 * s.v1 + s.be2 * s.v2);
    e.q1 = s.Aa * s.be1;
    e.q2 = -s.Aa * s.be2;
    e.q0 = -(e.q1 * s.v2 + e.q2 * s.v1);
    e.r1 = s.Ba * s.be1;
    e.r2 = -s.Ba * s.be2;
    back[B_ALF] = bp[BP_ALF];
    back[B_ALS] = bp[BP_ALS];
    back[B_AFCF] = bp[BP_AFCF];
    back[B_ASCS] = bp[BP_ASCS];
    back[B_ASR] = bp[BP_ASR];
    back[B_SSR] = bp[BP_SSR];
    back[B_RAG] = bp[BP_RA2] * rg1;
}

// One difference vector on all seven left eigenvectors: fast-, slow-, slow+,
// fast+ into o4, Alfven-, entropy, Alfven+ into o3.
__device__ __forceinline__ void project(const Eig64& e, const double (&x)[7], double (&o4)[4], double (&o3)[3]) {
    const double du = fma(e.nu, x[0], x[1]);
    const double vpar = fma(e.be1, x[2], fma(e.be2, x[3], e.nvb * x[0]));
    const double bpar = fma(e.be1, x[4], e.be2 * x[5]);
    double P = fma(e.hv2, x[0], x[6]);
    P = fma(e.nu, x[1], P);
    P = fma(e.nv1, x[2], P);
    P = fma(e.nv2, x[3], P);
    P = fma(e.nbm, bpar, P);
    const double tf1 = fma(e.Af, du, e.Bf * vpar), tf2 = fma(e.Cf, bpar, e.Df * P);
    const double ts1 = fma(e.As, du, e.Bs * vpar), ts2 = fma(e.Cs, bpar, e.Ds * P);
    o4[0] = tf2 - tf1;
    o4[1] = ts2 - ts1;
    o4[2] = ts2 + ts1;
    o4[3] = tf2 + tf1;
    const double t1 = fma(e.q1, x[3], fma(e.q2, x[2], e.q0 * x[0]));
    const double t2 = fma(e.r1, x[5], e.r2 * x[4]);
    o3[0] = t1 + t2;
    o3[1] = fma(e.nEe, P, x[0]);
    o3[2] = t1 - t2;
}

// Largest |lambda_s| over the six cells and the interface state.
template <int CS>
__device__ __forceinline__ double lf_speed64(const double* __restrict__ cell, int nc, int s, const Eig64& e) {
    const double nc_s = (s == 0 || s == 6) ? e.cf : ((s == 1 || s == 5) ? e.ca : e.cs);
    double al = s == 3 ? fabs(e.nu) : (s < 3 ? fabs(e.nu + nc_s) : fabs(e.nu - nc_s));
#pragma unroll
    for (int m = 0; m < 6; m++) al = tmax_nonneg(al, cell[(SL + s) * nc + m * CS]);
    return al;
}

// Flux through one interface: cell points at stencil cell 0, the six cells are
// CS values apart.
template <bool Z, int CS>
__device__ __forceinline__ void sweep_flux(const double* __restrict__ cell, int nc, double gamma, double rg1,
                                           double* __restrict__ slot, int sstride, double (&out)[7]) {
    // 1-2. interface state and eigen-structure
    Eig64 e;
    {
        auto mean = [&](int s) { return 0.5 * (cell[s * nc + 2 * CS] + cell[s * nc + 3 * CS]); };
        const double rho = mean(SU), u = mean(SP_U), v1 = mean(SP_V1), v2 = mean(SP_V2), bn = mean(SP_BN),
                     b1 = mean(SU + 4), b2 = mean(SU + 5), p = mean(SP_P);
        double back[kNBackV];
        eigen64(rho, u, v1, v2, bn, b1, b2, p, gamma, rg1, e, back);
#pragma unroll
        for (int k = 0; k < kNBackV; k++) slot[k * sstride] = back[k];
    }
    // 4. Lax-Friedrichs speeds
    double al[7];
#pragma unroll
    for (int s = 0; s < 7; s++) al[s] = lf_speed64<CS>(cell, nc, s, e);
    // 3-4. the five differences of the stencil's U and F on all seven fields,
    // split: 2 D+- = l dF +- alpha l dU (eight values per field; those of the
    // Alfven and entropy fields wait in this thread's slots)
    double* park = slot + kNBackV * sstride;
    double dp[7][4], dn[7][4];
    double u0[7], f0[6];
#pragma unroll
    for (int f = 0; f < 7; f++) u0[f] = cell[(SU + f) * nc];
#pragma unroll
    for (int f = 0; f < 6; f++) f0[f] = cell[at_f<double>(f + 1, nc, 0)];
#pragma unroll
    for (int m = 0; m < 5; m++) {
        double x[7], w4[4], w3[3], g4[4], g3[3];
#pragma unroll
        for (int f = 0; f < 7; f++) {
            const double u1 = cell[(SU + f) * nc + (m + 1) * CS];
            x[f] = u1 - u0[f];
            u0[f] = u1;
        }
        const double dm = x[1];                   // the mass flux is the normal momentum
        project(e, x, w4, w3);
        x[0] = dm;
#pragma unroll
        for (int f = 0; f < 6; f++) {
            const double f1 = cell[at_f<double>(f + 1, nc, (m + 1) * CS)];
            x[f + 1] = f1 - f0[f];
            f0[f] = f1;
        }
        project(e, x, g4, g3);
#pragma unroll
        for (int s = 0; s < 7; s++) {
            const double w = s & 1 ? w3[s >> 1] : w4[s >> 1], g = s & 1 ? g3[s >> 1] : g4[s >> 1];
            double* mine = park + (s >> 1) * 8 * sstride;
            if (m < 4) {
                const double d = fma(al[s], w, g);
                if (s & 1) mine[m * sstride] = d;
                else dp[s][m] = d;
            }
            if (m > 0) {
                const double d = fma(-al[s], w, g);
                if (s & 1) mine[(3 + m) * sstride] = d;
                else dn[s][m - 1] = d;
            }
        }
    }
    // 5. weights, fast and slow fields, then Alfven and entropy
    double corr[7];
#pragma unroll
    for (int s = 0; s < 7; s += 2) corr[s] = weno_corr<Z>(dp[s], dn[s]);
#pragma unroll
    for (int s = 1; s < 7; s += 2) {
#pragma unroll
        for (int m = 0; m < 4; m++) {
            dp[s][m] = park[((s >> 1) * 8 + m) * sstride];
            dn[s][m] = park[((s >> 1) * 8 + 4 + m) * sstride];
        }
        corr[s] = weno_corr<Z>(dp[s], dn[s]);
    }
    // 6. back-projection: sum_s r_s corr_s in primitive variables, then dU/dW,
    // and the central flux (7 (F_i + F_{i+1}) - (F_{i-1} + F_{i+2})) / 12
    const double alf = slot[B_ALF * sstride], als = slot[B_ALS * sstride];
    const double afcf = slot[B_AFCF * sstride], ascs = slot[B_ASCS * sstride];
    const double ssr = slot[B_SSR * sstride];
    const double Fp = corr[6] + corr[0], Fm = corr[6] - corr[0];
    const double Sp = corr[4] + corr[2], Sm = corr[4] - corr[2];
    const double Ap = corr[5] + corr[1], nAm = corr[1] - corr[5];
    const double fs = fma(alf, Fp, als * Sp);
    const double drho = fma(e.rho, fs, corr[3]);
    const double du = fma(afcf, Fm, ascs * Sm);
    const double sg = ssr < 0.0 ? -1.0 : 1.0;          // sgn(B_n)
    const double dvpar = sg * (afcf * Sm - ascs * Fm);
    const double dbpar = slot[B_ASR * sstride] * (als * Fp - alf * Sp);
    const double dbper = ssr * nAm;
    const double dpg = slot[B_RAG * sstride] * fs;             // dp / (gamma - 1)
    const double dv1 = fma(e.be1, dvpar, e.nbe2 * Ap), dv2 = fma(e.be2, dvpar, e.be1 * Ap);
    double dF[7];
    dF[0] = drho;
    dF[4] = fma(e.be1, dbpar, e.nbe2 * dbper);
    dF[5] = fma(e.be2, dbpar, e.be1 * dbper);
    const double nd = -drho;
    dF[1] = fma(e.nu, nd, e.rho * du);
    dF[2] = fma(e.nv1, nd, e.rho * dv1);
    dF[3] = fma(e.nv2, nd, e.rho * dv2);
    const double vdv = fma(e.nu, du, fma(e.nv1, dv1, e.nv2 * dv2));       // -v dv
    dF[6] = fma(e.hv2, drho, dpg - fma(e.nbm, dbpar, e.rho * vdv));
#pragma unroll
    for (int f = 0; f < 7; f++) {
        const double* F = cell + at_f<double>(f, nc, 0);
        const double in = F[2 * CS] + F[3 * CS], ex = F[CS] + F[4 * CS];
        out[f] = fma(fma(in, 7.0, -ex), 1.0 / 12.0, dF[f]);
    }
}

// The flux through the lower face of cell c, rotated back, to the axis' arrays.
template <class T, int AXIS>
__device__ __forceinline__ void store_flux(const SweepArgs<T>& A, long long c, const T (&F)[7]) {
    const long long N = A.ncells;
    T* __restrict__ fo = A.flux;
    T fx, fy, fz;
    if (AXIS == 0) { fx = F[1]; fy = F[2]; fz = F[3]; }
    else if (AXIS == 1) { fy = F[1]; fz = F[2]; fx = F[3]; }
    else { fz = F[1]; fx = F[2]; fy = F[3]; }
    fo[c] = F[0];
    fo[N + c] = fx;
    fo[2 * N + c] = fy;
    fo[3 * N + c] = fz;
    fo[4 * N + c] = F[6];
    fo[5 * N + c] = F[4];
    fo[6 * N + c] = F[5];
}

// ---- one tile ------------------------------------------------------------------------
// Stages the TA + 5 cells of each of the TP pencils, then one thread per
// interface.  Cell s of pencil tp lies at tp * NS + s (x sweep) or s * TP + tp.
template <class T, int AXIS, int TA, int NCMAX, bool Z>
__device__ __forceinline__ void tile_body(const SweepArgs<T>& A, const Tile& tile, const PatchDev& P,
                                          T* __restrict__ sm, int tid) {
    constexpr int NT = kSweepNT, TP = kSweepNT / TA, NS = TA + 5, NC = NS * TP;
    constexpr int CS = AXIS == 0 ? 1 : TP;         // distance of a pencil's neighbouring cells
    const int na = AXIS == 0 ? P.nx : (AXIS == 1 ? P.ny : P.nz);
    const int np = AXIS == 0 ? P.ny : P.nx, n3 = AXIS == 2 ? P.ny : P.nz;

    __shared__ LinkTab tab;
    if (A.links) tab.load(A.patches, A.links, tile.x, tid);

    // staging: cells tile.y-3 .. tile.y+TA+1 along the axis, TP pencils
    constexpr int NIT = (NC + NT - 1) / NT;
    RawCell<T> raw[NIT];
    long long rc[NIT];
    bool rok[NIT], rown[NIT];
#pragma unroll
    for (int it = 0; it < NIT; it++) {
        const int e = tid + it * NT;
        int s, tp;
        if (AXIS == 0) { tp = e / NS; s = e - tp * NS; }
        else { s = e / TP; tp = e - s * TP; }
        int cp, w;
        tile_pencil(tile, tp, np, cp, w);
        const int raw_a = tile.y - 3 + s;
        // cells past the last interface's stencil serve idle threads only
        // (160^3 in 64 bricks: 2.66 -> 2.63 ms, 320 patches 8.44 -> 8.40)
        rok[it] = e < NC && w < n3 && raw_a < na + 2;
        rown[it] = raw_a >= tile.y && raw_a < tile.y + TA && raw_a < na;
        if (rok[it]) {
            int i, j, k;
            if (AXIS == 0) { i = raw_a; j = cp; k = w; }
            else if (AXIS == 1) { i = cp; j = raw_a; k = w; }
            else { i = cp; j = w; k = raw_a; }
            load_cell_tile<T, AXIS>(A, tab, P, i, j, k, raw[it], rc[it]);
        }
    }
#pragma unroll
    for (int it = 0; it < NIT; it++)
        if (rok[it])
            derive_cell<T, AXIS>(A, raw[it], rc[it], sm, NC, tid + it * NT, rown[it] && A.er != nullptr);
    __syncthreads();

    int ta, tp;
    if (AXIS == 0) { ta = tid & (TA - 1); tp = tid / TA; }
    else { tp = tid & (TP - 1); ta = tid / TP; }
    const int ia = tile.y + ta;
    int ip, w3;
    tile_pencil(tile, tp, np, ip, w3);
    if (ia >= na || w3 >= n3) return;
    const int mine = tile_cell<AXIS>(P, ia, ip, w3);
    const int i0 = (int)chk(AXIS == 0 ? tp * NS + ta : ta * TP + tp, NC - 5 * CS, A.flag);
    T F[7];
    T* slot = sm + kNSlot * NCMAX + tid;
    if constexpr (sizeof(T) == 8) {
        sweep_flux<Z, CS>(sm + i0, NC, T(A.gamma), T(A.rg1), slot, NT, F);
    } else {
        int id[6];
#pragma unroll
        for (int m = 0; m < 6; m++) id[m] = i0 + m * CS;
        JsWeights<Z> js;
        interface_flux<T, JsWeights<Z>, true>(sm, NC, id, T(A.gamma), slot, NT, js, F);
    }

    store_flux<T, AXIS>(A, chk(P.off + mine, A.ncells, A.flag), F);
}

// ---- an axis of one cell ----------------------------------------------------------------
// A periodic patch one cell deep along the axis (2-D and 1-D runs): all six
// stencil cells of an interface are its one cell, every projected difference
// is zero, and the flux is the central combination of four equal fluxes (or NaN,
// where the cell's state has no eigen-structure).  One
// thread per cell; tile.y is the first of kSweepNT cells.  As ordinary tiles
// these sweeps ran one warp per block at half its lanes through the whole
// interface arithmetic (64^2 x 1, RK4, FP64, four steps: 2.24 -> 1.24 ms).
template <class T, int AXIS>
__device__ __forceinline__ void flat_body(const SweepArgs<T>& A, const Tile& tile, const PatchDev& P,
                                          T* __restrict__ sm, int tid) {
    const int local = tile.y + tid, nxy = P.nx * P.ny;
    if (local >= nxy * P.nz) return;
    const int k = local / nxy, rem = local - k * nxy, j = rem / P.nx, i = rem - j * P.nx;
    RawCell<T> r;
    long long c;
    load_cell<T>(A, P, i, j, k, r, c);
    derive_cell<T, AXIS>(A, r, c, sm, kSweepNT, tid, A.er != nullptr);
    // a state without an eigen-structure gives NaN, as the interface arithmetic does
    // (the zero differences times its infinite or NaN coefficients)
    const T p = sm[SP_P * kSweepNT + tid];
    bool sound = r.rho > T(0) && p > T(0) && isfinite(r.rho) && isfinite(p);
    T F[7];
#pragma unroll
    for (int f = 0; f < 7; f++) {
        const T f1 = sm[at_f<T>(f, kSweepNT, tid)], f2 = f1 + f1;
        F[f] = (T(7) * f2 - f2) * T(1.0 / 12.0);
        sound = sound && isfinite(f1);
    }
    if (!sound) {
#pragma unroll
        for (int f = 0; f < 7; f++) F[f] = T(NAN);
    }
    store_flux<T, AXIS>(A, c, F);
}

template <class T, int AXIS>
__global__ void __launch_bounds__(kSweepNT) sweep_flat_kernel(const SweepArgs<T> A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Tile tile = A.tiles[blockIdx.x];
    tile.x &= 0xffffff;
    const PatchDev P = A.patches[tile.x];
    flat_body<T, AXIS>(A, tile, P, reinterpret_cast<T*>(smem_raw), threadIdx.x);
}

// One tile per block of one shape S, a launch for each shape's range of a tile
// table.  (One persistent launch over tiles of all shapes, its three bodies in
// one register allocation with 800 bytes of spills, took 18 ms per axis of 4 096
// patches against 13, and 1.55 ms for a 128^3 FP32 WENO-Z step's sweeps against
// 1.13; separately compiled, it also rounded differently.)
template <class T, int AXIS, int S, bool Z>
__global__ void __launch_bounds__(kSweepNT, kMinBlocks<T>) sweep_kernel_fixed(const SweepArgs<T> A) {
    constexpr int NC0 = nc_of(shape_ta(AXIS, S));
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sm = reinterpret_cast<T*>(smem_raw);
    Tile tile = A.tiles[blockIdx.x];
    tile.x &= 0xffffff;
    const PatchDev P = A.patches[tile.x];
    tile_body<T, AXIS, shape_ta(AXIS, S), NC0, Z>(A, tile, P, sm, threadIdx.x);
}

template <class T>
constexpr size_t tile_smem(int nc) {
    return sizeof(T) * (kNSlot * (size_t)nc + (size_t)kSlots<T> * kSweepNT);
}
template <class T, int AXIS, int S>
constexpr size_t smem_bytes_fixed() { return tile_smem<T>(nc_of(shape_ta(AXIS, S))); }

// f(axis, shape, z) over every fixed kernel
template <class T, int AX, int S, bool Z>
cudaError_t prepare_fixed() {
    return cudaFuncSetAttribute(sweep_kernel_fixed<T, AX, S, Z>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)smem_bytes_fixed<T, AX, S>());
}
template <class T, int AX, bool Z>
cudaError_t prepare_axis() {
    cudaError_t e = prepare_fixed<T, AX, 0, Z>();
    if (e == cudaSuccess) e = prepare_fixed<T, AX, 1, Z>();
    if (e == cudaSuccess) e = prepare_fixed<T, AX, 2, Z>();
    return e;
}
template <class T, bool Z, int S>
void launch_fixed_shape(int axis, const SweepArgs<T>& a, int ntiles, cudaStream_t s) {
    if (axis == 0) sweep_kernel_fixed<T, 0, S, Z><<<ntiles, kSweepNT, smem_bytes_fixed<T, 0, S>(), s>>>(a);
    else if (axis == 1) sweep_kernel_fixed<T, 1, S, Z><<<ntiles, kSweepNT, smem_bytes_fixed<T, 1, S>(), s>>>(a);
    else sweep_kernel_fixed<T, 2, S, Z><<<ntiles, kSweepNT, smem_bytes_fixed<T, 2, S>(), s>>>(a);
}

template <class T>
void launch_flat(int axis, const SweepArgs<T>& a, int ntiles, cudaStream_t s) {
    constexpr size_t smem = sizeof(T) * kNSlot * kSweepNT;
    static_assert(smem <= 48 * 1024, "within the default limit");
    if (axis == 0) sweep_flat_kernel<T, 0><<<ntiles, kSweepNT, smem, s>>>(a);
    else if (axis == 1) sweep_flat_kernel<T, 1><<<ntiles, kSweepNT, smem, s>>>(a);
    else sweep_flat_kernel<T, 2><<<ntiles, kSweepNT, smem, s>>>(a);
}

template <class T, bool Z>
cudaError_t launch_sweep_w(int axis, const SweepArgs<T>& a, cudaStream_t s) {
    SweepArgs<T> b = a;
    if (a.split[0]) launch_fixed_shape<T, Z, 0>(axis, b, a.split[0], s);
    b.tiles += a.split[0];
    if (a.split[1]) launch_fixed_shape<T, Z, 1>(axis, b, a.split[1], s);
    b.tiles += a.split[1];
    if (a.split[2]) launch_fixed_shape<T, Z, 2>(axis, b, a.split[2], s);
    b.tiles += a.split[2];
    if (a.split[3]) launch_flat<T>(axis, b, a.split[3], s);
    return cudaGetLastError();
}

}  // namespace

template <class T>
cudaError_t prepare_sweep_kernels() {
    cudaError_t e = prepare_axis<T, 0, false>();
    if (e == cudaSuccess) e = prepare_axis<T, 1, false>();
    if (e == cudaSuccess) e = prepare_axis<T, 2, false>();
    if (e == cudaSuccess) e = prepare_axis<T, 0, true>();
    if (e == cudaSuccess) e = prepare_axis<T, 1, true>();
    if (e == cudaSuccess) e = prepare_axis<T, 2, true>();
    return e;
}

template <class T>
cudaError_t launch_sweep(int axis, const SweepArgs<T>& a, cudaStream_t s) {
    return a.zweights ? launch_sweep_w<T, true>(axis, a, s) : launch_sweep_w<T, false>(axis, a, s);
}

}  // namespace wb
