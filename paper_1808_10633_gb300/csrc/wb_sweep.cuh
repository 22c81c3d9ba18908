// wb_sweep.cuh -- characteristic WENO5 flux sweeps (Donnert et al. 2018,
// Sec. 2.1 eq. FWENO; Sec. 2.2 dimension-by-dimension sweeps).  Included by
// wb_sweep_f32.cu (compiled with fast single-precision division and square
// root) and wb_sweep_f64.cu, which instantiate it for float and double.
//
// One thread computes the numerical flux through one interface.  A block
// owns a 2-D slab of interfaces: TA along the sweep axis times TP pencils.
// The TA+5 cells each pencil needs (3 below, 2 above the slab) are staged
// once in shared memory with everything the interface step reads per cell:
// the rotated conserved 7-vector, its physical flux, the seven |lambda| and
// the primitives used by the interface average.  The sweep never moves the
// grid ("rotation" of Sec. 2.2 is an index mapping): for the x sweep the
// thread's x index walks the axis, for y and z the thread's x index walks
// the pencils, so every global load and store is x-contiguous.
//
// Per interface (cells i-2..i+3 of the stencil):
//   1. interface state = mean of the primitives of cells i, i+1;
//   2. closed-form 7-wave eigensystem (Roe-Balsara normalisation) at it;
//   3. projection of the stencil's five U and F differences on the left
//      eigenvectors, done as (dW/dU) x followed by the sparse left vectors; the
//      Alfven and entropy fields wait in shared memory while the fast and slow
//      ones are reconstructed (FP32 here, U and F in one packed pair; FP64 in
//      wb_sweep_js.cuh; the tensor-core learned sweep projects the six cells,
//      in two groups of fields);
//   4. local Lax-Friedrichs splitting, alpha_s = max |lambda_s| over the
//      stencil and the interface state;
//   5. WENO5-JS weights and phi_N for both split fluxes;
//   6. back-projection (dU/dW applied to the primitive right vectors) plus
//      the fourth-order central flux (-F_{i-1} + 7F_i + 7F_{i+1} - F_{i+2})/12.
// The flux is written in global component order (rho, mx, my, mz, E,
// B_t1, B_t2) to the face array of the lower face of cell i+1.
#pragma once
#include "../../include/wombat_gb300.h"
#include "wb_internal.h"
#include "wb_math.cuh"

namespace wb {
namespace {

// ---- shared-memory slots per staged cell ----------------------------------
enum : int {
    SU = 0,      // U7: rho, m_n, m_t1, m_t2, B_t1, B_t2, E        (0..6)
    SF = 7,      // F7 in the same order                           (7..13)
    SL = 14,     // |lambda_s|, s = 0..6                           (14..20)
    SP_U = 21, SP_V1, SP_V2, SP_BN, SP_P,   // primitives for the mean
    kNSlot = 26
};
// Place of U_f and F_f of staged cell idx.  FP32 keeps them side by side: the
// projection works on (U, F) pairs, one 8-byte load each; FP64 by field, the
// mass flux F_0 being U_1 = m_n.
template <class T> __device__ __forceinline__ constexpr int at_u(int f, int nc, int idx) {
    return sizeof(T) == 4 ? 2 * (f * nc + idx) : (SU + f) * nc + idx;
}
template <class T> __device__ __forceinline__ constexpr int at_f(int f, int nc, int idx) {
    return sizeof(T) == 4 ? 2 * (f * nc + idx) + 1 : (f == 0 ? SU + 1 : SF + f) * nc + idx;
}

template <class T> __device__ __forceinline__ T tmax(T a, T b) { return a > b ? a : b; }
// |a| by clearing the sign bit (no floating-point compare on the FP64 pipe)
__device__ __forceinline__ float tabs(float a) { return fabsf(a); }
__device__ __forceinline__ double tabs(double a) { return fabs(a); }
// max of two values >= 0: for non-negative IEEE values the bit patterns
// order like the values, so FP64 takes an integer max, off the FP64 pipe
__device__ __forceinline__ float tmax_nonneg(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double tmax_nonneg(double a, double b) {
    return __longlong_as_double(max(__double_as_longlong(a), __double_as_longlong(b)));
}

__device__ __forceinline__ int wrap(int v, int n) {
    int r = v % n;
    return r < 0 ? r + n : r;
}

// The same for v within one period of [0, n) in nearly every call (a tile's
// halo): no division then.
__device__ __forceinline__ int wrap_near(int v, int n) {
    if (v < 0) v += n;
    else if (v >= n) v -= n;
    return (unsigned)v < (unsigned)n ? v : wrap(v, n);
}

// Sec. 2.1: phi_N(a,b,c,d) = 1/3 w0 (a-2b+c) + 1/6 (w2-1/2)(b-2c+d) with
// IS_0..2 as printed, alpha_k = d_k/(eps+IS_k)^2, d = (1, 6, 3), eps = 1e-6.
// The weights depend only on the ratios of the eps + IS_k, so each is formed
// divided by three, (13/3) t^2 + t'^2 + eps/3: one multiply and two fused
// multiply-adds, the eps folded in.
// eps3 = eps / 3; phi_N(s a, s b, s c, s d) with s^2 eps3 is s phi_N(a, b, c, d).
constexpr float kEps3f = 1e-6f / 3.0f;
__device__ __forceinline__ float phi_n(float a, float b, float c, float d, float eps3 = kEps3f) {
    const float k13 = 13.0f / 3.0f;
    const float t0 = a - b, t1 = a - 3.0f * b;
    const float t2 = b - c, t3 = b + c;
    const float t4 = c - d, t5 = 3.0f * c - d;
    const float e0 = fmaf(k13 * t0, t0, fmaf(t1, t1, eps3));
    const float e1 = fmaf(k13 * t2, t2, fmaf(t3, t3, eps3));
    const float e2 = fmaf(k13 * t4, t4, fmaf(t5, t5, eps3));
    // reciprocals keep the FP32 range: (eps+IS)^2 products could overflow
    float a0 = 1.0f / (e0 * e0), a1 = 6.0f / (e1 * e1), a2 = 3.0f / (e2 * e2);
    float r = 1.0f / (a0 + a1 + a2);
    float w0 = a0 * r, w2 = a2 * r;
    return w0 * (a - 2.0f * b + c) * (1.0f / 3.0f) + (w2 - 0.5f) * (b - 2.0f * c + d) * (1.0f / 6.0f);
}

// phi_N of the minus side (lane x) and the plus side (lane y) of one field
// at once, in packed FP32 pairs (one instruction for both lanes); each lane
// computes what phi_n(float) does, with the products and sums spelled as
// fused multiply-adds.
__device__ __forceinline__ float2 splat2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 phi_n2(float2 a, float2 b, float2 c, float2 d, float eps3f = kEps3f) {
    // (eps + IS_k) / 3 as in phi_n
    const float2 k13 = splat2(13.0f / 3.0f), eps3 = splat2(eps3f);
    const float2 t0 = __ffma2_rn(b, splat2(-1.0f), a), t1 = __ffma2_rn(b, splat2(-3.0f), a);
    const float2 t2 = __ffma2_rn(c, splat2(-1.0f), b), t3 = __fadd2_rn(b, c);
    // t5 enters squared: d - 3c serves for 3c - d
    const float2 t4 = __ffma2_rn(d, splat2(-1.0f), c), t5 = __ffma2_rn(c, splat2(-3.0f), d);
    float2 e0 = __ffma2_rn(__fmul2_rn(t0, k13), t0, __ffma2_rn(t1, t1, eps3));
    float2 e1 = __ffma2_rn(__fmul2_rn(t2, k13), t2, __ffma2_rn(t3, t3, eps3));
    float2 e2 = __ffma2_rn(__fmul2_rn(t4, k13), t4, __ffma2_rn(t5, t5, eps3));
    e0 = __fmul2_rn(e0, e0);
    e1 = __fmul2_rn(e1, e1);
    e2 = __fmul2_rn(e2, e2);
    const float2 a0 = make_float2(1.0f / e0.x, 1.0f / e0.y);
    const float2 a1 = __fmul2_rn(make_float2(1.0f / e1.x, 1.0f / e1.y), splat2(6.0f));
    const float2 a2 = __fmul2_rn(make_float2(1.0f / e2.x, 1.0f / e2.y), splat2(3.0f));
    const float2 sum = __fadd2_rn(__fadd2_rn(a0, a1), a2);
    const float2 r = make_float2(1.0f / sum.x, 1.0f / sum.y);
    const float2 w0 = __fmul2_rn(a0, r);
    const float2 h2 = __ffma2_rn(a2, r, splat2(-0.5f));
    const float2 p = __ffma2_rn(b, splat2(-2.0f), __fadd2_rn(a, c));
    const float2 q = __ffma2_rn(c, splat2(-2.0f), __fadd2_rn(b, d));
    return __ffma2_rn(__fmul2_rn(w0, splat2(1.0f / 3.0f)), p, __fmul2_rn(__fmul2_rn(h2, splat2(1.0f / 6.0f)), q));
}

// Interface eigen-structure: everything the projection and back-projection
// need, with 1/rho and (gamma-1) folded into the left coefficients.
template <class T>
struct Eig {
    T rho, u, v1, v2, hv2;
    T bm;                        // B_perp along beta: b1 x1 + b2 x2 = bm (be1 x1 + be2 x2)
    T be1, be2;
    T cf, cs, ca;
    T Af, Bf, Cf, Df, As, Bs, Cs, Ds, Aa, Ba, Ee;
};

// Coefficients only the back-projection needs; parked in shared memory (one
// slot per thread) while the WENO step runs, to keep registers for it.
enum : int { BP_ALF = 0, BP_ALS, BP_AFCF, BP_ASCS, BP_ASR, BP_SSR, BP_RA2, BP_IGM1, kNBack = 8 };
// Per-thread slots after the back-projection ones where the Alfven/entropy
// split differences (3 fields x 2 sides x the steps the weights read) wait
// while the fast/slow group is reconstructed, when each stencil vector is
// projected only once.
constexpr int thread_slots(int steps) { return kNBack + 6 * steps; }

// |lambda_s| of the interface state, s = 0..6 (u-cf, u-ca, u-cs, u, u+cs,
// u+ca, u+cf)
template <class T>
__device__ __forceinline__ T lam_avg(const Eig<T>& e, int s) {
    const T c = (s == 0 || s == 6) ? e.cf : (s == 1 || s == 5) ? e.ca : (s == 2 || s == 4) ? e.cs : T(0);
    return tabs(s < 3 ? e.u - c : e.u + c);
}

// beta and (alpha_f, alpha_s) with the degeneracy rules, from 1/rho, a^2 and
// ca^2; FP64 throughout.
__device__ __forceinline__ void degenerate_rules(double rinv, double a2, double ca2, double bn, double b1, double b2,
                                                 double& be1, double& be2, double& alf, double& als,
                                                 double& cf2o) {
    const double bp2 = b1 * b1 + b2 * b2;
    const double bt2 = bn * bn + bp2;
    if (bp2 > 1e-24 * (bt2 > 1.0 ? bt2 : 1.0)) {
        const double ibp = rsq_root(bp2);
        be1 = b1 * ibp;
        be2 = b2 * ibp;
    } else {
        be1 = be2 = 0.70710678118654752440;
    }
    // D = cf^2 - cs^2 from a sum of non-negative terms (t = B_perp^2 / rho),
    // cf^2 from the sum of the roots: no cancellation near B_perp -> 0 or the
    // triple point.  alpha_f^2 = x / D, alpha_s^2 = y / D with x = a^2 - cs^2,
    // y = cf^2 - a^2: the larger of x, y from x + y = D and the smaller from
    // x y = a^2 t, so the vanishing weight goes to zero with B_perp
    const double t = bp2 * rinv;
    // D and 1/D from one reciprocal square root (D = 0 kept exact)
    const double dA = a2 - ca2, sA = a2 + ca2;
    const double D2 = fma(dA, dA, t * fma(2.0, sA, t));
    const double iD = D2 > 0.0 ? rsq_root(D2) : 0.0;
    const double D = D2 * iD;
    cf2o = 0.5 * ((sA + t) + D);
    if (D <= 1e-12 * (a2 + bt2 * rinv)) {
        if (a2 >= ca2) { alf = 1.0; als = 0.0; } else { alf = 0.0; als = 1.0; }
    } else {
        double x = 0.5 * (D + dA - t);
        double y = 0.5 * (D - dA + t);
        const bool fast = x >= y;
        const double small = a2 * t * recip(fast ? x : y);
        if (fast) y = small;
        else x = small;
        alf = x > 0.0 ? sq_root(x * iD) : 0.0;
        als = y > 0.0 ? sq_root(y * iD) : 0.0;
    }
}

template <class T>
__device__ __forceinline__ void eigen(T rho, T u, T v1, T v2, T bn, T b1, T b2, T p, T gamma,
                                      Eig<T>& e, T* __restrict__ bp, int bstride) {
    const T isr = rsq_root(rho), rinv = isr * isr;     // 1/sqrt(rho), 1/rho
    const T a2 = gamma * p * rinv;
    const T ca2 = bn * bn * rinv;
    T cf2, be1, be2, alf, als;
    if constexpr (sizeof(T) == 8) {
        degenerate_rules(rinv, a2, ca2, bn, b1, b2, be1, be2, alf, als, cf2);
    } else {
        // FP32 bulk; the normalisation near B_perp -> 0 and near cf = cs
        // (fast/slow/Alfven coincidence) is taken in FP64.
        const T bp2 = b1 * b1 + b2 * b2;
        const T bt2 = bn * bn + bp2;
        const T b2r = bt2 * rinv;
        const T t = bp2 * rinv;
        const T D2 = (a2 - ca2) * (a2 - ca2) + t * (T(2) * (a2 + ca2) + t);
        const T iD = D2 > T(0) ? rsq_root(D2) : T(0);
        const T D = D2 * iD;
        cf2 = T(0.5) * ((a2 + ca2 + t) + D);
        const bool near_bperp = !(bp2 > T(1e-6) * bt2);
        const bool near_triple = !(D > T(1e-3) * (a2 + b2r));
        if (near_bperp || near_triple) {
            double dbe1, dbe2, dalf, dals, dcf2;
            const double dr = recip(double(rho));
            degenerate_rules(dr, double(gamma) * double(p) * dr, double(bn) * double(bn) * dr, bn, b1, b2, dbe1, dbe2,
                             dalf, dals, dcf2);
            be1 = T(dbe1); be2 = T(dbe2); alf = T(dalf); als = T(dals);
            cf2 = T(dcf2);
        } else {
            const T ibp = rsq_root(bp2);
            be1 = b1 * ibp;
            be2 = b2 * ibp;
            T x = T(0.5) * (D + (a2 - ca2) - t), y = T(0.5) * (D - (a2 - ca2) + t);
            if (x >= y) y = a2 * t / x;
            else x = a2 * t / y;
            alf = sq_root(tmax(x * iD, T(0)));
            als = sq_root(tmax(y * iD, T(0)));
        }
    }
    // sqrt(rho), sqrt(a^2), cf and their reciprocals from one reciprocal
    // square root each (isr above); ca = |B_n| / sqrt(rho) and, from the
    // product of the roots cf^2 cs^2 = a^2 ca^2, cs = a ca / cf
    const T ia = rsq_root(a2);
    const T sr = rho * isr, a = a2 * ia;
    const T icf = cf2 > T(0) ? rsq_root(cf2) : T(0);
    const T cf = cf2 * icf, ca = tabs(bn) * isr;
    const T cs = a * ca * icf, cs2 = cs * cs;
    const T S = bn >= T(0) ? T(1) : T(-1);
    const T gm1 = gamma - T(1);
    const T X = alf * alf * cf2 + als * als * cs2;
    const T hXr = T(0.5) * recip(X) * rinv;
    const T hia = T(0.5) * ia * isr;         // 1 / (2 a sqrt(rho))
    const T Ee = gm1 * ia * ia;              // (gamma-1) / a^2
    const T hgp = T(0.5) * Ee * rinv;        // (gamma-1) / (2 rho a^2)
    e.rho = rho; e.u = u; e.v1 = v1; e.v2 = v2;
    e.bm = b1 * be1 + b2 * be2;
    e.hv2 = T(0.5) * (u * u + v1 * v1 + v2 * v2);
    e.be1 = be1; e.be2 = be2;
    e.cf = cf; e.cs = cs; e.ca = ca;
    bp[BP_ALF * bstride] = alf;
    bp[BP_ALS * bstride] = als;
    bp[BP_AFCF * bstride] = alf * cf;
    bp[BP_ASCS * bstride] = als * cs;
    bp[BP_ASR * bstride] = a * sr;
    bp[BP_SSR * bstride] = S * sr;
    bp[BP_RA2 * bstride] = rho * a2;
    bp[BP_IGM1 * bstride] = T(1) / gm1;
    e.Af = alf * cf * hXr;
    e.Bf = -als * cs * S * hXr;
    e.Cf = als * hia;
    e.Df = alf * hgp;
    e.As = als * cs * hXr;
    e.Bs = alf * cf * S * hXr;
    e.Cs = -alf * hia;
    e.Ds = als * hgp;
    e.Aa = T(0.5) * rinv;
    e.Ba = T(0.5) * S * isr;
    e.Ee = Ee;
}

// ---- staging ---------------------------------------------------------------
// Per cell: cell B from the faces, rotation into the (n, t1, t2) frame,
// primitives, the physical flux along n, the seven |lambda| and, in the x
// sweep, the cell value of -v x B for the constrained-transport EMFs.  The
// loads of all cells a thread stages are issued first (load_cell), the
// derived quantities computed afterwards (derive_cell), so one global-load
// latency covers a thread's whole share of the tile.
template <class T>
struct RawCell {
    T rho, mx, my, mz, E, bx0, bx1, by0, by1, bz0, bz1;
};

// Loads of one staged cell: the cell values and its three upper faces.
template <class T>
__device__ __forceinline__ void load_cell_at(const SweepArgs<T>& A, long long c, long long cxp,
                                             long long cyp, long long czp, RawCell<T>& r) {
    const long long N = A.ncells;
    const T* __restrict__ q = A.src;
    c = chk(c, N, A.flag);
    cxp = chk(cxp, N, A.flag);
    cyp = chk(cyp, N, A.flag);
    czp = chk(czp, N, A.flag);
    r.rho = q[c]; r.mx = q[N + c]; r.my = q[2 * N + c]; r.mz = q[3 * N + c]; r.E = q[4 * N + c];
    r.bx0 = q[5 * N + c]; r.bx1 = q[5 * N + cxp];
    r.by0 = q[6 * N + c]; r.by1 = q[6 * N + cyp];
    r.bz0 = q[7 * N + c]; r.bz1 = q[7 * N + czp];
}

// Cell (i, j, k) of a periodic patch P, all three indices inside it.
template <class T>
__device__ __forceinline__ void load_cell(const SweepArgs<T>& A, const PatchDev& P, int i, int j,
                                          int k, RawCell<T>& r, long long& c) {
    c = P.off + ((long long)k * P.ny + j) * P.nx + i;
    const int ip = (i + 1 == P.nx) ? 0 : i + 1;
    const int jp = (j + 1 == P.ny) ? 0 : j + 1;
    const int kp = (k + 1 == P.nz) ? 0 : k + 1;
    load_cell_at(A, c, c + (ip - i), c + (long long)(jp - j) * P.nx,
                 c + (long long)(kp - k) * P.nx * P.ny, r);
}

// Pencil tp of a tile: the pencils of a patch are numbered along the pencil
// axis and then along the third, and a tile takes consecutive ones from (tile.z,
// tile.w) on, past the end of a row into the next.  cp: place along the pencil
// axis (of np), w: along the third.
__device__ __forceinline__ void tile_pencil(const Tile& tile, int tp, int np, int& cp, int& w) {
    cp = tile.z + tp;
    w = tile.w;
    if (cp >= np) {
        cp -= np;
        w++;
        if (cp >= np) {                // rows shorter than the tile is wide
            const int r = cp / np;
            cp -= r * np;
            w += r;
        }
    }
}

// Cell of the patch at place ia along the sweep axis of pencil (ip, w).
template <int AXIS>
__device__ __forceinline__ int tile_cell(const PatchDev& P, int ia, int ip, int w) {
    const int i = AXIS == 0 ? ia : ip, j = AXIS == 0 ? ip : (AXIS == 1 ? ia : w), k = AXIS == 2 ? ia : w;
    return (k * P.ny + j) * P.nx + i;
}

// Cell (i, j, k) of a tile's patch as the tile meets it: outside along the
// sweep axis where the stencil reaches past the patch's end (tab: its links, of
// a linked grid).  Most cells lie inside with
// their three upper neighbours and need no wrap and no link.
template <class T, int AXIS>
__device__ __forceinline__ void load_cell_tile(const SweepArgs<T>& A, const LinkTab& tab, const PatchDev& P, int i,
                                               int j, int k, RawCell<T>& r, long long& c) {
    long long cx, cy, cz;
    const int nxy = P.nx * P.ny;
    if ((unsigned)i < (unsigned)(P.nx - 1) && (unsigned)j < (unsigned)(P.ny - 1) && (unsigned)k < (unsigned)(P.nz - 1)) {
        c = P.off + (k * P.ny + j) * P.nx + i;
        cx = c + 1;
        cy = c + P.nx;
        cz = c + nxy;
    } else if (A.links) {
        // beyond the patch's end as inside it, the upper neighbours are a fixed
        // distance away unless the cell is its patch's last (160^3 in 64 bricks,
        // sweeps of a step: 2.84 -> 2.66 ms)
        int qi = i, qj = j, qk = k, qx, qy, qz;
        c = tab.find(P, qi, qj, qk, qx, qy, qz);
        cx = qi + 1 < qx ? c + 1 : tab.at(P, i + 1, j, k);
        cy = qj + 1 < qy ? c + qx : tab.at(P, i, j + 1, k);
        cz = qk + 1 < qz ? c + (long long)qx * qy : tab.at(P, i, j, k + 1);
    } else {
        if (AXIS == 0) i = wrap_near(i, P.nx);
        else if (AXIS == 1) j = wrap_near(j, P.ny);
        else k = wrap_near(k, P.nz);
        c = P.off + (k * P.ny + j) * P.nx + i;
        cx = c + (i + 1 == P.nx ? 1 - P.nx : 1);
        cy = c + (j + 1 == P.ny ? P.nx - nxy : P.nx);
        cz = c + (k + 1 == P.nz ? (long long)nxy * (1 - P.nz) : nxy);
    }
    load_cell_at(A, c, cx, cy, cz, r);
}

template <class T, int AXIS>
__device__ __forceinline__ void derive_cell(const SweepArgs<T>& A, const RawCell<T>& r, long long c,
                                            T* __restrict__ sm, int nc, int idx, bool write_er) {
    const long long N = A.ncells;
    idx = (int)chk(idx, nc, A.flag);
    const T rho = r.rho, E = r.E;
    const T Bx = T(0.5) * (r.bx0 + r.bx1);
    const T By = T(0.5) * (r.by0 + r.by1);
    const T Bz = T(0.5) * (r.bz0 + r.bz1);
    const T mx = r.mx, my = r.my, mz = r.mz;
    T mn, m1, m2, bn, b1, b2;
    if (AXIS == 0) { mn = mx; m1 = my; m2 = mz; bn = Bx; b1 = By; b2 = Bz; }
    else if (AXIS == 1) { mn = my; m1 = mz; m2 = mx; bn = By; b1 = Bz; b2 = Bx; }
    else { mn = mz; m1 = mx; m2 = my; bn = Bz; b1 = Bx; b2 = By; }
    const T g = T(A.gamma);
    const T isr = rsq_root(rho), rinv = isr * isr;
    const T u = mn * rinv, v1 = m1 * rinv, v2 = m2 * rinv;
    const T bb = bn * bn + b1 * b1 + b2 * b2;
    const T kin = T(0.5) * (mn * u + m1 * v1 + m2 * v2);
    const T p = (g - T(1)) * (E - kin - T(0.5) * bb);
    const T pt = p + T(0.5) * bb;
    const T vb = u * bn + v1 * b1 + v2 * b2;
    const T U[7] = {rho, mn, m1, m2, b1, b2, E};
    const T F[7] = {mn, mn * u + pt - bn * bn, m1 * u - bn * b1, m2 * u - bn * b2, u * b1 - v1 * bn, u * b2 - v2 * bn,
                    (E + pt) * u - bn * vb};
#pragma unroll
    for (int f = 0; f < 7; f++) {
        if constexpr (sizeof(T) == 4) {
            *reinterpret_cast<float2*>(sm + at_u<T>(f, nc, idx)) = make_float2(U[f], F[f]);
        } else {
            sm[at_u<T>(f, nc, idx)] = U[f];
            if (f > 0) sm[at_f<T>(f, nc, idx)] = F[f];
        }
    }
    const T a2 = g * p * rinv;
    const T ca2 = bn * bn * rinv;
    // fast and slow speeds without cancellation: D = cf^2 - cs^2 from a sum
    // of non-negative terms (t = B_perp^2 / rho), cf^2 from the sum of the
    // roots and cs^2 = a^2 ca^2 / cf^2 from their product
    const T t = (b1 * b1 + b2 * b2) * rinv;
    const T D = sq_root((a2 - ca2) * (a2 - ca2) + t * (T(2) * (a2 + ca2) + t));
    const T cf2 = T(0.5) * ((a2 + ca2 + t) + D);
    const T icf = cf2 > T(0) ? rsq_root(cf2) : T(0);
    const T cf = cf2 * icf;
    const T ca = tabs(bn) * isr;
    const T cs = sq_root(a2) * ca * icf;       // sqrt(a^2 ca^2 / cf^2)
    sm[(SL + 0) * nc + idx] = tabs(u - cf);
    sm[(SL + 1) * nc + idx] = tabs(u - ca);
    sm[(SL + 2) * nc + idx] = tabs(u - cs);
    sm[(SL + 3) * nc + idx] = tabs(u);
    sm[(SL + 4) * nc + idx] = tabs(u + cs);
    sm[(SL + 5) * nc + idx] = tabs(u + ca);
    sm[(SL + 6) * nc + idx] = tabs(u + cf);
    sm[SP_U * nc + idx] = u;
    sm[SP_V1 * nc + idx] = v1;
    sm[SP_V2 * nc + idx] = v2;
    sm[SP_BN * nc + idx] = bn;
    sm[SP_P * nc + idx] = p;
    if (AXIS == 0 && write_er) {
        // -v x B in the global frame (x sweep: u = vx, v1 = vy, v2 = vz)
        c = chk(c, N, A.flag);
        A.er[c] = v2 * b1 - v1 * b2;
        A.er[N + c] = u * b2 - v2 * bn;
        A.er[2 * N + c] = v1 * bn - u * b1;
    }
}

// ---- one interface ----------------------------------------------------------
template <class T>
__device__ __forceinline__ void load7(const T* __restrict__ sm, int nc, int base, int idx, T (&x)[7]) {
#pragma unroll
    for (int f = 0; f < 7; f++) x[f] = sm[base == SF ? at_f<T>(f, nc, idx) : at_u<T>(f, nc, idx)];
}

// first projection group: fast-, slow-, slow+, fast+ (s = 0, 2, 4, 6)
template <class T>
__device__ __forceinline__ void project_fs(const Eig<T>& e, const T (&x)[7], T (&o)[4]) {
    const T du = x[1] - e.u * x[0];
    const T dv1 = x[2] - e.v1 * x[0];
    const T dv2 = x[3] - e.v2 * x[0];
    const T vpar = e.be1 * dv1 + e.be2 * dv2;
    const T bpar = e.be1 * x[4] + e.be2 * x[5];
    const T P = x[6] + e.hv2 * x[0] - e.u * x[1] - e.v1 * x[2] - e.v2 * x[3] - e.bm * bpar;
    const T tf1 = e.Af * du + e.Bf * vpar, tf2 = e.Cf * bpar + e.Df * P;
    const T ts1 = e.As * du + e.Bs * vpar, ts2 = e.Cs * bpar + e.Ds * P;
    o[0] = tf2 - tf1;
    o[1] = ts2 - ts1;
    o[2] = ts2 + ts1;
    o[3] = tf2 + tf1;
}

// second projection group: Alfven-, entropy, Alfven+ (s = 1, 3, 5)
template <class T>
__device__ __forceinline__ void project_ae(const Eig<T>& e, const T (&x)[7], T (&o)[3]) {
    const T dv1 = x[2] - e.v1 * x[0];
    const T dv2 = x[3] - e.v2 * x[0];
    const T bpar = e.be1 * x[4] + e.be2 * x[5];
    const T P = x[6] + e.hv2 * x[0] - e.u * x[1] - e.v1 * x[2] - e.v2 * x[3] - e.bm * bpar;
    const T vperp = e.be1 * dv2 - e.be2 * dv1;
    const T bperp = e.be1 * x[5] - e.be2 * x[4];
    const T t1 = e.Aa * vperp, t2 = e.Ba * bperp;
    o[0] = t1 + t2;
    o[1] = x[0] - e.Ee * P;
    o[2] = t1 - t2;
}

// All seven fields of a (U difference, F difference) pair in packed FP32 lanes:
// the same coefficients act on both, one instruction for the two.
__device__ __forceinline__ void project_all2(const Eig<float>& e, const float2 (&x)[7], float2 (&o4)[4],
                                             float2 (&o3)[3]) {
    const float2 du = __ffma2_rn(splat2(-e.u), x[0], x[1]);
    const float2 dv1 = __ffma2_rn(splat2(-e.v1), x[0], x[2]);
    const float2 dv2 = __ffma2_rn(splat2(-e.v2), x[0], x[3]);
    float2 P = __ffma2_rn(splat2(e.hv2), x[0], x[6]);
    P = __ffma2_rn(splat2(-e.u), x[1], P);
    P = __ffma2_rn(splat2(-e.v1), x[2], P);
    P = __ffma2_rn(splat2(-e.v2), x[3], P);
    const float2 vpar = __ffma2_rn(splat2(e.be1), dv1, __fmul2_rn(splat2(e.be2), dv2));
    const float2 bpar = __ffma2_rn(splat2(e.be1), x[4], __fmul2_rn(splat2(e.be2), x[5]));
    P = __ffma2_rn(splat2(-e.bm), bpar, P);
    const float2 tf1 = __ffma2_rn(splat2(e.Af), du, __fmul2_rn(splat2(e.Bf), vpar));
    const float2 tf2 = __ffma2_rn(splat2(e.Cf), bpar, __fmul2_rn(splat2(e.Df), P));
    const float2 ts1 = __ffma2_rn(splat2(e.As), du, __fmul2_rn(splat2(e.Bs), vpar));
    const float2 ts2 = __ffma2_rn(splat2(e.Cs), bpar, __fmul2_rn(splat2(e.Ds), P));
    o4[0] = __ffma2_rn(tf1, splat2(-1.0f), tf2);
    o4[1] = __ffma2_rn(ts1, splat2(-1.0f), ts2);
    o4[2] = __fadd2_rn(ts2, ts1);
    o4[3] = __fadd2_rn(tf2, tf1);
    const float2 vperp = __ffma2_rn(splat2(e.be1), dv2, __fmul2_rn(splat2(-e.be2), dv1));
    const float2 bperp = __ffma2_rn(splat2(e.be1), x[5], __fmul2_rn(splat2(-e.be2), x[4]));
    const float2 t1 = __fmul2_rn(splat2(e.Aa), vperp), t2 = __fmul2_rn(splat2(e.Ba), bperp);
    o3[0] = __fadd2_rn(t1, t2);
    o3[1] = __ffma2_rn(splat2(-e.Ee), P, x[0]);
    o3[2] = __ffma2_rn(t2, splat2(-1.0f), t1);
}

// single field pair projections (fields processed two at a time keep the
// projected stencil small): G = 0 fast-/fast+ (s = 0, 6), 1 slow-/slow+
// (s = 2, 4), 2 Alfven-/Alfven+ (s = 1, 5), 3 entropy (s = 3).
template <int G, class T>
__device__ __forceinline__ void project_pair(const Eig<T>& e, const T (&x)[7], T (&o)[2]) {
    const T dv1 = x[2] - e.v1 * x[0];
    const T dv2 = x[3] - e.v2 * x[0];
    if constexpr (G == 2) {
        const T t1 = e.Aa * (e.be1 * dv2 - e.be2 * dv1);
        const T t2 = e.Ba * (e.be1 * x[5] - e.be2 * x[4]);
        o[0] = t1 + t2;
        o[1] = t1 - t2;
    } else {
        const T bpar = e.be1 * x[4] + e.be2 * x[5];
        const T P = x[6] + e.hv2 * x[0] - e.u * x[1] - e.v1 * x[2] - e.v2 * x[3] - e.bm * bpar;
        if constexpr (G == 3) {
            o[0] = x[0] - e.Ee * P;
            o[1] = o[0];
        } else {
            const T du = x[1] - e.u * x[0];
            const T vpar = e.be1 * dv1 + e.be2 * dv2;
            const T t1 = G == 0 ? e.Af * du + e.Bf * vpar : e.As * du + e.Bs * vpar;
            const T t2 = G == 0 ? e.Cf * bpar + e.Df * P : e.Cs * bpar + e.Ds * P;
            o[0] = t2 - t1;
            o[1] = t2 + t1;
        }
    }
}

template <class T>
__device__ __forceinline__ T lf_speed(const T* __restrict__ sm, int nc, const int (&id)[6],
                                      int s, T lam_avg) {
    T al = lam_avg;
#pragma unroll
    for (int m = 0; m < 6; m++) al = tmax_nonneg(al, sm[(SL + s) * nc + id[m]]);
    return al;
}

template <class T, class Wt, bool PARK = false>
__device__ __forceinline__ void interface_flux(const T* __restrict__ sm, int nc, const int (&id)[6],
                                               T gamma, T* __restrict__ bp, int bstride, Wt& wt,
                                               T (&out)[7]) {
    // 1-2. interface state and eigen-structure
    Eig<T> e;
    {
        const int l = id[2], r = id[3];
        const T h = T(0.5);
        eigen<T>(h * (sm[at_u<T>(0, nc, l)] + sm[at_u<T>(0, nc, r)]),
                 h * (sm[SP_U * nc + l] + sm[SP_U * nc + r]),
                 h * (sm[SP_V1 * nc + l] + sm[SP_V1 * nc + r]),
                 h * (sm[SP_V2 * nc + l] + sm[SP_V2 * nc + r]),
                 h * (sm[SP_BN * nc + l] + sm[SP_BN * nc + r]),
                 h * (sm[at_u<T>(4, nc, l)] + sm[at_u<T>(4, nc, r)]),
                 h * (sm[at_u<T>(5, nc, l)] + sm[at_u<T>(5, nc, r)]),
                 h * (sm[SP_P * nc + l] + sm[SP_P * nc + r]), gamma, e, bp, bstride);
    }
    T corr[7];
    if constexpr (PARK) {
        // 3. the five differences of the stencil's U and F, each projected once
        // onto all seven fields; the Alfven/entropy values wait in this
        // thread's shared-memory slots
        constexpr bool kSplit = Wt::kSplit;
        constexpr int K = kSplit ? 4 : 5;      // values per field, twice
        T* park = bp + kNBack * bstride;
        T fa[4][K], fb[4][K];
        // 4. kSplit: the projected differences are split at once, 2 D+- = l dF
        // +- alpha l dU (steps 0..3 and 1..4 of the two sides), which keeps
        // eight values per field instead of ten; the learned weights read all
        // five steps of both sides and split them themselves
        T al[7];
        if constexpr (kSplit)
#pragma unroll
            for (int s = 0; s < 7; s++) al[s] = lf_speed(sm, nc, id, s, lam_avg(e, s));
        // U and F differences of a stencil step as one packed pair
        float2 p0[7];
#pragma unroll
        for (int f = 0; f < 7; f++) p0[f] = *reinterpret_cast<const float2*>(sm + at_u<T>(f, nc, id[0]));
#pragma unroll
        for (int m = 0; m < 5; m++) {
            float2 p1[7], x[7], o4[4], o3[3];
#pragma unroll
            for (int f = 0; f < 7; f++) {
                p1[f] = *reinterpret_cast<const float2*>(sm + at_u<T>(f, nc, id[m + 1]));
                x[f] = __ffma2_rn(p0[f], splat2(-1.0f), p1[f]);
            }
            project_all2(e, x, o4, o3);
            const int lo = kSplit ? m - 1 : m;
#pragma unroll
            for (int f = 0; f < 4; f++) {
                if (m < K) fa[f][m] = kSplit ? fmaf(al[2 * f], o4[f].x, o4[f].y) : o4[f].x;
                if (lo >= 0) fb[f][lo] = kSplit ? fmaf(-al[2 * f], o4[f].x, o4[f].y) : o4[f].y;
            }
#pragma unroll
            for (int f = 0; f < 3; f++) {
                if (m < K) park[(2 * f * K + m) * bstride] = kSplit ? fmaf(al[2 * f + 1], o3[f].x, o3[f].y) : o3[f].x;
                if (lo >= 0)
                    park[((2 * f + 1) * K + lo) * bstride] = kSplit ? fmaf(-al[2 * f + 1], o3[f].x, o3[f].y) : o3[f].y;
            }
#pragma unroll
            for (int f = 0; f < 7; f++) p0[f] = p1[f];
        }
        // 5. fast and slow fields, then Alfven and entropy
#pragma unroll
        for (int f = 0; f < 4; f++) {
            const int s = 2 * f;
            if constexpr (kSplit) corr[s] = wt.corr_s(fa[f], fb[f]);
            else corr[s] = wt.corr_d(s, fa[f], fb[f], lf_speed(sm, nc, id, s, lam_avg(e, s)));
        }
#pragma unroll
        for (int f = 0; f < 3; f++) {
            T pa[K], na[K];
#pragma unroll
            for (int m = 0; m < K; m++) {
                pa[m] = park[(2 * f * K + m) * bstride];
                na[m] = park[((2 * f + 1) * K + m) * bstride];
            }
            const int s = 2 * f + 1;
            if constexpr (kSplit) corr[s] = wt.corr_s(pa, na);
            else corr[s] = wt.corr_d(s, pa, na, lf_speed(sm, nc, id, s, lam_avg(e, s)));
        }
    } else {
    // 3-5. fast and slow fields
    {
        T w[4][6], g[4][6];
#pragma unroll
        for (int m = 0; m < 6; m++) {
            T x[7], o[4];
            load7(sm, nc, SU, id[m], x);
            project_fs(e, x, o);
#pragma unroll
            for (int f = 0; f < 4; f++) w[f][m] = o[f];
            load7(sm, nc, SF, id[m], x);
            project_fs(e, x, o);
#pragma unroll
            for (int f = 0; f < 4; f++) g[f][m] = o[f];
        }
#pragma unroll
        for (int f = 0; f < 4; f++) {
            const int s = 2 * f;
            corr[s] = wt.corr(s, w[f], g[f], lf_speed(sm, nc, id, s, lam_avg(e, s)));
        }
    }
    // 3-5. Alfven and entropy fields
    {
        T w[3][6], g[3][6];
#pragma unroll
        for (int m = 0; m < 6; m++) {
            T x[7], o[3];
            load7(sm, nc, SU, id[m], x);
            project_ae(e, x, o);
#pragma unroll
            for (int f = 0; f < 3; f++) w[f][m] = o[f];
            load7(sm, nc, SF, id[m], x);
            project_ae(e, x, o);
#pragma unroll
            for (int f = 0; f < 3; f++) g[f][m] = o[f];
        }
#pragma unroll
        for (int f = 0; f < 3; f++) {
            const int s = 2 * f + 1;
            corr[s] = wt.corr(s, w[f], g[f], lf_speed(sm, nc, id, s, lam_avg(e, s)));
        }
    }
    }
    // 6. back-projection: sum_s r_s corr_s in primitive variables, then dU/dW,
    // added to the central flux (-F_{i-1} + 7F_i + 7F_{i+1} - F_{i+2}) / 12
    const T alf = bp[BP_ALF * bstride], als = bp[BP_ALS * bstride];
    const T afcf = bp[BP_AFCF * bstride], ascs = bp[BP_ASCS * bstride];
    const T Fp = corr[6] + corr[0], Fm = corr[6] - corr[0];
    const T Sp = corr[4] + corr[2], Sm = corr[4] - corr[2];
    const T Ap = corr[5] + corr[1], Am = corr[5] - corr[1];
    const T fs = alf * Fp + als * Sp;
    const T drho = e.rho * fs + corr[3];
    const T du = afcf * Fm + ascs * Sm;
    const T dvpar = afcf * Sm - ascs * Fm;     // times sgn(B_n), folded into Ssr below
    const T dvperp = Ap;
    const T dbpar = bp[BP_ASR * bstride] * (als * Fp - alf * Sp);
    const T ssr = bp[BP_SSR * bstride];
    const T S = ssr < T(0) ? T(-1) : T(1);
    const T dbperp = -ssr * Am;
    const T dp = bp[BP_RA2 * bstride] * fs;
    const T dv1 = e.be1 * S * dvpar - e.be2 * dvperp;
    const T dv2 = e.be2 * S * dvpar + e.be1 * dvperp;
    const T db1 = e.be1 * dbpar - e.be2 * dbperp;
    const T db2 = e.be2 * dbpar + e.be1 * dbperp;
#pragma unroll
    for (int f = 0; f < 7; f++) {
        auto F = [&](int m) { return sm[at_f<T>(f, nc, id[m])]; };
        out[f] = (T(7) * (F(2) + F(3)) - (F(1) + F(4))) * T(1.0 / 12.0);
    }
    out[0] += drho;
    out[1] += e.u * drho + e.rho * du;
    out[2] += e.v1 * drho + e.rho * dv1;
    out[3] += e.v2 * drho + e.rho * dv2;
    out[4] += db1;
    out[5] += db2;
    out[6] += e.hv2 * drho + e.rho * (e.u * du + e.v1 * dv1 + e.v2 * dv2)
            + e.bm * dbpar + dp * bp[BP_IGM1 * bstride];
}

// ---- the kernel -------------------------------------------------------------
// Tile shapes (interfaces along the axis x pencils).
#ifndef WB_SWEEP_TA_X
#define WB_SWEEP_TA_X 32
#endif
#ifndef WB_SWEEP_TA_YZ
#define WB_SWEEP_TA_YZ 16
#endif
// interfaces per tile of the Jiang-Shu / WENO-Z sweeps
constexpr int kSweepNT = 128;
static_assert(kSweepNT == kFlatCells, "a flat tile is one cell per thread");
template <int AXIS> struct Shape;
template <> struct Shape<0> { static constexpr int TA = WB_SWEEP_TA_X, TP = 256 / WB_SWEEP_TA_X; };
template <> struct Shape<1> { static constexpr int TA = WB_SWEEP_TA_YZ, TP = 256 / WB_SWEEP_TA_YZ; };
template <> struct Shape<2> { static constexpr int TA = WB_SWEEP_TA_YZ, TP = 256 / WB_SWEEP_TA_YZ; };

// Tile shapes a tile may use, per axis: TA interfaces along the axis times
// TP = kSweepNT / TA pencils.  Shape 0 is the default; the host picks a shape per
// patch (fewest thread slots for the patch's sizes) and stores it in the top
// byte of the tile's patch field.
#ifndef WB_SWEEP_TA_X1
#define WB_SWEEP_TA_X1 8
#endif
__host__ __device__ constexpr int shape_ta(int axis, int s) {
    return axis == 0 ? (s == 0 ? WB_SWEEP_TA_X : (s == 1 ? WB_SWEEP_TA_X1 : 16))
                     : (s == 0 ? WB_SWEEP_TA_YZ : (s == 1 ? 8 : 32));
}
constexpr int kNShape = 3;
__host__ __device__ constexpr int nc_of(int ta) { return (ta + 5) * (kSweepNT / ta); }

}  // namespace
}  // namespace wb

// ---- training-record harvest -------------------------------------------------
// For each sampled interface (the lower face of cell `cells[t]` along `axis`
// of patch 0) and each characteristic field and side, one record of
// WB_MLP_RECORD floats: field, x[6], q[3], T, flag.  v is the split flux g+
// over the stencil cells i-2..i+3 ('-' side: g- reversed), x = (v - mean) /
// (max|v - mean| + 1e-12), q the three third-order candidate reconstructions
// of v at the face, T the face value of the split flux built from hU, hF (the
// exact face reconstructions of U and F, supplied by the caller) with the
// same left eigenvector and Lax-Friedrichs speed, q and T normalised like x;
// flag = 1 when the jump detector (largest of the four differences phi_N
// reads above kappa times the mean of the other three) or the pressure
// detector (max p > (1 + pjump) min p over the six cells) fires.
namespace wb {
namespace {

template <class T>
struct HarvestArgs {
    const T* src;
    long long ncells;
    PatchDev P;
    int axis;
    const long long* cells;
    long long n;
    const double* hU;
    const double* hF;
    double gamma, kappa, pjump;
    float* out;
};

template <class T, int AXIS>
__device__ void harvest_one(const HarvestArgs<T>& H, long long t, T* sm, int nc, int base, T* bp,
                            int bstride) {
    const PatchDev& P = H.P;
    const long long cell = H.cells[t];
    const int i0 = (int)(cell % P.nx), j0 = (int)((cell / P.nx) % P.ny), k0 = (int)(cell / ((long long)P.nx * P.ny));
    SweepArgs<T> A;
    A.src = H.src; A.flux = nullptr; A.er = nullptr; A.tiles = nullptr; A.patches = nullptr;
    A.ncells = H.ncells; A.gamma = H.gamma;
    const int na = AXIS == 0 ? P.nx : (AXIS == 1 ? P.ny : P.nz);
    const int a0 = AXIS == 0 ? i0 : (AXIS == 1 ? j0 : k0);
    T pmin = T(1e300), pmax = T(-1e300);
    int id[6];
    for (int m = 0; m < 6; m++) {
        const int a = wrap(a0 - 3 + m, na);
        int i = i0, j = j0, k = k0;
        if (AXIS == 0) i = a; else if (AXIS == 1) j = a; else k = a;
        RawCell<T> r;
        long long c;
        load_cell<T>(A, P, i, j, k, r, c);
        id[m] = base + m;
        derive_cell<T, AXIS>(A, r, c, sm, nc, id[m], false);
        const T p = sm[SP_P * nc + id[m]];
        pmin = p < pmin ? p : pmin;
        pmax = p > pmax ? p : pmax;
    }
    const bool pfire = pmax > (T(1) + T(H.pjump)) * pmin;
    Eig<T> e;
    {
        const int l = id[2], r = id[3];
        const T h = T(0.5);
        eigen<T>(h * (sm[at_u<T>(0, nc, l)] + sm[at_u<T>(0, nc, r)]), h * (sm[SP_U * nc + l] + sm[SP_U * nc + r]),
                 h * (sm[SP_V1 * nc + l] + sm[SP_V1 * nc + r]), h * (sm[SP_V2 * nc + l] + sm[SP_V2 * nc + r]),
                 h * (sm[SP_BN * nc + l] + sm[SP_BN * nc + r]), h * (sm[at_u<T>(4, nc, l)] + sm[at_u<T>(4, nc, r)]),
                 h * (sm[at_u<T>(5, nc, l)] + sm[at_u<T>(5, nc, r)]), h * (sm[SP_P * nc + l] + sm[SP_P * nc + r]),
                 T(H.gamma), e, bp, bstride);
    }
    T hu[7], hf[7];
    for (int f = 0; f < 7; f++) { hu[f] = T(H.hU[t * 7 + f]); hf[f] = T(H.hF[t * 7 + f]); }
    for (int G = 0; G < 4; G++) {
        T w[2][6], g[2][6], tu[2], tf[2];
        for (int m = 0; m < 6; m++) {
            T x[7], o[2];
            load7(sm, nc, SU, id[m], x);
            if (G == 0) project_pair<0>(e, x, o); else if (G == 1) project_pair<1>(e, x, o);
            else if (G == 2) project_pair<2>(e, x, o); else project_pair<3>(e, x, o);
            w[0][m] = o[0]; w[1][m] = o[1];
            load7(sm, nc, SF, id[m], x);
            if (G == 0) project_pair<0>(e, x, o); else if (G == 1) project_pair<1>(e, x, o);
            else if (G == 2) project_pair<2>(e, x, o); else project_pair<3>(e, x, o);
            g[0][m] = o[0]; g[1][m] = o[1];
        }
        {
            T o[2];
            if (G == 0) project_pair<0>(e, hu, o); else if (G == 1) project_pair<1>(e, hu, o);
            else if (G == 2) project_pair<2>(e, hu, o); else project_pair<3>(e, hu, o);
            tu[0] = o[0]; tu[1] = o[1];
            if (G == 0) project_pair<0>(e, hf, o); else if (G == 1) project_pair<1>(e, hf, o);
            else if (G == 2) project_pair<2>(e, hf, o); else project_pair<3>(e, hf, o);
            tf[0] = o[0]; tf[1] = o[1];
        }
        const int sl[2] = {G == 0 ? 0 : (G == 1 ? 2 : (G == 2 ? 1 : 3)), G == 0 ? 6 : (G == 1 ? 4 : (G == 2 ? 5 : 3))};
        const int nsl = G == 3 ? 1 : 2;
        for (int q = 0; q < nsl; q++) {
            const int s = sl[q];
            const T al = lf_speed(sm, nc, id, s, lam_avg(e, s));
            for (int side = 0; side < 2; side++) {
                const T sg = side == 0 ? T(1) : T(-1);
                T v[6];
                for (int m = 0; m < 6; m++) {
                    const int mm = side == 0 ? m : 5 - m;
                    v[m] = T(0.5) * (g[q][mm] + sg * al * w[q][mm]);
                }
                const T Tg = T(0.5) * (tf[q] + sg * al * tu[q]);
                T mean = T(0);
                for (int m = 0; m < 6; m++) mean += v[m];
                mean *= T(1.0 / 6.0);
                T mx = T(0);
                for (int m = 0; m < 6; m++) { const T d = tabs(v[m] - mean); mx = d > mx ? d : mx; }
                const T inv = T(1) / (mx + T(1e-12));
                T D[4];
                for (int m = 0; m < 4; m++) D[m] = tabs(v[m + 1] - v[m]);
                T dmax = D[0], dsum = D[0];
                for (int m = 1; m < 4; m++) { dmax = D[m] > dmax ? D[m] : dmax; dsum += D[m]; }
                const bool jfire = dmax > T(H.kappa) * (dsum - dmax) * T(1.0 / 3.0) + T(1e-300);
                float* o = H.out + ((t * 7 + s) * 2 + side) * WB_MLP_RECORD;
                o[0] = float(s);
                for (int m = 0; m < 6; m++) o[1 + m] = float((v[m] - mean) * inv);
                const T q0 = (T(2) * v[0] - T(7) * v[1] + T(11) * v[2]) * T(1.0 / 6.0);
                const T q1 = (-v[1] + T(5) * v[2] + T(2) * v[3]) * T(1.0 / 6.0);
                const T q2 = (T(2) * v[2] + T(5) * v[3] - v[4]) * T(1.0 / 6.0);
                o[7] = float((q0 - mean) * inv);
                o[8] = float((q1 - mean) * inv);
                o[9] = float((q2 - mean) * inv);
                o[10] = float((Tg - mean) * inv);
                o[11] = (jfire || pfire) ? 1.f : 0.f;
            }
        }
    }
}

template <class T>
__global__ void __launch_bounds__(32) harvest_kernel(const HarvestArgs<T> H) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sm = reinterpret_cast<T*>(smem_raw);
    const int nc = 6 * 32;
    T* bp = sm + kNSlot * nc + threadIdx.x;
    const long long t = (long long)blockIdx.x * 32 + threadIdx.x;
    if (t >= H.n) return;
    const int base = threadIdx.x * 6;
    if (H.axis == 0) harvest_one<T, 0>(H, t, sm, nc, base, bp, 32);
    else if (H.axis == 1) harvest_one<T, 1>(H, t, sm, nc, base, bp, 32);
    else harvest_one<T, 2>(H, t, sm, nc, base, bp, 32);
}

// Rotated conserved 7-vector (rho, m_n, m_t1, m_t2, B_t1, B_t2, E) and its
// physical flux along AXIS for every cell of a periodic patch: the sweep's
// own staging arithmetic (cell B from the faces, rotation, primitives, flux),
// written as FP64 arrays [7][cells] each.  The training pipeline reconstructs
// exact face values of these for its targets.
template <class T, int AXIS>
__global__ void __launch_bounds__(128) cell_state_flux_kernel(const SweepArgs<T> A, const PatchDev P,
                                                              double* __restrict__ X,
                                                              double* __restrict__ F) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sm = reinterpret_cast<T*>(smem_raw);
    const long long np = (long long)P.nx * P.ny * P.nz;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= np) return;
    const int nc = blockDim.x;
    const int i = (int)(t % P.nx), j = (int)((t / P.nx) % P.ny), k = (int)(t / ((long long)P.nx * P.ny));
    RawCell<T> r;
    long long c;
    load_cell<T>(A, P, i, j, k, r, c);
    derive_cell<T, AXIS>(A, r, c, sm, nc, threadIdx.x, false);
    for (int f = 0; f < 7; f++) {
        X[f * np + t] = double(sm[at_u<T>(f, nc, threadIdx.x)]);
        F[f * np + t] = double(sm[at_f<T>(f, nc, threadIdx.x)]);
    }
}

}  // namespace

template <class T>
cudaError_t launch_cell_state_flux(const T* src, long long ncells, const PatchDev& P, int axis,
                                   double gamma, double* X, double* F, cudaStream_t s) {
    SweepArgs<T> A;
    A.src = src; A.flux = nullptr; A.er = nullptr; A.tiles = nullptr; A.patches = nullptr;
    A.ncells = ncells; A.gamma = gamma;
    const long long np = (long long)P.nx * P.ny * P.nz;
    const int nt = 128;
    const unsigned nb = (unsigned)((np + nt - 1) / nt);
    const size_t smem = sizeof(T) * kNSlot * nt;
    if (axis == 0) cell_state_flux_kernel<T, 0><<<nb, nt, smem, s>>>(A, P, X, F);
    else if (axis == 1) cell_state_flux_kernel<T, 1><<<nb, nt, smem, s>>>(A, P, X, F);
    else cell_state_flux_kernel<T, 2><<<nb, nt, smem, s>>>(A, P, X, F);
    return cudaGetLastError();
}

template <class T>
cudaError_t launch_harvest(const T* src, long long ncells, const PatchDev& P, int axis,
                           const long long* cells, long long n, const double* hU, const double* hF,
                           double gamma, double kappa, double pjump, float* out, cudaStream_t s) {
    HarvestArgs<T> H{src, ncells, P, axis, cells, n, hU, hF, gamma, kappa, pjump, out};
    const size_t smem = sizeof(T) * (kNSlot * 6 * 32 + kNBack * 32);
    cudaError_t e = cudaFuncSetAttribute(harvest_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    harvest_kernel<T><<<(unsigned)((n + 31) / 32), 32, smem, s>>>(H);
    return cudaGetLastError();
}

}  // namespace wb
