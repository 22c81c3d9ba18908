// wb_reduce.cu -- CFL time step (FP64 max reduction with warp shuffles),
// deterministic FP64 conserved totals, and the FP64 <-> state conversions
// used at the ABI.
#include "wb_internal.h"
#include "wb_math.cuh"

#include <cfloat>
#include <limits>

namespace wb {
namespace {

// dt rule: s = sum_d (|v_d| + c_f,d) / dx_d per cell, maximised over cells;
// the fast speed along d uses B_d as the normal field.  The per-cell speed is
// taken in the state's precision (FP32 in FP32 mode: FP64 division and square
// root run at a small fraction of the FP32 rate on this GPU); the maximum is
// reduced in FP64, which is exact.
// Upper neighbour of cell (i, j, k) of patch p along each axis: the wrap
// round a periodic patch, or the link table's neighbour.
template <bool LINKED>
__device__ __forceinline__ long long upper(const PatchDev* __restrict__ patches,
                                           const int* __restrict__ links, int p, const PatchDev& P,
                                           int i, int j, int k) {
    if constexpr (LINKED) return locate(patches, links, p, P, i, j, k);
    i = i == P.nx ? 0 : i;
    j = j == P.ny ? 0 : j;
    k = k == P.nz ? 0 : k;
    return P.off + ((long long)k * P.ny + j) * P.nx + i;
}

// Folds one cell's signal rate into the running maximum s (kept in T: the
// largest of FP32 values converted to FP64 once is the largest of their FP64
// conversions, the conversion being exact and monotonic, so FP32 grids keep
// the FP64 pipe out of the loop); flags NaN/Inf and rho, p <= 0.
template <class T>
__device__ __forceinline__ void fold_signal(T& s, T rho, T m0, T m1, T m2, T E, T B0, T B1, T B2,
                                            T g, T id0, T id1, T id2, unsigned int* flag) {
    T p;
    T sc = cell_signal<T>(rho, m0, m1, m2, E, B0, B1, B2, g, id0, id1, id2, p);
    unsigned int bad = 0;
    if (!(sc <= std::numeric_limits<T>::max())) bad |= 1u;   // NaN or Inf
    if (!(rho > T(0)) || !(p > T(0))) bad |= 2u;
    if (bad) {
        atomicOr(flag, bad);
        sc = T(0);
    }
    s = sc > s ? sc : s;
}

// Block maximum of s, folded into *smax_bits as an FP64 bit pattern (s >= 0,
// so the IEEE bit patterns order like the values).
template <class T>
__device__ __forceinline__ void block_max_out(T s, unsigned long long* smax_bits) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const T r = __shfl_xor_sync(0xffffffffu, s, o);
        s = r > s ? r : s;
    }
    __shared__ T red[kCellBlock / 32];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        s = threadIdx.x < kCellBlock / 32 ? red[threadIdx.x] : T(0);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const T r = __shfl_xor_sync(0xffffffffu, s, o);
            s = r > s ? r : s;
        }
        if (threadIdx.x == 0)
            atomicMax(smax_bits, (unsigned long long)__double_as_longlong(double(s)));
    }
}

// One thread per cell, any patches (linked ones too).
template <class T, bool LINKED>
__global__ void __launch_bounds__(kCellBlock)
cfl_kernel(const T* __restrict__ q, const CellBlock* __restrict__ blocks, int nblocks,
           const PatchDev* __restrict__ patches, const int* __restrict__ links, long long N,
           double idx, double idy, double idz, double gamma, unsigned long long* smax_bits,
           unsigned int* flag) {
    T s = T(0);
    const T g = T(gamma), i0 = T(idx), i1 = T(idy), i2 = T(idz);
    // grid-stride over the cell blocks: one atomic per resident block, not
    // one per 256 cells (same-address atomics serialise in L2)
    for (int b = blockIdx.x; b < nblocks; b += gridDim.x) {
        const CellBlock cb = blocks[b];
        const PatchDev P = patches[cb.x];
        const int local = cb.y + threadIdx.x;
        const int nxy = P.nx * P.ny;
        if (local < nxy * P.nz) {
            const int k = local / nxy;
            const int rem = local - k * nxy;
            const int j = rem / P.nx;
            const int i = rem - j * P.nx;
            const long long c = chk(P.off + local, N, flag);
            const long long cx = chk(upper<LINKED>(patches, links, cb.x, P, i + 1, j, k), N, flag);
            const long long cy = chk(upper<LINKED>(patches, links, cb.x, P, i, j + 1, k), N, flag);
            const long long cz = chk(upper<LINKED>(patches, links, cb.x, P, i, j, k + 1), N, flag);
            fold_signal<T>(s, q[c], q[N + c], q[2 * N + c], q[3 * N + c], q[4 * N + c],
                           rn::mul(T(0.5), rn::add(q[5 * N + c], q[5 * N + cx])),
                           rn::mul(T(0.5), rn::add(q[6 * N + c], q[6 * N + cy])),
                           rn::mul(T(0.5), rn::add(q[7 * N + c], q[7 * N + cz])), g, i0, i1, i2, flag);
        }
    }
    block_max_out<T>(s, smax_bits);
}

template <class T> struct CflVec;
template <> struct CflVec<float> { using type = float4; static constexpr int V = 4; };
template <> struct CflVec<double> { using type = double2; static constexpr int V = 2; };

template <class T, int V>
__device__ __forceinline__ void vget(const T* __restrict__ p, T (&v)[V]) {
    const typename CflVec<T>::type x = *reinterpret_cast<const typename CflVec<T>::type*>(p);
    if constexpr (V == 4) { v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w; }
    else { v[0] = x.x; v[1] = x.y; }
}

// One thread per 16-byte vector of cells along x, for periodic patches whose
// x extent is a multiple of the vector width (vector blocks of the grid):
// four times the bytes in flight per thread, the same per-cell arithmetic.
template <class T>
__global__ void __launch_bounds__(kCellBlock)
cfl_kernel_vec(const T* __restrict__ q, const CellBlock* __restrict__ vblocks, int nvblocks,
               const PatchDev* __restrict__ patches, long long N, double idx, double idy, double idz,
               double gamma, unsigned long long* smax_bits, unsigned int* flag) {
    constexpr int V = CflVec<T>::V;
    T s = T(0);
    const T g = T(gamma), i0 = T(idx), i1 = T(idy), i2 = T(idz);
    for (int b = blockIdx.x; b < nvblocks; b += gridDim.x) {
        const CellBlock cb = vblocks[b];
        const PatchDev P = patches[cb.x];
        const int local = cb.y + threadIdx.x * V;
        const int nxy = P.nx * P.ny;
        if (local < nxy * P.nz) {
            const int k = local / nxy;
            const int rem = local - k * nxy;
            const int j = rem / P.nx;
            const int i = rem - j * P.nx;
            const int ip = i + V == P.nx ? 0 : i + V;
            const int jp = j + 1 == P.ny ? 0 : j + 1, kp = k + 1 == P.nz ? 0 : k + 1;
            auto at = [&](int a, int bb, int cc) { return P.off + ((long long)cc * P.ny + bb) * P.nx + a; };
            const long long c = P.off + local, cxp = at(ip, j, k), cyp = at(i, jp, k), czp = at(i, j, kp);
#if WB_BOUNDS_CHECK
            auto vec_ok = [&](long long a) { return a >= 0 && a + V <= N && a % V == 0; };
            if (!(vec_ok(c) && vec_ok(cyp) && vec_ok(czp) && cxp >= 0 && cxp < N)) {
                atomicOr(flag, kFlagBounds);
                continue;
            }
#endif
            T rho[V], m0[V], m1[V], m2[V], E[V], bx[V], by[V], bz[V], byp[V], bzp[V];
            vget<T, V>(q + c, rho);
            vget<T, V>(q + N + c, m0);
            vget<T, V>(q + 2 * N + c, m1);
            vget<T, V>(q + 3 * N + c, m2);
            vget<T, V>(q + 4 * N + c, E);
            vget<T, V>(q + 5 * N + c, bx);
            vget<T, V>(q + 6 * N + c, by);
            vget<T, V>(q + 7 * N + c, bz);
            vget<T, V>(q + 6 * N + cyp, byp);
            vget<T, V>(q + 7 * N + czp, bzp);
            const T bx_next = q[5 * N + cxp];
#pragma unroll
            for (int v = 0; v < V; v++) {
                const T bxu = v + 1 < V ? bx[v + 1] : bx_next;
                fold_signal<T>(s, rho[v], m0[v], m1[v], m2[v], E[v], rn::mul(T(0.5), rn::add(bx[v], bxu)),
                               rn::mul(T(0.5), rn::add(by[v], byp[v])), rn::mul(T(0.5), rn::add(bz[v], bzp[v])),
                               g, i0, i1, i2, flag);
            }
        }
    }
    block_max_out<T>(s, smax_bits);
}

// s + e = a + b exactly, s rounded (Knuth's two-sum); e is NaN where s overflows.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float t = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
}

// (xp - x) idx + (yp - y) idy + (zp - z) idz in FP64.
__device__ __forceinline__ double face_div(double xp, double x, double yp, double y, double zp, double z, double idx,
                                           double idy, double idz) {
    return (xp - x) * idx + (yp - y) * idy + (zp - z) * idz;
}
// FP32 faces: an upper bound of its magnitude, and whether that is below
// `least`, from pairs of FP32 values (differences exact, products and sums to
// 2^-42 of the terms' magnitudes; ih + il = 1 / dx to 2^-48, for 1 / dx from
// 1e-30 on).
__device__ __forceinline__ bool face_div_below(float xp, float x, float yp, float y, float zp, float z, float2 ix,
                                               float2 iy, float2 iz, float least) {
    float hi = 0.f, lo = 0.f, mag = 0.f;
    auto term = [&](float up, float own, float2 inv) {
        float d, e, s, r;
        two_sum(up, -own, d, e);
        const float p = __fmul_rn(d, inv.x);
        const float pe = __fmaf_rn(d, inv.x, -p) + (d * inv.y + e * inv.x);
        two_sum(hi, p, s, r);
        hi = s;
        lo += r + pe;
        mag += fabsf(p);
    };
    term(xp, x, ix);
    term(yp, y, iy);
    term(zp, z, iz);
    // NaN and overflow compare false: the caller then takes the FP64 value
    return fabsf(hi + lo) * 1.000001f + mag * 3e-13f + 1e-37f < least;
}

// Face divergence of b per cell (the quantity constrained transport keeps at
// round-off, Sec. 2.1): (bx(i+1) - bx(i))/dx + (by(j+1) - by(j))/dy +
// (bz(k+1) - bz(k))/dz, in FP64; out_bits[0] = max |div b|, out_bits[1] =
// max |b| over the faces, both as FP64 bit patterns (non-negative values, so
// an integer maximum orders them).
template <class T, bool LINKED>
__global__ void __launch_bounds__(kCellBlock)
divb_kernel(const T* __restrict__ q, const CellBlock* __restrict__ blocks, int nblocks,
            const PatchDev* __restrict__ patches, const int* __restrict__ links, long long N,
            double idx, double idy, double idz, unsigned long long* out_bits, unsigned int* flag) {
    // |d| as its FP64 bit pattern (non-negative values: an integer maximum
    // orders them), max |b| in the grid's precision; NaN counts in neither.
    // FP32 grids evaluate d in FP64 only where it can exceed the warp's largest
    // so far (`least`, rounded down), which a few cells of a warp's share do:
    // the FP64 pipe was the bound (192^3: 235 -> 88 us with the host's part).
    long long dmax = 0;
    T bmax = T(0);
    float least = 0.f;
    auto pair = [](double v) { const float h = float(v); return make_float2(h, float(v - double(h))); };
    const float2 ix = pair(idx), iy = pair(idy), iz = pair(idz);
    // below 1e-30 the pairs lose bits to the subnormal numbers
    const bool pairs = sizeof(T) == 4 && fminf(ix.x, fminf(iy.x, iz.x)) >= 1e-30f;
    for (int b = blockIdx.x; b < nblocks; b += gridDim.x) {
        const CellBlock cb = blocks[b];
        const PatchDev P = patches[cb.x];
        const int local = cb.y + threadIdx.x;
        const int nxy = P.nx * P.ny;
        const bool in = local < nxy * P.nz;
        T bx = T(0), by = T(0), bz = T(0), xp = T(0), yp = T(0), zp = T(0);
        if (in) {
            const int k = local / nxy;
            const int rem = local - k * nxy;
            const int j = rem / P.nx;
            const int i = rem - j * P.nx;
            const long long c = chk(P.off + local, N, flag);
            const long long cx = chk(upper<LINKED>(patches, links, cb.x, P, i + 1, j, k), N, flag);
            const long long cy = chk(upper<LINKED>(patches, links, cb.x, P, i, j + 1, k), N, flag);
            const long long cz = chk(upper<LINKED>(patches, links, cb.x, P, i, j, k + 1), N, flag);
            bx = q[5 * N + c]; by = q[6 * N + c]; bz = q[7 * N + c];
            xp = q[5 * N + cx]; yp = q[6 * N + cy]; zp = q[7 * N + cz];
            bmax = fmax(bmax, fmax(fabs(bx), fmax(fabs(by), fabs(bz))));
        }
        bool need = in;
        if constexpr (sizeof(T) == 4) {
            need = in && !(pairs && face_div_below(xp, bx, yp, by, zp, bz, ix, iy, iz, least));
            if (!__any_sync(0xffffffffu, need)) continue;
        }
        if (need) {
            double d;
            if constexpr (sizeof(T) == 4)
                d = face_div(widen(xp), widen(bx), widen(yp), widen(by), widen(zp), widen(bz), idx, idy, idz);
            else
                d = face_div(xp, bx, yp, by, zp, bz, idx, idy, idz);
            const long long bits = __double_as_longlong(d) & 0x7fffffffffffffffll;
            if (bits <= 0x7ff0000000000000ll) dmax = max(dmax, bits);
        }
        if constexpr (sizeof(T) == 4) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) dmax = max(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
            least = __double2float_rd(__longlong_as_double(dmax));
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        dmax = max(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
        bmax = fmax(bmax, __shfl_xor_sync(0xffffffffu, bmax, o));
    }
    __shared__ long long rd[kCellBlock / 32];
    __shared__ T rb[kCellBlock / 32];
    if ((threadIdx.x & 31) == 0) {
        rd[threadIdx.x >> 5] = dmax;
        rb[threadIdx.x >> 5] = bmax;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        // one pair of atomics per block (same-address atomics serialise in L2)
#pragma unroll
        for (int w = 1; w < kCellBlock / 32; w++) {
            dmax = max(dmax, rd[w]);
            bmax = fmax(bmax, rb[w]);
        }
        atomicMax(out_bits, (unsigned long long)dmax);
        atomicMax(out_bits + 1, (unsigned long long)__double_as_longlong(double(bmax)));
    }
}

__global__ void set_dt_kernel(const unsigned long long* smax_bits, double cfl, double fixed_dt,
                              double* dt, double* time) {
    double d = fixed_dt;
    if (!(fixed_dt > 0.0)) {
        const double smax = __longlong_as_double((long long)*smax_bits);
        d = smax > 0.0 ? cfl / smax : 0.0;
    }
    *dt = d;
    *time += d;
}

// Totals: sum over cells of rho, m, E and of the face fields (for a periodic
// patch the sum of the face means equals the sum over faces).  Pass 1: each
// block reduces a fixed contiguous chunk in a fixed order; pass 2: one block
// reduces the partials.  Same order on every call, so bitwise repeatable.
// Sum over the block of each thread's eight values, in a fixed order: warp f
// adds field f, each lane eight threads' values and then the lanes (a tree over
// all fields on the block's first warps would queue on one scheduler's FP64
// pipe).  Valid in lane 0 of warp f.
__device__ __forceinline__ double block_sum8(const double (&acc)[8], double (*red)[256]) {
#pragma unroll
    for (int f = 0; f < 8; f++) red[f][threadIdx.x] = acc[f];
    __syncthreads();
    const int f = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double s = red[f][lane];
#pragma unroll
    for (int u = 1; u < 8; u++) s += red[f][lane + 32 * u];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

template <class T>
__global__ void __launch_bounds__(256)
totals_pass1(const T* __restrict__ q, long long N, long long chunk, double* __restrict__ partial) {
    const long long beg = (long long)blockIdx.x * chunk;
    long long end = beg + chunk;
    if (end > N) end = N;
    double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if constexpr (sizeof(T) == 4) {
        // FP32 values are added in FP32 with every rounding error kept: s the
        // running sum, eh + el the sum of its errors (two-sum at both levels,
        // el rounds at 2^-72 of the sum), added in FP64 at the end.  An FP64
        // addition per value was the bound (the pipe 79 % busy): 192^3, totals
        // of a state 153 -> 91 us with the host's part.
        float s[8] = {0, 0, 0, 0, 0, 0, 0, 0}, eh[8] = {0, 0, 0, 0, 0, 0, 0, 0}, el[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (long long c = beg + threadIdx.x; c < end; c += 512) {
            const bool two = c + 256 < end;
            float x[8][2];
#pragma unroll
            for (int f = 0; f < 8; f++) {
                x[f][0] = q[f * N + c];
                x[f][1] = two ? q[f * N + c + 256] : 0.f;
            }
#pragma unroll
            for (int f = 0; f < 8; f++)
#pragma unroll
                for (int u = 0; u < 2; u++) {
                    float e, r;
                    two_sum(s[f], x[f][u], s[f], e);
                    two_sum(eh[f], e, eh[f], r);
                    el[f] += r;
                }
        }
#pragma unroll
        for (int f = 0; f < 8; f++) {
            if (fabsf(s[f]) <= 3.4e38f && fabsf(eh[f]) <= 3.4e38f) {
                // s + eh + el without FP64 additions of zeros (a thread of a small grid
                // has a value or two, and every block pays the narrow pipe for them)
                float e, r;
                two_sum(eh[f], el[f], e, r);
                acc[f] = widen(s[f]);
                if (r != 0.f) acc[f] += widen(e) + widen(r);
                else if (e != 0.f) acc[f] += widen(e);
            } else {                           // out of the FP32 range, infinite or NaN
                for (long long c = beg + threadIdx.x; c < end; c += 256) acc[f] += widen(q[f * N + c]);
            }
        }
    } else {
        for (long long c = beg + threadIdx.x; c < end; c += 256) {
#pragma unroll
            for (int f = 0; f < 8; f++) acc[f] += q[f * N + c];
        }
    }
    __shared__ double red[8][256];
    const double sum = block_sum8(acc, red);
    if ((threadIdx.x & 31) == 0) partial[blockIdx.x * 8 + (threadIdx.x >> 5)] = sum;
}

__global__ void __launch_bounds__(256)
totals_pass2(const double* __restrict__ partial, int npartial, double dV, double* __restrict__ out) {
    double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int b = threadIdx.x; b < npartial; b += 256) {
#pragma unroll
        for (int f = 0; f < 8; f++) acc[f] += partial[b * 8 + f];
    }
    __shared__ double red[8][256];
    const double sum = block_sum8(acc, red);
    // state order rho, mx, my, mz, E, bx, by, bz -> ABI order
    // rho, mx, my, mz, Bx, By, Bz, E
    const int f = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) out[f < 4 ? f : (f == 4 ? 7 : f - 1)] = sum * dV;
}

// ABI layout (FP64, or FP32 for the FP32 entry points, type H): U[patch][8][cells]
// with (rho, mx, my, mz, Bx, By, Bz, E), b[patch][3][cells]; state layout:
// field-major over all patches.
//
// To and from page-locked host arrays (HOST) both copies are bound by the link, which
// moves whole 128-byte lines: each field's threads are shifted so that a warp covers
// one line of its host array
// (the fields of a patch of odd size start at odd places), and the ragged
// accesses fall on device memory.  FP32 state in and out, GB/s over the link:
// 320 uneven patches 190 / 142 -> 210 / 192, 64 uneven bricks 187 / 127 -> 205 /
// 188; 192^3, aligned as it is, 207 / 190 -> 208 / 190.  From device staging
// (pageable arrays) they are bound by the latency of the loads: one cell per thread,
// all its loads before the first store (192^3, FP64 arrays and an FP32 state, in and
// out: 190 / 347 us with the shifted threads' field by field, 98 / 253 so).
template <class H>
__device__ __forceinline__ int line_offset(const H* p) {
    return (int)((reinterpret_cast<unsigned long long>(p) / sizeof(H)) % (128 / sizeof(H)));
}
// Calls f(l) for the cells l of this block's share of a field whose host array
// starts at p: the block's 256 cells moved down to a line boundary, the patch's
// last block with the rest.
template <class H, class F>
__device__ __forceinline__ void line_cells(const H* p, int first, int np, F&& f) {
    const int l = first + (int)threadIdx.x - line_offset(p);
    if (l >= 0 && l < np) f(l);
    if (first + kCellBlock >= np && l + kCellBlock < np) f(l + kCellBlock);
}

template <class T, class H, bool HOST>
__global__ void __launch_bounds__(kCellBlock)
import_kernel(const H* __restrict__ U, const H* __restrict__ b, T* __restrict__ q,
              const CellBlock* __restrict__ blocks, const PatchDev* __restrict__ patches,
              long long N) {
    const CellBlock cb = blocks[blockIdx.x];
    const PatchDev P = patches[cb.x];
    const int np = P.nx * P.ny * P.nz;
    auto from = [&](int f) {
        return f < 5 ? U + 8 * P.off + (long long)(f == 4 ? 7 : f) * np : b + 3 * P.off + (long long)(f - 5) * np;
    };
    if constexpr (HOST) {
#pragma unroll
        for (int f = 0; f < 8; f++) {
            T* to = q + f * N + P.off;
            line_cells(from(f), cb.y, np, [&](int l) { to[l] = T(from(f)[l]); });
        }
    } else {
        const int l = cb.y + threadIdx.x;
        if (l >= np) return;
        H v[8];
#pragma unroll
        for (int f = 0; f < 8; f++) v[f] = from(f)[l];
#pragma unroll
        for (int f = 0; f < 8; f++) q[f * N + P.off + l] = T(v[f]);
    }
}

template <class T, class H, bool LINKED, bool HOST>
__global__ void __launch_bounds__(kCellBlock)
export_kernel(const T* __restrict__ q, H* __restrict__ U, H* __restrict__ b,
              const CellBlock* __restrict__ blocks, const PatchDev* __restrict__ patches,
              const int* __restrict__ links, long long N) {
    const CellBlock cb = blocks[blockIdx.x];
    const PatchDev P = patches[cb.x];
    const int nxy = P.nx * P.ny, np = nxy * P.nz;
    if constexpr (!HOST) {
        const int l = cb.y + threadIdx.x;
        if (l >= np) return;
        const int k = l / nxy;
        const int rem = l - k * nxy;
        const int j = rem / P.nx;
        const int i = rem - j * P.nx;
        const long long c = P.off + l;
        T v[5], face[3], up[3];
#pragma unroll
        for (int f = 0; f < 3; f++) face[f] = q[(5 + f) * N + c];
        if (U) {
#pragma unroll
            for (int f = 0; f < 5; f++) v[f] = q[f * N + c];
            up[0] = q[5 * N + upper<LINKED>(patches, links, cb.x, P, i + 1, j, k)];
            up[1] = q[6 * N + upper<LINKED>(patches, links, cb.x, P, i, j + 1, k)];
            up[2] = q[7 * N + upper<LINKED>(patches, links, cb.x, P, i, j, k + 1)];
            H* u = U + 8 * P.off + l;
#pragma unroll
            for (int f = 0; f < 4; f++) u[(long long)f * np] = H(double(v[f]));
#pragma unroll
            for (int f = 0; f < 3; f++) u[(long long)(4 + f) * np] = H(0.5 * (double(face[f]) + double(up[f])));
            u[7LL * np] = H(double(v[4]));
        }
        if (b) {
            H* o = b + 3 * P.off + l;
#pragma unroll
            for (int f = 0; f < 3; f++) o[(long long)f * np] = H(double(face[f]));
        }
        return;
    }
    if (U) {
#pragma unroll
        for (int f = 0; f < 8; f++) {
            H* to = U + 8 * P.off + (long long)f * np;
            const T* from = q + (f < 4 ? f : (f == 7 ? 4 : f + 1)) * N;
            line_cells(to, cb.y, np, [&](int l) {
                const T v = from[P.off + l];
                if (f < 4 || f == 7) {
                    to[l] = H(double(v));
                } else {
                    const int k = l / nxy;
                    const int rem = l - k * nxy;
                    const int j = rem / P.nx;
                    const int i = rem - j * P.nx;
                    const long long up = upper<LINKED>(patches, links, cb.x, P, i + (f == 4), j + (f == 5), k + (f == 6));
                    to[l] = H(0.5 * (double(v) + double(from[up])));
                }
            });
        }
    }
    if (b) {
#pragma unroll
        for (int f = 0; f < 3; f++) {
            H* to = b + 3 * P.off + (long long)f * np;
            const T* from = q + (5 + f) * N + P.off;
            line_cells(to, cb.y, np, [&](int l) { to[l] = H(double(from[l])); });
        }
    }
}

// Face fluxes of one axis to the ABI's patch-major FP64 layout [7][cells].
template <class T>
__global__ void __launch_bounds__(kCellBlock)
export_flux_kernel(const T* __restrict__ F, double* __restrict__ out,
                   const CellBlock* __restrict__ blocks, const PatchDev* __restrict__ patches,
                   long long N) {
    const CellBlock cb = blocks[blockIdx.x];
    const PatchDev P = patches[cb.x];
    const long long np = (long long)P.nx * P.ny * P.nz;
    const int local = cb.y + threadIdx.x;
    if (local >= np) return;
    const long long c = P.off + local;
    double* o = out + 7 * P.off + local;
#pragma unroll
    for (int q = 0; q < 7; q++) o[q * np] = double(F[q * N + c]);
}

}  // namespace

template <class T>
cudaError_t launch_export_flux(const T* flux, double* out, const CellBlock* blocks,
                               const PatchDev* patches, long long ncells, int nblocks,
                               cudaStream_t s) {
    export_flux_kernel<T><<<nblocks, kCellBlock, 0, s>>>(flux, out, blocks, patches, ncells);
    return cudaGetLastError();
}

template <class T>
cudaError_t launch_cfl(const T* state, const CellBlock* blocks, const PatchDev* patches,
                       const int* links, long long ncells, int nblocks, const CellBlock* vblocks,
                       int nvblocks, double idx, double idy, double idz, double gamma,
                       unsigned long long* smax_bits, unsigned int* flag, cudaStream_t s) {
    if (nblocks <= 0) return cudaSuccess;
    static int grid_cap = 0;
    if (grid_cap == 0) {
        int dev = 0, nsm = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        grid_cap = 8 * (nsm > 0 ? nsm : 152);      // one wave of 256-thread blocks
    }
    if (vblocks && nvblocks > 0 && !links) {
        const int vgrid = nvblocks < grid_cap ? nvblocks : grid_cap;
        cfl_kernel_vec<T><<<vgrid, kCellBlock, 0, s>>>(state, vblocks, nvblocks, patches, ncells, idx, idy,
                                                       idz, gamma, smax_bits, flag);
        return cudaGetLastError();
    }
    const int grid = nblocks < grid_cap ? nblocks : grid_cap;
    if (links)
        cfl_kernel<T, true><<<grid, kCellBlock, 0, s>>>(state, blocks, nblocks, patches, links, ncells,
                                                        idx, idy, idz, gamma, smax_bits, flag);
    else
        cfl_kernel<T, false><<<grid, kCellBlock, 0, s>>>(state, blocks, nblocks, patches, links, ncells,
                                                         idx, idy, idz, gamma, smax_bits, flag);
    return cudaGetLastError();
}

template <class T>
cudaError_t launch_divb(const T* state, const CellBlock* blocks, const PatchDev* patches,
                        const int* links, long long ncells, int nblocks, double idx, double idy,
                        double idz, unsigned long long* out_bits, unsigned int* flag, cudaStream_t s) {
    if (nblocks <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(out_bits, 0, 2 * sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int cap = 8 * (nsm > 0 ? nsm : 152);
    const int grid = nblocks < cap ? nblocks : cap;
    if (links)
        divb_kernel<T, true><<<grid, kCellBlock, 0, s>>>(state, blocks, nblocks, patches, links, ncells,
                                                         idx, idy, idz, out_bits, flag);
    else
        divb_kernel<T, false><<<grid, kCellBlock, 0, s>>>(state, blocks, nblocks, patches, links, ncells,
                                                          idx, idy, idz, out_bits, flag);
    return cudaGetLastError();
}

cudaError_t launch_set_dt(const unsigned long long* smax_bits, double cfl, double fixed_dt,
                          double* dt, double* time, cudaStream_t s) {
    set_dt_kernel<<<1, 1, 0, s>>>(smax_bits, cfl, fixed_dt, dt, time);
    return cudaGetLastError();
}

template <class T>
cudaError_t launch_totals(const T* state, const PatchDev*, int, long long ncells,
                          double* partial, int npartial, double dV, double* out, cudaStream_t s) {
    const long long chunk = (ncells + npartial - 1) / npartial;
    totals_pass1<T><<<npartial, 256, 0, s>>>(state, ncells, chunk, partial);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    totals_pass2<<<1, 256, 0, s>>>(partial, npartial, dV, out);
    return cudaGetLastError();
}

template <class T, class H>
cudaError_t launch_import(const H* U, const H* b, T* state, const CellBlock* blocks,
                          const PatchDev* patches, long long ncells, int nblocks, bool host, cudaStream_t s) {
    if (host) import_kernel<T, H, true><<<nblocks, kCellBlock, 0, s>>>(U, b, state, blocks, patches, ncells);
    else import_kernel<T, H, false><<<nblocks, kCellBlock, 0, s>>>(U, b, state, blocks, patches, ncells);
    return cudaGetLastError();
}

template <class T, class H, bool LINKED>
void launch_export_links(const T* state, H* U, H* b, const CellBlock* blocks, const PatchDev* patches,
                         const int* links, long long ncells, int nblocks, bool host, cudaStream_t s) {
    if (host)
        export_kernel<T, H, LINKED, true><<<nblocks, kCellBlock, 0, s>>>(state, U, b, blocks, patches, links, ncells);
    else
        export_kernel<T, H, LINKED, false><<<nblocks, kCellBlock, 0, s>>>(state, U, b, blocks, patches, links, ncells);
}

template <class T, class H>
cudaError_t launch_export(const T* state, H* U, H* b, const CellBlock* blocks,
                          const PatchDev* patches, const int* links, long long ncells, int nblocks,
                          bool host, cudaStream_t s) {
    if (links) launch_export_links<T, H, true>(state, U, b, blocks, patches, links, ncells, nblocks, host, s);
    else launch_export_links<T, H, false>(state, U, b, blocks, patches, links, ncells, nblocks, host, s);
    return cudaGetLastError();
}

#define WB_INST(T)                                                                            \
    template cudaError_t launch_cfl<T>(const T*, const CellBlock*, const PatchDev*, const int*, \
                                       long long, int, const CellBlock*, int, double, double, \
                                       double, double, unsigned long long*, unsigned int*,    \
                                       cudaStream_t);                                         \
    template cudaError_t launch_divb<T>(const T*, const CellBlock*, const PatchDev*, const int*, \
                                        long long, int, double, double, double,              \
                                        unsigned long long*, unsigned int*, cudaStream_t);    \
    template cudaError_t launch_totals<T>(const T*, const PatchDev*, int, long long, double*, \
                                          int, double, double*, cudaStream_t);                \
    template cudaError_t launch_import<T, double>(const double*, const double*, T*,          \
                                                  const CellBlock*, const PatchDev*, long long, \
                                                  int, bool, cudaStream_t);                    \
    template cudaError_t launch_export<T, double>(const T*, double*, double*, const CellBlock*, \
                                                  const PatchDev*, const int*, long long, int,  \
                                                  bool, cudaStream_t);                         \
    template cudaError_t launch_export_flux<T>(const T*, double*, const CellBlock*,           \
                                               const PatchDev*, long long, int, cudaStream_t);
WB_INST(float)
template cudaError_t launch_import<float, float>(const float*, const float*, float*, const CellBlock*,
                                                 const PatchDev*, long long, int, bool, cudaStream_t);
template cudaError_t launch_export<float, float>(const float*, float*, float*, const CellBlock*,
                                                 const PatchDev*, const int*, long long, int, bool, cudaStream_t);
WB_INST(double)
#undef WB_INST

}  // namespace wb
