// wb_mlp.cu -- training of the learned WENO weights: one small network per
// characteristic field (6 -> 32 -> 32 -> 3, GELU, softmax) that predicts the
// three nonlinear weights of phi_N (Sec. 2.1) from the normalised stencil.
//
// Records (12 floats): field, x[6] (normalised stencil), q[3] (normalised
// third-order sub-stencil fluxes), T (normalised target reconstruction),
// flag (1 = the jump detector fired; such records are not trained on).
// Loss per record: (sum_k w_k q_k - T)^2 + lam * sum_k d_k log(d_k / w_k).
//
// One training step, all seven networks at once, B records per field, in two
// launches:
//   grad_kernel      a block walks chunks of 32 records of one field: forward
//                    and backward pass out of shared memory, then every
//                    thread adds its share of the 1 380 gradient (and loss)
//                    entries, record by record in a fixed order;
//   apply_kernel     one thread per entry: the blocks' sums in a fixed order,
//                    the mean, and the Adam step of its parameter.
// Every sum over records has at least the bits and the range of an FP64 one, in
// a fixed order, so the gradient is bitwise repeatable.
// Minibatch indices come from a counter-based generator (splitmix64 of seed,
// step, field, slot), so a run is reproducible.
#include "../../include/wombat_gb300.h"
#include "wb_internal.h"
#include "wb_math.cuh"

#include <algorithm>
#include <vector>

namespace {

constexpr int NIN = 6, NH = 32, NOUT = 3;
constexpr int NP = WB_MLP_NPARAM;            // 1379
constexpr int NF = WB_MLP_NFIELD;            // 7
constexpr int REC = WB_MLP_RECORD;           // 12
constexpr int O_W1 = 0, O_B1 = O_W1 + NH * NIN, O_W2 = O_B1 + NH, O_B2 = O_W2 + NH * NH,
              O_W3 = O_B2 + NH, O_B3 = O_W3 + NOUT * NH;
static_assert(O_B3 + NOUT == NP, "parameter layout");

// One record's row in shared memory (floats): x(6) 1 h1(32) h2(32) da1(32)
// da2(32) dz(3) loss; every gradient entry is the sum over records of a
// product of two entries of the row (the biases' second factor is the 1).
constexpr int S_X = 0, S_ONE = 6, S_H1 = 8, S_H2 = 40, S_DA1 = 72, S_DA2 = 104, S_DZ = 136, S_L = 139,
              SROW = 140;
constexpr int NE = NP + 1;                   // entries per field: the parameters and the loss
constexpr int kChunk = 32;                   // records per pass of a block
constexpr int kGradThreads = 256;
// Blocks per field: two resident blocks per SM over seven fields, which cuts
// a 4 096-record batch into three chunks per block (three and four blocks per SM
// with 64 to 128 of them per field: 2 to 8 % slower per step).
constexpr int kGradBlocks = 43;

// GELU in its sigmoid form, gelu(t) = t sigma(1.702 t) = t/2 (1 + tanh(0.851 t)),
// and its derivative sigma + 1.702 t sigma (1 - sigma).
__device__ __forceinline__ float gelu(float t, float& dgelu) {
    const float sig = 0.5f * (1.0f + tanhf(0.851f * t));
    dgelu = sig + 1.702f * t * sig * (1.0f - sig);
    return t * sig;
}

__device__ __forceinline__ unsigned long long splitmix64(unsigned long long z) {
    z += 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

// Record index for (field, slot) of this step: either all records of the
// field in order (full batch) or a counter-based random draw.
__device__ __forceinline__ long long pick(const long long* off, const long long* cnt, int f,
                                          long long slot, int full, unsigned long long seed,
                                          long long step) {
    if (full) return off[f] + slot;
    const unsigned long long h =
        splitmix64(seed ^ splitmix64((unsigned long long)step * 131071ULL + (unsigned long long)f * 8191ULL +
                                     (unsigned long long)slot));
    return off[f] + (long long)(h % (unsigned long long)cnt[f]);
}

// Two entries' sums over one chunk, in the lanes of the packed FP32 instructions:
// each an unevaluated hi + mid + lo, += a b (nb = -b).  The product and every sum
// but lo's are split into their rounded value and its exact error (Dekker's and
// Knuth's error-free transformations), so a chunk's sum is good to 2^-72 of its
// magnitudes (errors of products below 2^-102 vanish: under half of the least
// FP32 number in a mean).  22 FP32 operations for two entries, 5.7 ms in
// the case below; FP64 fused multiply-adds on their 64 times narrower pipe take
// 8.5, and a pair hi + lo of ten operations takes 4.2 but loses four of
// FP64's bits.
struct Sum3 {
    float2 hi = {0.f, 0.f}, mid = {0.f, 0.f}, lo = {0.f, 0.f};
    static __device__ __forceinline__ float2 minus(float2 a, float2 b) {          // a - b
        return __ffma2_rn(b, make_float2(-1.f, -1.f), a);
    }
    // s += x, returns the rounding error
    static __device__ __forceinline__ float2 add_exact(float2& s, float2 x) {
        const float2 t = __fadd2_rn(s, x), z = minus(t, s), back = minus(s, minus(t, z));
        s = t;
        return __fadd2_rn(back, minus(x, z));
    }
    __device__ __forceinline__ void add(float2 a, float2 b, float2 nb) {
        const float2 n = __fmul2_rn(a, nb), e = __ffma2_rn(a, b, n);              // -p, a b - p
        const float2 t = minus(hi, n), z = minus(t, hi), back = minus(hi, minus(t, z));
        const float2 err = minus(back, __fadd2_rn(n, z));                         // + (p - z)
        hi = t;
        const float2 r = add_exact(mid, err);
        lo = __fadd2_rn(lo, __fadd2_rn(r, add_exact(mid, e)));
    }
};
// A lane of a chunk's sum in FP64; NaN where it left the FP32 range.
__device__ __forceinline__ double joined(float hi, float mid, float lo) {
    return wb::widen(hi) + (wb::widen(mid) + wb::widen(lo));
}

// The two factors of gradient entry j in a record's row.
__device__ __forceinline__ void entry_factors(int j, int& ga, int& gb) {
    gb = S_ONE;
    if (j < O_B1) { ga = S_DA1 + j / NIN; gb = S_X + j % NIN; }
    else if (j < O_W2) { ga = S_DA1 + (j - O_B1); }
    else if (j < O_B2) { ga = S_DA2 + (j - O_W2) / NH; gb = S_H1 + (j - O_W2) % NH; }
    else if (j < O_W3) { ga = S_DA2 + (j - O_B2); }
    else if (j < O_B3) { ga = S_DZ + (j - O_W3) / NH; gb = S_H2 + (j - O_W3) % NH; }
    else if (j < NP) { ga = S_DZ + (j - O_B3); }
    else { ga = S_L; }
}

// Block (field f, slot g of kGradBlocks): chunks g, g + kGradBlocks, ... of
// the field's batch.  A warp takes four of a chunk's 32 records through the
// network with one lane per hidden unit (weights in shared memory, rows
// padded so that rows and columns of W2 are both read without bank
// conflicts); then the block adds the chunk's outer products, a 2 x 2 tile of
// dW2 per thread and the 356 other entries one or two per thread.  Bound by
// the FP32 pipe: the exact sums are 22 of the 25 operations per two entries and
// record.  60 steps of 4 096 records per field and one full-batch gradient, host
// side included: 83.5 -> 5.7 ms against a serial loop over the records per entry
// with FP64 accumulators (and a loss copied to the host every step).
__global__ void __launch_bounds__(kGradThreads, 2)
grad_kernel(const float* __restrict__ rec, const long long* __restrict__ perm, const long long* __restrict__ off,
            const long long* __restrict__ cnt, const float* __restrict__ params, int batch, int full,
            unsigned long long seed, long long step, float lam, double* __restrict__ part) {
    __shared__ __align__(16) float row[kChunk][SROW];
    __shared__ __align__(16) float W1[NIN][NH], W2[NH][NH + 1], W3[NOUT][NH];
    __shared__ float B1[NH], B2[NH], B3[NOUT + 1];
    const int f = blockIdx.x / kGradBlocks, g = blockIdx.x - f * kGradBlocks;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float* p = params + (long long)f * NP;
    for (int j = tid; j < NP; j += kGradThreads) {
        const float v = p[j];
        if (j < O_B1) W1[j % NIN][j / NIN] = v;
        else if (j < O_W2) B1[j - O_B1] = v;
        else if (j < O_B2) W2[(j - O_W2) / NH][(j - O_W2) % NH] = v;
        else if (j < O_W3) B2[j - O_B2] = v;
        else if (j < O_B3) W3[(j - O_W3) / NH][(j - O_W3) % NH] = v;
        else B3[j - O_B3] = v;
    }
    if (tid < kChunk) row[tid][S_ONE] = 1.f;
    const long long n = cnt[f] == 0 ? 0 : (full ? cnt[f] : (long long)batch);
    // this thread's entries: rows 2 ti, 2 ti + 1 and columns 2 tk, 2 tk + 1 of
    // dW2, and entries e0, e1 of the rest (counted with dW2 left out)
    const int ti = tid >> 4, tk = tid & 15;
    constexpr int kRest = NE - NH * NH;
    static_assert(kChunk / (kGradThreads / 32) == 4, "four records per warp");
    static_assert(kRest > kGradThreads && kRest <= 2 * kGradThreads, "two further entries per thread at most");
    const int e0 = tid < O_W2 ? tid : tid + NH * NH, e1 = tid + kGradThreads + NH * NH;
    const bool two = tid + kGradThreads < kRest;
    int ga0, gb0, ga1, gb1;
    entry_factors(e0, ga0, gb0);
    entry_factors(two ? e1 : e0, ga1, gb1);
    double acc[6] = {0, 0, 0, 0, 0, 0};    // the chunks' sums: the tile by rows, e0, e1
    __syncthreads();
    for (long long c = (long long)g * kChunk; c < n; c += (long long)kGradBlocks * kChunk) {
        // forward and backward, four records per warp, lane = hidden unit
        constexpr int Q = kChunk / (kGradThreads / 32);
        float d1[Q], d2[Q];
        const int first = warp * Q;
        // lane q of the first four draws record q; slots past the batch repeat
        // its last record, and their rows are not summed
        const long long slot = c + first + lane;
        const float* rr = rec;
        if (lane < Q) rr += perm[pick(off, cnt, f, slot < n ? slot : n - 1, full, seed, step)] * REC;
        {
            // lane 8 q + k reads x_k of record q
            const float* r = reinterpret_cast<const float*>(
                __shfl_sync(0xffffffffu, (unsigned long long)rr, lane >> 3));
            if ((lane & 7) < NIN) row[first + (lane >> 3)][S_X + (lane & 7)] = r[1 + (lane & 7)];
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < Q; q++) {
            float a = B1[lane];
#pragma unroll
            for (int k = 0; k < NIN; k++) a += W1[k][lane] * row[first + q][S_X + k];
            row[first + q][S_H1 + lane] = gelu(a, d1[q]);
        }
        __syncwarp();
        {
            float a[Q];
#pragma unroll
            for (int q = 0; q < Q; q++) a[q] = B2[lane];
#pragma unroll
            for (int k = 0; k < NH; k += 4) {
                const float w[4] = {W2[lane][k], W2[lane][k + 1], W2[lane][k + 2], W2[lane][k + 3]};
#pragma unroll
                for (int q = 0; q < Q; q++) {
                    const float4 h = *reinterpret_cast<const float4*>(&row[first + q][S_H1 + k]);
                    a[q] += w[0] * h.x;
                    a[q] += w[1] * h.y;
                    a[q] += w[2] * h.z;
                    a[q] += w[3] * h.w;
                }
            }
#pragma unroll
            for (int q = 0; q < Q; q++) {
                row[first + q][S_H2 + lane] = gelu(a[q], d2[q]);
            }
        }
        __syncwarp();
        // output layer: lane 3 q + o sums output o of record q over the hidden
        // units in their order
        float zo = 0.f;
        if (lane < Q * NOUT) {
            const int q = lane / NOUT, o = lane - q * NOUT;
            zo = B3[o];
#pragma unroll
            for (int k = 0; k < NH; k += 4) {
                const float4 h = *reinterpret_cast<const float4*>(&row[first + q][S_H2 + k]);
                const float4 w = *reinterpret_cast<const float4*>(&W3[o][k]);
                zo += w.x * h.x;
                zo += w.y * h.y;
                zo += w.z * h.z;
                zo += w.w * h.w;
            }
        }
        float zz[NOUT];
#pragma unroll
        for (int o = 0; o < NOUT; o++) zz[o] = __shfl_sync(0xffffffffu, zo, (lane < Q ? NOUT * lane : 0) + o);
        // softmax, loss and its gradient: lane q of the first four takes record q
        float dz[NOUT] = {0.f, 0.f, 0.f};
        if (lane < Q) {
            const float zm = fmaxf(zz[0], fmaxf(zz[1], zz[2]));
            float e[NOUT], es = 0.f;
#pragma unroll
            for (int o = 0; o < NOUT; o++) { e[o] = expf(zz[o] - zm); es += e[o]; }
            float om[NOUT];
#pragma unroll
            for (int o = 0; o < NOUT; o++) om[o] = e[o] / es;
            const float qv[NOUT] = {rr[7], rr[8], rr[9]};
            const float T = rr[10];
            const float d[NOUT] = {0.1f, 0.6f, 0.3f};
            const float y = om[0] * qv[0] + om[1] * qv[1] + om[2] * qv[2];
            float kl = 0.f;
#pragma unroll
            for (int o = 0; o < NOUT; o++) kl += d[o] * (logf(d[o]) - logf(om[o]));
            float dom[NOUT], sdom = 0.f;
#pragma unroll
            for (int o = 0; o < NOUT; o++) {
                dom[o] = 2.f * (y - T) * qv[o] - lam * d[o] / om[o];
                sdom += om[o] * dom[o];
            }
#pragma unroll
            for (int o = 0; o < NOUT; o++) {
                dz[o] = om[o] * (dom[o] - sdom);
                row[first + lane][S_DZ + o] = dz[o];
            }
            row[first + lane][S_L] = (y - T) * (y - T) + lam * kl;
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < Q; q++) {
            float a = 0.f;
#pragma unroll
            for (int o = 0; o < NOUT; o++) a += row[first + q][S_DZ + o] * W3[o][lane];
            row[first + q][S_DA2 + lane] = a * d2[q];
        }
        __syncwarp();
        {
            float a[Q];
#pragma unroll
            for (int q = 0; q < Q; q++) a[q] = 0.f;
#pragma unroll
            for (int i = 0; i < NH; i += 4) {
                const float w[4] = {W2[i][lane], W2[i + 1][lane], W2[i + 2][lane], W2[i + 3][lane]};
#pragma unroll
                for (int q = 0; q < Q; q++) {
                    const float4 h = *reinterpret_cast<const float4*>(&row[first + q][S_DA2 + i]);
                    a[q] += w[0] * h.x;
                    a[q] += w[1] * h.y;
                    a[q] += w[2] * h.z;
                    a[q] += w[3] * h.w;
                }
            }
#pragma unroll
            for (int q = 0; q < Q; q++) row[first + q][S_DA1 + lane] = a[q] * d1[q];
        }
        __syncthreads();
        const int m = n - c < kChunk ? (int)(n - c) : kChunk;
        Sum3 top, bot, rest;       // the tile's two rows, and e0 with e1
#pragma unroll 2
        for (int q = 0; q < m; q++) {
            const float* w = row[q];
            const float2 da = *reinterpret_cast<const float2*>(w + S_DA2 + 2 * ti);
            const float2 h = *reinterpret_cast<const float2*>(w + S_H1 + 2 * tk);
            const float2 nh = make_float2(-h.x, -h.y);
            top.add(make_float2(da.x, da.x), h, nh);
            bot.add(make_float2(da.y, da.y), h, nh);
            const float2 f = make_float2(w[gb0], w[gb1]);
            rest.add(make_float2(w[ga0], w[ga1]), f, make_float2(-f.x, -f.y));
        }
        double sum[6] = {joined(top.hi.x, top.mid.x, top.lo.x),    joined(top.hi.y, top.mid.y, top.lo.y),
                         joined(bot.hi.x, bot.mid.x, bot.lo.x),    joined(bot.hi.y, bot.mid.y, bot.lo.y),
                         joined(rest.hi.x, rest.mid.x, rest.lo.x), joined(rest.hi.y, rest.mid.y, rest.lo.y)};
#pragma unroll
        for (int k = 0; k < 6; k++) {
            if (!isfinite(sum[k])) {                   // out of the FP32 range, infinite or NaN
                const int ga = k < 4 ? S_DA2 + 2 * ti + (k >> 1) : (k == 4 ? ga0 : ga1);
                const int gb = k < 4 ? S_H1 + 2 * tk + (k & 1) : (k == 4 ? gb0 : gb1);
                sum[k] = 0.0;
                for (int q = 0; q < m; q++) sum[k] = fma(double(row[q][ga]), double(row[q][gb]), sum[k]);
            }
            acc[k] += sum[k];
        }
        __syncthreads();
    }
    double* o = part + (long long)blockIdx.x * NE;
    const int j = O_W2 + 2 * ti * NH + 2 * tk;
    o[j] = acc[0];
    o[j + 1] = acc[1];
    o[j + NH] = acc[2];
    o[j + NH + 1] = acc[3];
    o[e0] = acc[4];
    if (two) o[e1] = acc[5];
}

// Gradient entry j of field f: the blocks' sums added in FP64 in the order of
// the blocks, over the number of records; entry NP is the loss.  With m given
// also the parameter's Adam step.
__global__ void __launch_bounds__(64)
apply_kernel(const double* __restrict__ part, const long long* __restrict__ cnt, int batch, int full,
             float* __restrict__ grad, float* __restrict__ loss, float* __restrict__ params, float* __restrict__ m,
             float* __restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2) {
    const int gid = blockIdx.x * blockDim.x + threadIdx.x;
    const int f = gid / NE, j = gid - f * NE;
    if (f >= NF) return;
    const long long n = cnt[f] == 0 ? 0 : (full ? cnt[f] : (long long)batch);
    const double* s = part + (long long)f * kGradBlocks * NE + j;
    double sum = 0.0;
#pragma unroll
    for (int b = 0; b < kGradBlocks; b++) sum += s[(long long)b * NE];
    const float g = float(n > 0 ? sum / double(n) : 0.0);
    if (j == NP) {
        loss[f] = g;
        return;
    }
    const int i = f * NP + j;
    grad[i] = g;
    if (!m) return;
    const float mi = b1 * m[i] + (1.f - b1) * g;
    const float vi = b2 * v[i] + (1.f - b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    params[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// Device buffers of one call, cut from one allocation.
struct Dev {
    char* all = nullptr;
    float* rec = nullptr;
    long long* perm = nullptr;     // the records to train on, by field, in their order
    long long* off = nullptr;      // 7 offsets, then 7 counts
    long long* cnt = nullptr;
    float* params = nullptr;
    float* grad = nullptr;
    float* m = nullptr;            // Adam's moments, m then v
    float* v = nullptr;
    double* part = nullptr;        // the blocks' sums
    float* loss = nullptr;         // 7 per step
    ~Dev() {
        if (all) cudaFree(all);
    }
};

// Uploads the records, the order of the unflagged ones by field, and the
// parameters; room for the losses of `steps` steps.
int setup(Dev& D, const float* records, long long n, const float* params, long long steps, int full,
          long long* cnt_out) {
    std::vector<long long> cnt(NF, 0), off(NF, 0);
    for (long long r = 0; r < n; r++) {
        const int f = (int)records[r * REC];
        if (f < 0 || f >= NF) return wb::set_last_error(WB_EINVAL, "mlp: record with a field outside 0..6");
        if (records[r * REC + 11] == 0.f) cnt[f]++;
    }
    long long pos = 0;
    for (int f = 0; f < NF; f++) {
        off[f] = pos;
        pos += cnt[f];
        cnt_out[f] = cnt[f];
    }
    std::vector<long long> perm(std::max<long long>(pos, 1), 0), at = off;
    for (long long r = 0; r < n; r++)
        if (records[r * REC + 11] == 0.f) perm[at[(int)records[r * REC]]++] = r;
    if (full && *std::max_element(cnt.begin(), cnt.end()) > (1LL << 24))
        return wb::set_last_error(WB_EINVAL, "mlp: too many records per field");
    size_t used = 0;
    auto place = [&](size_t bytes) {
        const size_t at = used;
        used += (bytes + 255) & ~size_t(255);
        return at;
    };
    const size_t np = sizeof(float) * NF * NP;
    const size_t rec = place(sizeof(float) * n * REC), prm = place(sizeof(long long) * perm.size()),
                 tab = place(sizeof(long long) * 2 * NF), par = place(np), grd = place(np), mom = place(2 * np),
                 prt = place(sizeof(double) * NE * NF * kGradBlocks),
                 los = place(sizeof(float) * NF * std::max<long long>(steps, 1));
    if (cudaMalloc(&D.all, used) != cudaSuccess) {
        cudaGetLastError();
        return wb::set_last_error(WB_ENOMEM, "mlp: device allocation failed");
    }
    D.rec = reinterpret_cast<float*>(D.all + rec);
    D.perm = reinterpret_cast<long long*>(D.all + prm);
    D.off = reinterpret_cast<long long*>(D.all + tab);
    D.cnt = D.off + NF;
    D.params = reinterpret_cast<float*>(D.all + par);
    D.grad = reinterpret_cast<float*>(D.all + grd);
    D.m = reinterpret_cast<float*>(D.all + mom);
    D.v = D.m + NF * NP;
    D.part = reinterpret_cast<double*>(D.all + prt);
    D.loss = reinterpret_cast<float*>(D.all + los);
    long long table[2 * NF];
    for (int f = 0; f < NF; f++) {
        table[f] = off[f];
        table[NF + f] = cnt[f];
    }
    if (cudaMemcpy(D.rec, records, sizeof(float) * n * REC, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(D.perm, perm.data(), sizeof(long long) * perm.size(), cudaMemcpyHostToDevice) != cudaSuccess)
        return wb::set_last_error(WB_ECUDA, "mlp: record upload failed");
    if (cudaMemcpy(D.off, table, sizeof(table), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(D.params, params, np, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(D.m, 0, 2 * np) != cudaSuccess)
        return wb::set_last_error(WB_ECUDA, "mlp: upload failed");
    return WB_OK;
}

struct Adam {
    float lr = 0.f, b1 = 0.9f, b2 = 0.999f, eps = 1e-8f, c1 = 1.f, c2 = 1.f;
};

// Gradient and loss of one batch; with `adam` also the parameters' step.
int grad_step(Dev& D, int batch, int full, unsigned long long seed, long long step, float lam, float* loss,
              const Adam* adam) {
    grad_kernel<<<NF * kGradBlocks, kGradThreads>>>(D.rec, D.perm, D.off, D.cnt, D.params, batch, full, seed, step,
                                                    lam, D.part);
    const Adam a = adam ? *adam : Adam{};
    apply_kernel<<<(NF * NE + 63) / 64, 64>>>(D.part, D.cnt, batch, full, D.grad, loss, D.params,
                                              adam ? D.m : nullptr, D.v, a.lr, a.b1, a.b2, a.eps, a.c1, a.c2);
    return cudaGetLastError() == cudaSuccess ? WB_OK : wb::set_last_error(WB_ECUDA, "mlp: kernel launch failed");
}

}  // namespace

extern "C" int wb_mlp_loss_grad(const float* records, long long n, const float* params, double lam,
                                double* loss_out, float* grad_out) {
    if (!records || n < 1 || !params || !loss_out || !grad_out)
        return wb::set_last_error(WB_EINVAL, "mlp: null argument or no records");
    Dev D;
    long long cnt[NF];
    int rc = setup(D, records, n, params, 1, 1, cnt);
    if (rc != WB_OK) return rc;
    if ((rc = grad_step(D, 0, 1, 0, 0, (float)lam, D.loss, nullptr)) != WB_OK) return rc;
    float loss[NF];
    if (cudaMemcpy(grad_out, D.grad, sizeof(float) * NF * NP, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(loss, D.loss, sizeof(float) * NF, cudaMemcpyDeviceToHost) != cudaSuccess)
        return wb::set_last_error(WB_ECUDA, "mlp: download failed");
    for (int f = 0; f < NF; f++) loss_out[f] = loss[f];
    return wb::set_last_error(WB_OK, "");
}

extern "C" int wb_mlp_train(const float* records, long long n, float* params, int steps, int batch,
                            double lr, double lam, unsigned long long seed, float* loss_history) {
    if (!records || n < 1 || !params || steps < 0 || batch < 1 || batch > (1 << 20) || !(lr > 0))
        return wb::set_last_error(WB_EINVAL, "mlp: bad training arguments");
    Dev D;
    long long cnt[NF];
    int rc = setup(D, records, n, params, loss_history ? steps : 1, 0, cnt);
    if (rc != WB_OK) return rc;
    Adam adam;
    adam.lr = (float)lr;
    double p1 = 1.0, p2 = 1.0;
    for (int t = 0; t < steps; t++) {
        p1 *= adam.b1;
        p2 *= adam.b2;
        adam.c1 = (float)(1.0 - p1);
        adam.c2 = (float)(1.0 - p2);
        float* loss = D.loss + (loss_history ? (long long)t * NF : 0);
        if ((rc = grad_step(D, batch, 0, seed, t, (float)lam, loss, &adam)) != WB_OK) return rc;
    }
    // the losses stay on the device until the last step: one copy, one wait
    if (loss_history && steps > 0 &&
        cudaMemcpy(loss_history, D.loss, sizeof(float) * NF * steps, cudaMemcpyDeviceToHost) != cudaSuccess)
        return wb::set_last_error(WB_ECUDA, "mlp: loss download failed");
    if (cudaMemcpy(params, D.params, sizeof(float) * NF * NP, cudaMemcpyDeviceToHost) != cudaSuccess)
        return wb::set_last_error(WB_ECUDA, "mlp: parameter download failed");
    return wb::set_last_error(WB_OK, "");
}
