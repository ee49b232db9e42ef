// mlp.cu -- the learned variant selector's device code: the row_ptr feature
// kernel and the FP32 forward, backward and Adam kernels of a small
// multilayer perceptron (ReLU hidden layers, linear outputs, squared loss).
// Not in the paper: the selector only picks among the library's kernels and
// never changes their arithmetic.
#include <cuda_runtime.h>

#include <cmath>

#include "launch.cuh"

namespace ssspmv {

// ---------------------------------------------------------------------------
// features: one pass over the row lengths, block partial sums into 64-bit
// global counters, which the last block turns into the 16 features

constexpr int kFeatThreads = 256;
constexpr int kHistBins = 32;  // bin b: row length in [2^(b-1), 2^b), bin 0: empty

// counter layout (unsigned long long)
enum {
    FC_SUM2 = 0,        // sum of len^2
    FC_MAX,             // max len
    FC_EMPTY,           // empty rows
    FC_SHORT,           // rows with len <= 4
    FC_HEAVY,           // rows with len >= 2 * mean
    FC_LONGNNZ,         // entries in rows longer than 1024
    FC_JUMP,            // rows whose length differs from the previous row's by more than 2x
    FC_EMPTYRUN,        // empty rows followed by an empty row
    FC_XNNZ,            // entries in rows of at least 32 * mean
    FC_HIST,            // kHistBins counters
    FC_COUNT = FC_HIST + kHistBins
};

__device__ __forceinline__ int len_bin(int32_t len)
{
    return len <= 0 ? 0 : (32 - __clz((unsigned)len) < kHistBins ? 32 - __clz((unsigned)len)
                                                                  : kHistBins - 1);
}

// the features that m and nnz alone decide
struct HostFeatures {
    double mean;
    float f0, f1, f2, f13;
};

// All counters in one pass over row_ptr (the mean, and with it the thresholds
// t2 = ceil(2 mean) and t32 = ceil(32 mean), is nnz / m and needs none), then
// the last block to finish turns them into the features.  A warp takes 32 rows
// at a time, one load per row; its bound is instruction issue, so each thread
// keeps its own counts, and each warp its own histogram in shared memory.
// (64-bit shared atomics per row, two passes and a single thread's FP64
// divisions and logarithms at the end took 250 us of 2^21 rows; this takes 16,
// 10 of them whatever the size.)  The upper half of FC_SHORT counts the blocks
// that are done.
__global__ void __launch_bounds__(kFeatThreads)
    feature_kernel(const int32_t *__restrict__ row_ptr, int32_t m, int32_t nnz, uint32_t t2,
                   uint32_t t32, const HostFeatures host, unsigned long long *__restrict__ cnt,
                   float *__restrict__ f)
{
    constexpr int WARPS = kFeatThreads / 32;
    __shared__ unsigned long long s[FC_COUNT];
    __shared__ uint32_t s_hist[WARPS][kHistBins];
    __shared__ bool s_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < FC_COUNT; i += blockDim.x) s[i] = 0ull;
    s_hist[warp][lane] = 0u;
    __syncthreads();
    unsigned long long sum2 = 0, longnnz = 0, xnnz = 0;
    int32_t mx = 0;
    uint32_t empty = 0, shrt = 0, heavy = 0, jump = 0, erun = 0;
    // (indices stay below 2^32: m is below 2^31, and so are U strides)
    const uint32_t stride = gridDim.x * WARPS * 32u, rows = (uint32_t)m;
    constexpr int U = 4;  // chunks of 32 rows in flight
    for (uint32_t c = (blockIdx.x * WARPS + warp) * 32u; c < rows; c += U * stride) {
        int32_t a[U], edge[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t r = c + u * stride + lane;
            a[u] = edge[u] = 0;
            if (r <= rows) a[u] = __ldg(row_ptr + r);
            // lane 0: the row before the chunk's; lane 31: the chunk's end
            if (lane == 0 && r > 0 && r <= rows) edge[u] = __ldg(row_ptr + r - 1);
            if (lane == 31 && r < rows) edge[u] = __ldg(row_ptr + r + 1);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t r = c + u * stride + lane;
            int32_t b = __shfl_down_sync(FULL, a[u], 1);
            int32_t before = __shfl_up_sync(FULL, a[u], 1);
            if (lane == 31) b = edge[u];
            if (lane == 0) before = edge[u];
            if (r >= rows) continue;
            const int32_t len = b - a[u], p = a[u] - before;  // p: the previous row's length
            sum2 += (unsigned long long)(uint32_t)len * (uint32_t)len;
            mx = max(mx, len);
            if (len > 1024) longnnz += (uint32_t)len;
            if ((uint32_t)len >= t32) xnnz += (uint32_t)len;
            if (len == 0) ++empty;
            if (len <= 4) ++shrt;
            if ((uint32_t)len >= t2) ++heavy;
            if (r > 0) {
                if (len > 2 * p + 1 || p > 2 * len + 1) ++jump;
                if (len == 0 && p == 0) ++erun;
            }
            atomicAdd(&s_hist[warp][len_bin(len)], 1u);
        }
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        sum2 += __shfl_xor_sync(FULL, sum2, d);
        longnnz += __shfl_xor_sync(FULL, longnnz, d);
        xnnz += __shfl_xor_sync(FULL, xnnz, d);
    }
    mx = __reduce_max_sync(FULL, mx);
    empty = __reduce_add_sync(FULL, empty);
    shrt = __reduce_add_sync(FULL, shrt);
    heavy = __reduce_add_sync(FULL, heavy);
    jump = __reduce_add_sync(FULL, jump);
    erun = __reduce_add_sync(FULL, erun);
    if (lane == 0) {
        atomicAdd(&s[FC_SUM2], sum2);
        atomicMax(&s[FC_MAX], (unsigned long long)mx);
        atomicAdd(&s[FC_EMPTY], (unsigned long long)empty);
        atomicAdd(&s[FC_SHORT], (unsigned long long)shrt);
        atomicAdd(&s[FC_HEAVY], (unsigned long long)heavy);
        atomicAdd(&s[FC_LONGNNZ], longnnz);
        atomicAdd(&s[FC_JUMP], (unsigned long long)jump);
        atomicAdd(&s[FC_EMPTYRUN], (unsigned long long)erun);
        atomicAdd(&s[FC_XNNZ], xnnz);
    }
    __syncthreads();
    if (threadIdx.x < kHistBins) {
        unsigned long long h = 0;
        for (int w = 0; w < WARPS; ++w) h += s_hist[w][threadIdx.x];
        s[FC_HIST + threadIdx.x] = h;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < FC_COUNT; i += blockDim.x) {
        if (i == FC_MAX) atomicMax(cnt + i, s[i]);
        else if (s[i]) atomicAdd(cnt + i, s[i]);
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0)
        s_last = (uint32_t)(atomicAdd(cnt + FC_SHORT, 1ull << 32) >> 32) == gridDim.x - 1u;
    __syncthreads();
    if (!s_last || warp > 2) return;
    __threadfence();

    // ---- the features.  A lone warp's FP64 instructions are 65 cycles apart, so
    // what depends on m and nnz alone comes from the host, and the rest goes by
    // three warps: ratios (one division for all lanes), the logarithm, the
    // percentiles
    const double md = m > 0 ? (double)m : 1.0, nz = nnz > 0 ? (double)nnz : 1.0;
    if (warp == 0) {
        int which = FC_EMPTY;  // lane 5
        if (lane == 3) which = FC_SUM2;
        if (lane == 6) which = FC_SHORT;
        if (lane == 7) which = FC_HEAVY;
        if (lane == 8) which = FC_LONGNNZ;
        if (lane == 12) which = FC_JUMP;
        if (lane == 14) which = FC_EMPTYRUN;
        if (lane == 15) which = FC_XNNZ;
        unsigned long long c = __ldcg(cnt + which);
        if (lane == 6) c &= 0xffffffffull;
        double v = (double)c / (lane == 8 || lane == 15 ? nz : md);
        if (lane == 3) {
            const double var = v - host.mean * host.mean;
            v = (var > 0 ? sqrt(var) : 0.0) / (host.mean + 1.0);
        }
        if (lane == 3 || (lane >= 5 && lane <= 8) || lane == 12 || lane == 14 || lane == 15)
            f[lane] = (float)v;
    } else if (warp == 1) {
        if (lane == 0) f[0] = host.f0;
        if (lane == 1) f[1] = host.f1;
        if (lane == 2) f[2] = host.f2;
        if (lane == 13) f[13] = host.f13;
        if (lane == 4) f[4] = (float)(log2((double)__ldcg(cnt + FC_MAX) + 1.0) / 24.0);
    } else {
        // the first bin of the histogram at which the count reaches q * m
        unsigned long long cum = __ldcg(cnt + FC_HIST + lane);
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned long long o = __shfl_up_sync(FULL, cum, d);
            if (lane >= d) cum += o;
        }
        const double qs = lane == 9 ? 0.5 : (lane == 10 ? 0.9 : 0.99);
        const double want = qs * md, have = (double)cum;
        for (int k = 9; k < 12; ++k) {
            const unsigned hit = __ballot_sync(FULL, have >= __shfl_sync(FULL, want, k));
            if (lane == k) f[k] = (float)(hit ? __ffs(hit) - 1 : 0) / 16.0f;
        }
    }
}

// the smallest row length at least k times the mean (as FP64 compares them)
static uint32_t at_least(double k, double mean)
{
    const double t = std::ceil(k * mean);
    return t >= 4294967295.0 ? 0xffffffffu : (uint32_t)t;
}

int run_features(const int32_t *row_ptr, int32_t m, int32_t n, int32_t nnz, float *out,
                 void *scratch, cudaStream_t s)
{
    (void)n;
    unsigned long long *cnt = static_cast<unsigned long long *>(scratch);
    cudaError_t e = cudaMemsetAsync(cnt, 0, sizeof(unsigned long long) * FC_COUNT, s);
    if (e != cudaSuccess) return record_cuda_error(e);
    // four chunks of 32 rows per warp, four blocks per SM at most (the blocks
    // meet in the counters' atomics)
    int64_t blocks = ((int64_t)m + 4 * kFeatThreads - 1) / (4 * kFeatThreads);
    const int64_t cap = 4LL * device_sm_count();
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    const double mean = m > 0 ? (double)nnz / (double)m : 0.0;
    const double md = m > 0 ? (double)m : 1.0;
    HostFeatures h;
    h.mean = (double)nnz / md;
    h.f0 = (float)(std::log2(md + 1.0) / 24.0);
    h.f1 = (float)(std::log2((double)nnz + 1.0) / 32.0);
    h.f2 = (float)(std::log2(h.mean + 1.0) / 8.0);
    h.f13 = (float)(std::log2(480.0 / (h.mean + 1e-9) + 1.0) / 16.0);  // rows per 480-entry tile
    feature_kernel<<<(unsigned)blocks, kFeatThreads, 0, s>>>(
        row_ptr, m, nnz, at_least(2.0, mean), at_least(32.0, mean), h, cnt, out);
    e = cudaGetLastError();
    if (e != cudaSuccess) return record_cuda_error(e);
    return SSSPMV_OK;
}

size_t features_scratch_bytes() { return sizeof(unsigned long long) * FC_COUNT; }

// ---------------------------------------------------------------------------
// dense layers of the perceptron, FP32.  Weights row-major W[O][I].

constexpr int kMlpThreads = 256;

// out[b][o] = act(sum_i W[o][i] * in[b][i] + bias[o]); pre[b][o] keeps the
// pre-activation for the backward pass (may be null)
__global__ void __launch_bounds__(kMlpThreads)
    dense_forward_kernel(const float *__restrict__ in, const float *__restrict__ Wt,
                         const float *__restrict__ bias, float *__restrict__ pre,
                         float *__restrict__ out, int B, int I, int O, int relu)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (int64_t)B * O) return;
    const int b = (int)(k / O), o = (int)(k % O);
    float acc = bias[o];
    for (int i = 0; i < I; ++i) acc = fmaf(Wt[o * I + i], in[(int64_t)b * I + i], acc);
    if (pre) pre[k] = acc;
    out[k] = relu ? fmaxf(acc, 0.0f) : acc;
}

// squared loss over the outputs whose target is finite (mask: target NaN =
// not measured): g = 2 (out - target) / count, loss accumulated in *loss
__global__ void __launch_bounds__(kMlpThreads)
    loss_grad_kernel(const float *__restrict__ out, const float *__restrict__ target,
                     float *__restrict__ g, int64_t n, float inv_count, float *loss)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    float l = 0.0f;
    if (k < n) {
        const float t = target[k];
        const float d = (t == t) ? out[k] - t : 0.0f;
        g[k] = 2.0f * d * inv_count;
        l = d * d * inv_count;
    }
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1) l += __shfl_xor_sync(FULL, l, s);
    if ((threadIdx.x & 31) == 0 && l != 0.0f) atomicAdd(loss, l);
}

// dW[o][i] = sum_b g[b][o] * in[b][i];  db[o] = sum_b g[b][o]  (one thread
// per weight, a fixed order over the batch: deterministic)
__global__ void __launch_bounds__(kMlpThreads)
    dense_grad_w_kernel(const float *__restrict__ in, const float *__restrict__ g,
                        float *__restrict__ dW, float *__restrict__ db, int B, int I, int O)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < (int64_t)O * I) {
        const int o = (int)(k / I), i = (int)(k % I);
        float acc = 0.0f;
        for (int b = 0; b < B; ++b) acc = fmaf(g[(int64_t)b * O + o], in[(int64_t)b * I + i], acc);
        dW[k] = acc;
    } else if (k < (int64_t)O * I + O) {
        const int o = (int)(k - (int64_t)O * I);
        float acc = 0.0f;
        for (int b = 0; b < B; ++b) acc += g[(int64_t)b * O + o];
        db[o] = acc;
    }
}

// gin[b][i] = (sum_o W[o][i] * g[b][o]) * (pre_in[b][i] > 0)  (ReLU below)
__global__ void __launch_bounds__(kMlpThreads)
    dense_grad_in_kernel(const float *__restrict__ Wt, const float *__restrict__ g,
                         const float *__restrict__ pre_in, float *__restrict__ gin, int B, int I,
                         int O)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (int64_t)B * I) return;
    const int b = (int)(k / I), i = (int)(k % I);
    float acc = 0.0f;
    for (int o = 0; o < O; ++o) acc = fmaf(Wt[o * I + i], g[(int64_t)b * O + o], acc);
    gin[k] = pre_in[k] > 0.0f ? acc : 0.0f;
}

// Adam (Kingma & Ba 2015) on n parameters, step t >= 1
__global__ void __launch_bounds__(kMlpThreads)
    adam_kernel(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m1,
                float *__restrict__ m2, int64_t n, float lr, float b1, float b2, float eps,
                float wd, int t)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    grid_dep_wait();  // the gradient comes from the kernel before
    grid_dep_trigger();
    if (k >= n) return;
    const float gk = g[k] + wd * p[k];
    const float a = b1 * m1[k] + (1.0f - b1) * gk;
    const float v = b2 * m2[k] + (1.0f - b2) * gk * gk;
    m1[k] = a;
    m2[k] = v;
    const float ah = a / (1.0f - powf(b1, (float)t));
    const float vh = v / (1.0f - powf(b2, (float)t));
    p[k] -= lr * ah / (sqrtf(vh) + eps);
}

// argmin over each row of the predictions (the chosen class)
__global__ void argmin_kernel(const float *__restrict__ out, int B, int K, int32_t *__restrict__ cls)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    int best = 0;
    float bv = out[(int64_t)b * K];
    for (int k = 1; k < K; ++k) {
        const float v = out[(int64_t)b * K + k];
        if (v < bv) {
            bv = v;
            best = k;
        }
    }
    cls[b] = best;
}

// ---------------------------------------------------------------------------
// The selector's own sizes (64 units in both hidden layers, up to 32 features
// and classes) in one kernel: a block takes kMlpTile samples through all
// layers with every weight and activation in shared memory, and for training
// back again, leaving its samples' share of the weight gradients in `parts`;
// mlp_reduce_kernel adds the blocks' shares in order.  One layer per launch
// and one thread per weight over the whole batch took 960 us for a training
// step on 2,000 samples, nearly all of it the weight gradients' serial sums;
// this takes 14.

constexpr int kMlpH = 64, kMlpMaxF = 32, kMlpMaxK = 32, kMlpTile = 16;
constexpr int kMlpLd = kMlpH + 4;  // rows of 64 a bank group apart, 16-byte aligned

struct MlpSmem {
    float W1t[kMlpMaxF][kMlpLd];  // W1t[i][o] = W1[o][i]
    float W2t[kMlpH][kMlpLd];
    float W2[kMlpH][kMlpLd];
    float W3[kMlpMaxK][kMlpLd];
    float b1[kMlpH], b2[kMlpH], b3[kMlpMaxK];
    float X[kMlpTile][kMlpMaxF];
    float a1[kMlpTile][kMlpLd], a2[kMlpTile][kMlpLd];
    float g2[kMlpTile][kMlpLd], g1[kMlpTile][kMlpLd];
    float o3[kMlpTile][kMlpMaxK], g3[kMlpTile][kMlpMaxK];
};

struct MlpArgs {
    const float *params, *X;
    float *out, *out2;     // predictions (out2 nullable)
    int32_t *cls;          // nullable: the least prediction's class
    const float *target;   // training: nullable otherwise
    float *parts;          // training: [blocks][count + 1], the last the loss
    float inv_count;
    int32_t B, F, K, count;
};

// acc[q] += W[i][o] * in[b + 4 q][i] over i < n in order (n a multiple of 4)
__device__ __forceinline__ void mlp_dot4(float (&acc)[4], const float (*W)[kMlpLd], int o,
                                         const float *in, int ld, int n)
{
#pragma unroll 4
    for (int i = 0; i < n; i += 4) {
        const float w0 = W[i][o], w1 = W[i + 1][o], w2 = W[i + 2][o], w3 = W[i + 3][o];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 v = *reinterpret_cast<const float4 *>(in + 4 * q * ld + i);
            acc[q] = fmaf(w0, v.x, acc[q]);
            acc[q] = fmaf(w1, v.y, acc[q]);
            acc[q] = fmaf(w2, v.z, acc[q]);
            acc[q] = fmaf(w3, v.w, acc[q]);
        }
    }
}

__global__ void __launch_bounds__(kMlpThreads) mlp_kernel(const MlpArgs a)
{
    extern __shared__ __align__(16) unsigned char mlp_smem[];
    __shared__ float s_loss[kMlpThreads / 32];
    MlpSmem &s = *reinterpret_cast<MlpSmem *>(mlp_smem);
    constexpr int H = kMlpH;
    const int t = threadIdx.x, F = a.F, K = a.K;
    const float *W1 = a.params, *b1 = W1 + H * F, *W2 = b1 + H, *b2 = W2 + H * H, *W3 = b2 + H,
                *b3 = W3 + K * H;
    grid_dep_wait();  // the parameters may come from the kernel before
    grid_dep_trigger();
    for (int k = t; k < H * F; k += kMlpThreads) s.W1t[k % F][k / F] = __ldg(W1 + k);
    float w2[H * H / kMlpThreads];  // all on their way at once
#pragma unroll
    for (int q = 0; q < H * H / kMlpThreads; ++q) w2[q] = __ldg(W2 + t + q * kMlpThreads);
#pragma unroll
    for (int q = 0; q < H * H / kMlpThreads; ++q) {
        const int k = t + q * kMlpThreads;
        s.W2[k / H][k % H] = w2[q];
        s.W2t[k % H][k / H] = w2[q];
    }
    for (int k = t; k < K * H; k += kMlpThreads) s.W3[k / H][k % H] = __ldg(W3 + k);
    if (t < H) {
        s.b1[t] = __ldg(b1 + t);
        s.b2[t] = __ldg(b2 + t);
    }
    if (t < K) s.b3[t] = __ldg(b3 + t);
    // tiles of samples (training: more than one where the scratch holds the
    // shares of fewer blocks than there are tiles)
    for (int b0 = blockIdx.x * kMlpTile; b0 < a.B; b0 += gridDim.x * kMlpTile) {
        const bool first = b0 == (int)blockIdx.x * kMlpTile;
        auto add = [&](float *at, float v) { *at = first ? v : *at + v; };
        __syncthreads();  // the tile before is done with
        for (int k = t; k < kMlpTile * F; k += kMlpThreads)
            s.X[k / F][k % F] = b0 + k / F < a.B ? __ldg(a.X + (int64_t)b0 * F + k) : 0.0f;
        __syncthreads();
        // hidden layers: a thread takes one unit of samples sb, sb + 4, ..
        const int o = t % H, sb = t / H;
        float acc[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = s.b1[o];
        mlp_dot4(acc, s.W1t, o, s.X[sb], kMlpMaxF, F);
#pragma unroll
        for (int q = 0; q < 4; ++q) s.a1[sb + 4 * q][o] = fmaxf(acc[q], 0.0f);
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = s.b2[o];
        mlp_dot4(acc, s.W2t, o, s.a1[sb], kMlpLd, H);
#pragma unroll
        for (int q = 0; q < 4; ++q) s.a2[sb + 4 * q][o] = fmaxf(acc[q], 0.0f);
        __syncthreads();
        float loss = 0.0f;
        for (int k = t; k < kMlpTile * K; k += kMlpThreads) {
            const int b = k / K, c = k % K;
            float v = s.b3[c];
#pragma unroll
            for (int i = 0; i < H; i += 4) {
                const float4 w = *reinterpret_cast<const float4 *>(&s.W3[c][i]);
                const float4 h = *reinterpret_cast<const float4 *>(&s.a2[b][i]);
                v = fmaf(w.x, h.x, v);
                v = fmaf(w.y, h.y, v);
                v = fmaf(w.z, h.z, v);
                v = fmaf(w.w, h.w, v);
            }
            s.o3[b][c] = v;
            float g = 0.0f;
            if (b0 + b < a.B) {
                const int64_t at = (int64_t)(b0 + b) * K + c;
                if (a.out) a.out[at] = v;
                if (a.out2) a.out2[at] = v;
                if (a.target) {
                    // a NaN target (a class not measured) counts as no error
                    const float y = __ldg(a.target + at);
                    const float d = (y == y) ? v - y : 0.0f;
                    g = 2.0f * d * a.inv_count;
                    loss += d * d * a.inv_count;
                }
            }
            s.g3[b][c] = g;
        }
        if (a.cls) {
            __syncthreads();
            if (t < kMlpTile && b0 + t < a.B) {
                int best = 0;
                for (int c = 1; c < K; ++c)
                    if (s.o3[t][c] < s.o3[t][best]) best = c;
                a.cls[b0 + t] = best;
            }
        }
        if (!a.target) continue;
        float *part = a.parts + (int64_t)blockIdx.x * (a.count + 1);
        float *dW1 = part, *db1 = dW1 + H * F, *dW2 = db1 + H, *db2 = dW2 + H * H, *dW3 = db2 + H,
              *db3 = dW3 + K * H;
        #pragma unroll
        for (int d = 16; d >= 1; d >>= 1) loss += __shfl_xor_sync(FULL, loss, d);
        if ((t & 31) == 0) s_loss[t >> 5] = loss;
        __syncthreads();
        if (t == 0) {
            float l = 0.0f;
            for (int w = 0; w < kMlpThreads / 32; ++w) l += s_loss[w];
            add(part + a.count, l);
        }
        // back through the output layer
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = 0.0f;
        for (int c = 0; c < K; ++c) {
            const float w = s.W3[c][o];
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[q] = fmaf(w, s.g3[sb + 4 * q][c], acc[q]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            s.g2[sb + 4 * q][o] = s.a2[sb + 4 * q][o] > 0.0f ? acc[q] : 0.0f;
        for (int k = t; k < K * H; k += kMlpThreads) {
            const int c = k / H, i = k % H;
            float v = 0.0f;
#pragma unroll
            for (int b = 0; b < kMlpTile; ++b) v = fmaf(s.g3[b][c], s.a2[b][i], v);
            add(dW3 + k, v);
        }
        if (t < K) {
            float v = 0.0f;
            for (int b = 0; b < kMlpTile; ++b) v += s.g3[b][t];
            add(db3 + t, v);
        }
        __syncthreads();
        // and through the second hidden layer
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = 0.0f;
        mlp_dot4(acc, s.W2, o, s.g2[sb], kMlpLd, H);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            s.g1[sb + 4 * q][o] = s.a1[sb + 4 * q][o] > 0.0f ? acc[q] : 0.0f;
        {
            // dW2: a thread takes 4 x 4 weights
            const int o4 = (t / 16) * 4, i4 = (t % 16) * 4;
            float w[4][4] = {};
#pragma unroll
            for (int b = 0; b < kMlpTile; ++b) {
                const float4 g = *reinterpret_cast<const float4 *>(&s.g2[b][o4]);
                const float4 v = *reinterpret_cast<const float4 *>(&s.a1[b][i4]);
                const float gg[4] = {g.x, g.y, g.z, g.w}, vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int p = 0; p < 4; ++p)
#pragma unroll
                    for (int q = 0; q < 4; ++q) w[p][q] = fmaf(gg[p], vv[q], w[p][q]);
            }
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) add(dW2 + (o4 + p) * H + i4 + q, w[p][q]);
        }
        if (t < H) {
            float v = 0.0f;
            for (int b = 0; b < kMlpTile; ++b) v += s.g2[b][t];
            add(db2 + t, v);
        }
        __syncthreads();
        for (int k = t; k < H * F; k += kMlpThreads) {
            const int u = k / F, i = k % F;
            float v = 0.0f;
#pragma unroll
            for (int b = 0; b < kMlpTile; ++b) v = fmaf(s.g1[b][u], s.X[b][i], v);
            add(dW1 + k, v);
        }
        if (t < H) {
            float v = 0.0f;
            for (int b = 0; b < kMlpTile; ++b) v += s.g1[b][t];
            add(db1 + t, v);
        }
    }
}

// grad[k] = the blocks' shares of weight k, added in order; the last one the loss
__global__ void __launch_bounds__(kMlpThreads)
    mlp_reduce_kernel(const float *__restrict__ parts, int32_t blocks, int32_t count,
                      float *__restrict__ grad, float *__restrict__ loss)
{
    // 32 weights per warp row, eight rows of the block each an eighth of the
    // blocks; their sums are joined in order
    __shared__ float s_sum[kMlpThreads / 32][32];
    grid_dep_wait();
    grid_dep_trigger();
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
    constexpr int ROWS = kMlpThreads / 32;
    const int32_t k = blockIdx.x * 32 + lane;
    const int32_t per = (blocks + ROWS - 1) / ROWS;
    const int32_t lo = row * per, hi = lo + per < blocks ? lo + per : blocks;
    float v = 0.0f;
    if (k <= count) {
#pragma unroll 8
        for (int32_t b = lo; b < hi; ++b) v += __ldcg(parts + (int64_t)b * (count + 1) + k);
    }
    s_sum[row][lane] = v;
    __syncthreads();
    if (row != 0 || k > count) return;
    v = 0.0f;
    for (int r = 0; r < ROWS; ++r) v += s_sum[r][lane];
    if (k < count) grad[k] = v;
    else if (loss) *loss = v;
}

// whether the one-kernel path takes these sizes
static bool mlp_fused(int32_t F, int32_t H1, int32_t H2, int32_t K)
{
    return H1 == kMlpH && H2 == kMlpH && F <= kMlpMaxF && F % 4 == 0 && K <= kMlpMaxK;
}

static int64_t mlp_tiles(int32_t B) { return ((int64_t)B + kMlpTile - 1) / kMlpTile; }

static cudaError_t launch_mlp(const MlpArgs &a, int64_t blocks, cudaStream_t s)
{
    static int done[64] = {0};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64 || !done[dev]) {
        const cudaError_t e = cudaFuncSetAttribute(
            mlp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MlpSmem));
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) done[dev] = 1;
    }
    return launch_dependent(mlp_kernel, (unsigned)blocks, kMlpThreads, sizeof(MlpSmem), s, a);
}

static unsigned blocks_for(int64_t n) { return (unsigned)((n + kMlpThreads - 1) / kMlpThreads); }

}  // namespace ssspmv

using namespace ssspmv;

// parameter block layout: W1[H1][F] b1[H1] W2[H2][H1] b2[H2] W3[K][H2] b3[K]
static int64_t mlp_param_count(int F, int H1, int H2, int K)
{
    return (int64_t)H1 * F + H1 + (int64_t)H2 * H1 + H2 + (int64_t)K * H2 + K;
}

extern "C" {

size_t ssspmv_features_scratch_bytes(void) { return features_scratch_bytes(); }

int ssspmv_features(int32_t m, int32_t n, int32_t nnz, const int32_t *row_ptr, float *features,
                    void *scratch, void *stream)
{
    if (m < 0 || n < 0 || nnz < 0 || (m > 0 && !row_ptr) || !features || !scratch)
        return SSSPMV_EINVAL;
    return run_features(row_ptr, m, n, nnz, features, scratch, static_cast<cudaStream_t>(stream));
}

int64_t ssspmv_mlp_param_count(int32_t F, int32_t H1, int32_t H2, int32_t K)
{
    if (F <= 0 || H1 <= 0 || H2 <= 0 || K <= 0) return 0;
    return mlp_param_count(F, H1, H2, K);
}

size_t ssspmv_mlp_scratch_floats(int32_t B, int32_t F, int32_t H1, int32_t H2, int32_t K)
{
    // pre1, act1, pre2, act2 (B x H), out (B x K), gout (B x K), g2 (B x H2), g1 (B x H1), loss
    return (size_t)B * (2 * H1 + 2 * H2 + 2 * K + H2 + H1) + 1;
}

static MlpArgs mlp_args(const float *params, const float *X, int32_t B, int32_t F, int32_t K)
{
    MlpArgs a = {};
    a.params = params;
    a.X = X;
    a.B = B;
    a.F = F;
    a.K = K;
    a.count = (int32_t)mlp_param_count(F, kMlpH, kMlpH, K);
    return a;
}

static int mlp_forward_impl(const float *params, const float *X, int32_t B, int32_t F, int32_t H1,
                            int32_t H2, int32_t K, float *scratch, cudaStream_t s)
{
    const float *W1 = params, *b1 = W1 + (int64_t)H1 * F;
    const float *W2 = b1 + H1, *b2 = W2 + (int64_t)H2 * H1;
    const float *W3 = b2 + H2, *b3 = W3 + (int64_t)K * H2;
    float *pre1 = scratch, *act1 = pre1 + (int64_t)B * H1;
    float *pre2 = act1 + (int64_t)B * H1, *act2 = pre2 + (int64_t)B * H2;
    float *out = act2 + (int64_t)B * H2;
    dense_forward_kernel<<<blocks_for((int64_t)B * H1), kMlpThreads, 0, s>>>(X, W1, b1, pre1, act1,
                                                                            B, F, H1, 1);
    dense_forward_kernel<<<blocks_for((int64_t)B * H2), kMlpThreads, 0, s>>>(act1, W2, b2, pre2,
                                                                            act2, B, H1, H2, 1);
    dense_forward_kernel<<<blocks_for((int64_t)B * K), kMlpThreads, 0, s>>>(act2, W3, b3, nullptr,
                                                                           out, B, H2, K, 0);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? SSSPMV_OK : record_cuda_error(e);
}

int ssspmv_mlp_forward(const float *params, const float *X, int32_t B, int32_t F, int32_t H1,
                       int32_t H2, int32_t K, float *scratch, float *out, void *stream)
{
    if (!params || !X || !scratch || B <= 0 || F <= 0 || H1 <= 0 || H2 <= 0 || K <= 0)
        return SSSPMV_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (mlp_fused(F, H1, H2, K)) {
        MlpArgs a = mlp_args(params, X, B, F, K);
        a.out = scratch + (int64_t)B * (2 * H1 + 2 * H2);
        a.out2 = out;
        const cudaError_t e = launch_mlp(a, mlp_tiles(B), s);
        return e == cudaSuccess ? SSSPMV_OK : record_cuda_error(e);
    }
    int rc = mlp_forward_impl(params, X, B, F, H1, H2, K, scratch, s);
    if (rc) return rc;
    if (out) {
        const float *o = scratch + (int64_t)B * (2 * H1 + 2 * H2);
        cudaError_t e = cudaMemcpyAsync(out, o, sizeof(float) * (size_t)B * K,
                                        cudaMemcpyDeviceToDevice, s);
        if (e != cudaSuccess) return record_cuda_error(e);
    }
    return SSSPMV_OK;
}

int ssspmv_mlp_backward(const float *params, const float *X, const float *target, int32_t B,
                        int32_t F, int32_t H1, int32_t H2, int32_t K, float *scratch, float *grad,
                        float *loss, void *stream)
{
    if (!params || !X || !target || !scratch || !grad || B <= 0 || F <= 0 || H1 <= 0 ||
        H2 <= 0 || K <= 0)
        return SSSPMV_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // a block per tile of samples, or as many as the scratch holds the shares of
    int64_t blocks = mlp_tiles(B);
    const int64_t room = (int64_t)(ssspmv_mlp_scratch_floats(B, F, H1, H2, K) /
                                   (size_t)(mlp_param_count(F, H1, H2, K) + 1));
    if (blocks > room) blocks = room;
    if (mlp_fused(F, H1, H2, K) && blocks > 0) {
        MlpArgs a = mlp_args(params, X, B, F, K);
        a.target = target;
        a.parts = scratch;
        a.inv_count = 1.0f / (float)((int64_t)B * K);
        cudaError_t e = launch_mlp(a, blocks, s);
        if (e == cudaSuccess)
            e = launch_dependent(mlp_reduce_kernel, (unsigned)((a.count + 1 + 31) / 32),
                                 kMlpThreads, 0, s, (const float *)scratch, (int32_t)blocks,
                                 a.count, grad, loss);
        return e == cudaSuccess ? SSSPMV_OK : record_cuda_error(e);
    }
    int rc = mlp_forward_impl(params, X, B, F, H1, H2, K, scratch, s);
    if (rc) return rc;
    const float *W2 = params + (int64_t)H1 * F + H1;
    const float *W3 = W2 + (int64_t)H2 * H1 + H2;
    float *pre1 = scratch, *act1 = pre1 + (int64_t)B * H1;
    float *pre2 = act1 + (int64_t)B * H1, *act2 = pre2 + (int64_t)B * H2;
    float *out = act2 + (int64_t)B * H2, *gout = out + (int64_t)B * K;
    float *g2 = gout + (int64_t)B * K, *g1 = g2 + (int64_t)B * H2;
    float *lacc = g1 + (int64_t)B * H1;
    float *dW1 = grad, *db1 = dW1 + (int64_t)H1 * F;
    float *dW2 = db1 + H1, *db2 = dW2 + (int64_t)H2 * H1;
    float *dW3 = db2 + H2, *db3 = dW3 + (int64_t)K * H2;
    cudaError_t e = cudaMemsetAsync(lacc, 0, sizeof(float), s);
    if (e != cudaSuccess) return record_cuda_error(e);
    // squared error averaged over all B*K outputs; a NaN target (a class not
    // measured) contributes neither loss nor gradient
    const int64_t n = (int64_t)B * K;
    loss_grad_kernel<<<blocks_for(n), kMlpThreads, 0, s>>>(out, target, gout, n, 1.0f / (float)n,
                                                          lacc);
    dense_grad_w_kernel<<<blocks_for((int64_t)K * H2 + K), kMlpThreads, 0, s>>>(act2, gout, dW3,
                                                                              db3, B, H2, K);
    dense_grad_in_kernel<<<blocks_for((int64_t)B * H2), kMlpThreads, 0, s>>>(W3, gout, pre2, g2, B,
                                                                            H2, K);
    dense_grad_w_kernel<<<blocks_for((int64_t)H2 * H1 + H2), kMlpThreads, 0, s>>>(act1, g2, dW2,
                                                                                db2, B, H1, H2);
    dense_grad_in_kernel<<<blocks_for((int64_t)B * H1), kMlpThreads, 0, s>>>(W2, g2, pre1, g1, B,
                                                                            H1, H2);
    dense_grad_w_kernel<<<blocks_for((int64_t)H1 * F + H1), kMlpThreads, 0, s>>>(X, g1, dW1, db1,
                                                                               B, F, H1);
    if (loss) {
        e = cudaMemcpyAsync(loss, lacc, sizeof(float), cudaMemcpyDeviceToDevice, s);
        if (e != cudaSuccess) return record_cuda_error(e);
    }
    e = cudaGetLastError();
    return e == cudaSuccess ? SSSPMV_OK : record_cuda_error(e);
}

int ssspmv_mlp_adam(float *params, const float *grad, float *m1, float *m2, int64_t n, float lr,
                    float beta1, float beta2, float eps, float weight_decay, int32_t step,
                    void *stream)
{
    if (!params || !grad || !m1 || !m2 || n <= 0 || step < 1) return SSSPMV_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    cudaError_t e = launch_dependent(adam_kernel, blocks_for(n), kMlpThreads, 0, s, params, grad,
                                     m1, m2, n, lr, beta1, beta2, eps, weight_decay, step);
    return e == cudaSuccess ? SSSPMV_OK : record_cuda_error(e);
}

int ssspmv_mlp_select(const float *params, const float *X, int32_t B, int32_t F, int32_t H1,
                      int32_t H2, int32_t K, float *scratch, int32_t *cls, void *stream)
{
    if (!cls) return SSSPMV_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (params && X && scratch && B > 0 && F > 0 && K > 0 && mlp_fused(F, H1, H2, K)) {
        MlpArgs a = mlp_args(params, X, B, F, K);
        a.out = scratch + (int64_t)B * (2 * H1 + 2 * H2);
        a.cls = cls;
        const cudaError_t e = launch_mlp(a, mlp_tiles(B), s);
        return e == cudaSuccess ? SSSPMV_OK : record_cuda_error(e);
    }
    int rc = ssspmv_mlp_forward(params, X, B, F, H1, H2, K, scratch, nullptr, stream);
    if (rc) return rc;
    const float *out = scratch + (int64_t)B * (2 * H1 + 2 * H2);
    argmin_kernel<<<(unsigned)((B + 127) / 128), 128, 0, s>>>(out, B, K, cls);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? SSSPMV_OK : record_cuda_error(e);
}

}  // extern "C"
