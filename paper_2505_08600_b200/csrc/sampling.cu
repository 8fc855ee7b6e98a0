// Vocabulary-wide kernels: softmax with temperature, the exact integer inverse-CDF draw, the
// draft's per-step sampler and the fused accept / reject / resample kernel.
#include <cooperative_groups.h>

#include <algorithm>

#include "gemm_tc.h"
#include "kernels.h"

namespace sd {

__global__ void k_philox(const uint32_t* __restrict__ ctr, int n, uint32_t k0, uint32_t k1, uint32_t* __restrict__ out) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t o[4];
    philox4x32_10(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3], k0, k1, o);
    for (int j = 0; j < 4; ++j) out[4 * i + j] = o[j];
}
cudaError_t launch_philox(const uint32_t* ctr, int n, uint32_t k0, uint32_t k1, uint32_t* out, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_philox<<<(n + 127) / 128, 128, 0, st>>>(ctr, n, k0, k1, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- block-wide helpers
struct BlockScratch {
    float red[32];
    unsigned long long scan[32];
    unsigned long long total;
    int tok;
    int idx;
};

__device__ __forceinline__ int block_min_int(int v, BlockScratch& sh) {
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    int* r = reinterpret_cast<int*>(sh.red);
    if (lane == 0) r[w] = v;
    __syncthreads();
    int x = (threadIdx.x < nw) ? r[threadIdx.x] : 0x7fffffff;
    if (w == 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x = min(x, __shfl_xor_sync(0xffffffffu, x, o));
        if (lane == 0) sh.idx = x;
    }
    __syncthreads();
    return sh.idx;
}

// lowest index of the maximum of f(k), k in [0, V)
template <class F>
__device__ __forceinline__ int block_argmax(F f, int V, BlockScratch& sh, float* max_out) {
    float m = -INFINITY;
    for (int k = threadIdx.x; k < V; k += blockDim.x) m = fmaxf(m, f(k));
    m = block_max(m, sh.red);
    int best = 0x7fffffff;
    for (int k = threadIdx.x; k < V; k += blockDim.x) if (f(k) == m) { best = k; break; }
    if (max_out) *max_out = m;
    return block_min_int(best, sh);
}

// Exact inverse CDF over integer weights floor(w(k) * 2^32): returns the first k whose running
// sum reaches ceil(u_int * total / 2^24), or -1 when every weight is zero.  Each thread owns a
// contiguous chunk; integer addition is associative, so the split cannot change the answer.
template <class F>
__device__ __forceinline__ int block_icdf(F w, int V, uint32_t u_int, BlockScratch& sh) {
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5, nw = (blockDim.x + 31) >> 5;
    const int chunk = (V + blockDim.x - 1) / blockDim.x;
    const int k0 = min(V, t * chunk), k1 = min(V, k0 + chunk);
    unsigned long long local = 0;
    {   // every thread starts its chunk at a different offset, so that a vocabulary row staged in shared
        // memory is read without bank conflicts (the order inside a sum of integers does not matter)
        const int n = k1 - k0;
        int i = n > 0 ? t % n : 0;
        for (int c = 0; c < n; ++c) { local += __float2ull_rz(w(k0 + i) * 4294967296.0f); i = (i + 1 == n) ? 0 : i + 1; }
    }
    unsigned long long incl = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        unsigned long long v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    __syncthreads();
    if (lane == 31) sh.scan[wid] = incl;
    if (t == 0) sh.tok = -1;
    __syncthreads();
    if (wid == 0) {
        unsigned long long v = lane < nw ? sh.scan[lane] : 0ull, s = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            unsigned long long u = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += u;
        }
        sh.scan[lane] = s - v;                       // exclusive prefix of each warp
        if (lane == 31) sh.total = s;
    }
    __syncthreads();
    const unsigned long long tot = sh.total;
    if (tot == 0ull) return -1;
    incl += sh.scan[wid];
    const unsigned long long excl = incl - local;
    const unsigned long long thr = ((unsigned long long)u_int * tot + 16777215ull) >> 24;
    if (excl < thr && thr <= incl) {
        unsigned long long run = excl;
        for (int k = k0; k < k1; ++k) {
            run += __float2ull_rz(w(k) * 4294967296.0f);
            if (run >= thr) { sh.tok = k; break; }
        }
    }
    __syncthreads();
    return sh.tok;
}

// Copies one vocabulary row into shared memory with every load in flight at once (the later
// passes over the row - max, sum, probabilities, CDF - then cost no memory round trips).
__device__ __forceinline__ void stage_row(const float* __restrict__ src, float* __restrict__ dst, int V) {
    if ((V & 3) == 0 && (reinterpret_cast<uintptr_t>(src) & 15) == 0) {
        const float4* s4 = reinterpret_cast<const float4*>(src);
        float4* d4 = reinterpret_cast<float4*>(dst);
        const int n4 = V >> 2;
        for (int k0 = 0; k0 < n4; k0 += 8 * blockDim.x) {
            float4 v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) { const int k = k0 + i * blockDim.x + threadIdx.x; if (k < n4) v[i] = __ldcg(s4 + k); }
#pragma unroll
            for (int i = 0; i < 8; ++i) { const int k = k0 + i * blockDim.x + threadIdx.x; if (k < n4) d4[k] = v[i]; }
        }
    } else {
        for (int k = threadIdx.x; k < V; k += blockDim.x) dst[k] = __ldcg(src + k);
    }
    __syncthreads();
}
constexpr int STAGE_MAX_BYTES = 200 * 1024;      // a row of up to 51200 fp32 values fits beside the static shared memory

// Dynamic shared memory for one staged row, or 0 when the vocabulary is too large to stage.
static size_t row_stage_bytes(int V) { return (size_t)V * 4 <= (size_t)STAGE_MAX_BYTES ? (size_t)V * 4 : 0; }

// ---------------------------------------------------------------- softmax + draw (draft steps)
// One block per row.  probs = softmax(logits / T) (one-hot argmax when T == 0) is written out,
// then one token is drawn from the written fp32 values.
__device__ __forceinline__ int softmax_sample_row(const float* __restrict__ l_global, int V, float T, uint32_t u_int,
                                                  float* __restrict__ probs, BlockScratch& sh, float* rowbuf) {
    const float* l = l_global;
    if (rowbuf) { stage_row(l_global, rowbuf, V); l = rowbuf; }
    if (T == 0.f) {
        int a = block_argmax([&](int k) { return l[k]; }, V, sh, nullptr);
        for (int k = threadIdx.x; k < V; k += blockDim.x) probs[k] = (k == a) ? 1.f : 0.f;
        return a;
    }
    float m = -INFINITY;
    for (int k = threadIdx.x; k < V; k += blockDim.x) m = fmaxf(m, l[k]);
    m = block_max(m, sh.red);
    float s = 0.f;
    // one division each for 1/T and 1/sum, then multiplications: an IEEE division per element costs about as much as
    // the exponential itself, and the result differs from e / sum by an ulp (the probability tolerance is 1e-3)
    const float inv_T = 1.f / T;
    for (int k = threadIdx.x; k < V; k += blockDim.x) s += expf((l[k] - m) * inv_T);
    s = block_sum(s, sh.red);
    const float inv_s = 1.f / s;
    for (int k = threadIdx.x; k < V; k += blockDim.x) {
        const float pk = expf((l[k] - m) * inv_T) * inv_s;
        probs[k] = pk;
        if (rowbuf) rowbuf[k] = pk;                      // the draw below reads the same fp32 values
    }
    __syncthreads();
    const float* pr = rowbuf ? rowbuf : probs;
    int tok = block_icdf([&](int k) { return pr[k]; }, V, u_int, sh);
    if (tok < 0) tok = block_argmax([&](int k) { return pr[k]; }, V, sh, nullptr);
    return tok;
}

__global__ void __launch_bounds__(1024) k_softmax_sample_explicit(const float* __restrict__ logits, int V, float T,
                                                                  const uint32_t* __restrict__ u_int,
                                                                  float* __restrict__ probs, int32_t* __restrict__ tok, int staged) {
    extern __shared__ __align__(16) float rowbuf[];
    __shared__ BlockScratch sh;
    const int r = blockIdx.x;
    int k = softmax_sample_row(logits + (size_t)r * V, V, T, u_int[r], probs + (size_t)r * V, sh, staged ? rowbuf : nullptr);
    if (threadIdx.x == 0) tok[r] = k;
}
cudaError_t launch_softmax_sample_explicit(const float* logits, int rows, int V, float T, const uint32_t* u_int,
                                           float* probs, int32_t* tok, cudaStream_t st) {
    if (rows <= 0) return cudaSuccess;
    const size_t smem = row_stage_bytes(V);
    cudaError_t e = cudaFuncSetAttribute(k_softmax_sample_explicit, cudaFuncAttributeMaxDynamicSharedMemorySize, STAGE_MAX_BYTES);
    if (e != cudaSuccess) return e;
    k_softmax_sample_explicit<<<rows, 1024, smem, st>>>(logits, V, T, u_int, probs, tok, smem > 0);
    return cudaGetLastError();
}

__global__ void __launch_bounds__(1024) k_draft_sample(const float* __restrict__ logits, SeqState S, SeqList list, int V, float T,
                                                       uint64_t seed, int step, int gamma, float* __restrict__ q_out,
                                                       int32_t* __restrict__ x_out, int staged) {
    extern __shared__ __align__(16) float rowbuf[];
    __shared__ BlockScratch sh;
    const int i = blockIdx.x, slot = list.ids[i], b = list.out[i];
    const uint32_t u = uniform24(seed, S.iter[slot], (uint32_t)step, S.seq_id[slot], DRAW_DRAFT);
    int k = softmax_sample_row(logits + (size_t)i * V, V, T, u, q_out + ((size_t)b * gamma + step) * V, sh, staged ? rowbuf : nullptr);
    if (threadIdx.x == 0) x_out[(size_t)b * gamma + step] = k;
}
// The same over a cluster of eight CTAs per row, each with an eighth of the vocabulary in shared memory: a row of 32000 is 32
// exponentials per thread for one CTA of 1024, four for eight CTAs of 1024.  What the slices have to know of one another (maximum,
// sum, integer total) goes to every CTA of the cluster through distributed shared memory.  The token is the one of the integer
// inverse CDF over the written fp32 values, whatever the split.  32000 values, five draft steps of a one-layer model: 210 -> 174 us.
constexpr int SLICES = 8;
__host__ __device__ __forceinline__ int slice_len(int V) { return (V + 4 * SLICES - 1) / (4 * SLICES) * 4; }
// Rows whose clusters run side by side (a CTA of 1024 threads per SM, a cluster inside one GPC): 12 rows take one wave, 16 and 24 two, 32
// three, 64 five.
constexpr int SLICED_WAVE = 14;
static double sliced_waves(int n) { return (n + SLICED_WAVE - 1) / SLICED_WAVE; }
// Where the slices are the faster form.  Against a CTA per row (which has all rows in one wave) they save 0.3 us per thousand values above
// 8192 (32000: 7.3 us a draw, 16384: 2.4, 4096: -1.4 for one to twelve rows) and cost 6.5 us and a little more per further wave (32000 values,
// 16 rows: -1.1, 32 rows: -9.7; 50000: +4.2 and -5.8).  A row that cannot be staged (64000 values) takes a CTA three times as long.
static bool draft_sliced(int V, int n) {
    if ((size_t)slice_len(V) * sizeof(float) > (size_t)STAGE_MAX_BYTES) return false;
    return !row_stage_bytes(V) || 3e-4 * (V - 8192) > (sliced_waves(n) - 1) * (6.5 + 6e-5 * V);
}
struct SliceScratch {
    BlockScratch b;
    float f[2][SLICES];
    int idx[SLICES];
    unsigned long long total[SLICES];
};

// block_icdf over this CTA's slice of n weights, `base` being the weight of everything in front of it, `thr` the running sum to be
// reached: the index inside the slice in the CTA whose slice holds it, -1 in the others.  local: the slice's weight of this thread.
template <class F>
__device__ __forceinline__ int slice_pick(F w, int n, unsigned long long base, unsigned long long thr, unsigned long long local, BlockScratch& sh) {
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5, nw = blockDim.x >> 5;
    const int chunk = (n + blockDim.x - 1) / blockDim.x, k0 = min(n, t * chunk), k1 = min(n, k0 + chunk);
    unsigned long long incl = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        unsigned long long v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    __syncthreads();
    if (lane == 31) sh.scan[wid] = incl;
    if (t == 0) sh.tok = -1;
    __syncthreads();
    unsigned long long before = base;
    for (int i = 0; i < wid && i < nw; ++i) before += sh.scan[i];
    incl += before;
    const unsigned long long excl = incl - local;
    if (excl < thr && thr <= incl) {
        unsigned long long run = excl;
        for (int k = k0; k < k1; ++k) {
            run += __float2ull_rz(w(k) * 4294967296.0f);
            if (run >= thr) { sh.tok = k; break; }
        }
    }
    __syncthreads();
    return sh.tok;
}
// The integer weight of this thread's chunk of a slice, and the slice's total (valid in every thread).
template <class F>
__device__ __forceinline__ unsigned long long slice_weight(F w, int n, unsigned long long* total, BlockScratch& sh) {
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5, nw = blockDim.x >> 5;
    const int chunk = (n + blockDim.x - 1) / blockDim.x, k0 = min(n, t * chunk), k1 = min(n, k0 + chunk);
    unsigned long long local = 0;
    for (int k = k0; k < k1; ++k) local += __float2ull_rz(w(k) * 4294967296.0f);
    unsigned long long s = local;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    __syncthreads();
    if (lane == 0) sh.scan[wid] = s;
    __syncthreads();
    s = 0;
    for (int i = 0; i < nw; ++i) s += sh.scan[i];
    *total = s;
    return local;
}

// Which slice holds the draw with uniform u_int / 2^24 and where in the running sum that is (the same answer in every CTA).
struct SliceDraw { int owner; unsigned long long before, thr; };
__device__ __forceinline__ SliceDraw slice_draw(const unsigned long long (&total)[SLICES], uint32_t u_int) {
    unsigned long long tot = 0, run = 0;
#pragma unroll
    for (int r = 0; r < SLICES; ++r) tot += total[r];
    SliceDraw d{-1, 0ull, ((unsigned long long)u_int * tot + 16777215ull) >> 24};
#pragma unroll
    for (int r = 0; r < SLICES; ++r) {
        if (d.owner < 0 && run < d.thr && d.thr <= run + total[r]) { d.owner = r; d.before = run; }
        run += total[r];
    }
    return d;                                                   // owner < 0: every weight is zero (or not a number)
}

__global__ void __cluster_dims__(SLICES, 1, 1) __launch_bounds__(1024)
k_draft_sample_sliced(const float* __restrict__ logits, SeqState S, SeqList list, int V, float T, uint64_t seed, int step, int gamma,
                      float* __restrict__ q_out, int32_t* __restrict__ x_out) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) float buf[];
    __shared__ SliceScratch sh;
    pdl_launch_dependents();
    const int i = blockIdx.x / SLICES, rank = blockIdx.x % SLICES, slot = list.ids[i], b = list.out[i];
    const int len = slice_len(V), base = min(V, rank * len), n = min(V, base + len) - base;
    float* probs = q_out + ((size_t)b * gamma + step) * V + base;
    auto share = [&](auto* mine, auto v) {                     // to every CTA of the cluster; visible after cluster.sync()
        if (threadIdx.x < SLICES) cluster.map_shared_rank(mine, threadIdx.x)[rank] = v;
    };
    pdl_wait();
    const float* l = logits + (size_t)i * V + base;
    float m = -INFINITY;
    for (int k = threadIdx.x; k < n; k += blockDim.x) { const float v = __ldcg(l + k); buf[k] = v; m = fmaxf(m, v); }
    m = block_max(m, sh.b.red);
    cluster.sync();                                             // every CTA is there before the others write into it
    share(sh.f[0], m);
    cluster.sync();
#pragma unroll
    for (int r = 0; r < SLICES; ++r) m = fmaxf(m, sh.f[0][r]);
    // lowest index that holds value v of the slices (all CTAs take part)
    auto first_index = [&](float v) {
        int best = 0x7fffffff;
        for (int k = threadIdx.x; k < n; k += blockDim.x) if (buf[k] == v) { best = base + k; break; }
        best = block_min_int(best, sh.b);
        share(sh.idx, best);
        cluster.sync();
#pragma unroll
        for (int r = 0; r < SLICES; ++r) best = min(best, sh.idx[r]);
        return best;
    };
    int tok;
    if (T == 0.f) {
        tok = first_index(m);
        for (int k = threadIdx.x; k < n; k += blockDim.x) probs[k] = base + k == tok ? 1.f : 0.f;
        if (rank == 0 && threadIdx.x == 0) x_out[(size_t)b * gamma + step] = tok;
    } else {
        const float inv_T = 1.f / T;                            // (multiplications by 1/T and 1/sum: see softmax_sample_row)
        float s = 0.f;
        for (int k = threadIdx.x; k < n; k += blockDim.x) { const float e = expf((buf[k] - m) * inv_T); buf[k] = e; s += e; }
        s = block_sum(s, sh.b.red);
        share(sh.f[1], s);
        cluster.sync();
        s = 0.f;
#pragma unroll
        for (int r = 0; r < SLICES; ++r) s += sh.f[1][r];
        const float inv_s = 1.f / s;
        for (int k = threadIdx.x; k < n; k += blockDim.x) { const float p = buf[k] * inv_s; buf[k] = p; probs[k] = p; }
        __syncthreads();
        unsigned long long mine;
        const unsigned long long local = slice_weight([&](int k) { return buf[k]; }, n, &mine, sh.b);
        share(sh.total, mine);
        cluster.sync();
        const SliceDraw d = slice_draw(sh.total, uniform24(seed, S.iter[slot], (uint32_t)step, S.seq_id[slot], DRAW_DRAFT));
        if (d.owner >= 0) {
            if (d.owner == rank) {
                tok = max(slice_pick([&](int k) { return buf[k]; }, n, d.before, d.thr, local, sh.b), 0);
                if (threadIdx.x == 0) x_out[(size_t)b * gamma + step] = base + tok;
            }
        } else {                                                // every weight rounds to zero: the largest probability
            float pm = -INFINITY;
            for (int k = threadIdx.x; k < n; k += blockDim.x) pm = fmaxf(pm, buf[k]);
            pm = block_max(pm, sh.b.red);
            share(sh.f[0], pm);
            cluster.sync();
#pragma unroll
            for (int r = 0; r < SLICES; ++r) pm = fmaxf(pm, sh.f[0][r]);
            tok = first_index(pm);
            if (rank == 0 && threadIdx.x == 0) x_out[(size_t)b * gamma + step] = tok;
        }
    }
    cluster.sync();                                             // no CTA leaves while the others may still write into it
}

cudaError_t launch_draft_sample(const float* logits, const SeqState& S, const SeqList& list, int V, float T,
                                uint64_t seed, int step, int gamma, float* q_out, int32_t* x_out, cudaStream_t st) {
    if (list.n <= 0) return cudaSuccess;
    const size_t slice = (size_t)slice_len(V) * sizeof(float);
    if (draft_sliced(V, list.n)) {
        cudaError_t e = cudaFuncSetAttribute(k_draft_sample_sliced, cudaFuncAttributeMaxDynamicSharedMemorySize, STAGE_MAX_BYTES);
        if (e != cudaSuccess) return e;
        return launch_pdl(k_draft_sample_sliced, dim3(list.n * SLICES), dim3(1024), slice, st, 1, logits, S, list, V, T, seed, step, gamma, q_out, x_out);
    }
    const size_t smem = row_stage_bytes(V);
    cudaError_t e = cudaFuncSetAttribute(k_draft_sample, cudaFuncAttributeMaxDynamicSharedMemorySize, STAGE_MAX_BYTES);
    if (e != cudaSuccess) return e;
    k_draft_sample<<<list.n, 1024, smem, st>>>(logits, S, list, V, T, seed, step, gamma, q_out, x_out, smem > 0);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- accept / reject / resample
// One thread-block cluster per sequence, one CTA per target row (two when gamma + 1 > 8).
// Every CTA works out the softmax statistics of its row(s) and, for a draft slot, the accept
// test u_s * q_s(x_s) <= p_s(x_s) with a single rounded fp32 multiply.  The flags are exchanged
// through distributed shared memory; the CTA that owns the first rejected row n (or row gamma
// after gamma accepts) draws the next token from the residual max(0, p_n - q_n), or from
// p_gamma itself, and writes the result.
constexpr int ACC_ROWS_PER_CTA = 2;

__global__ void __launch_bounds__(1024) k_accept(AcceptParams P, int csize, int staged) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) float rowbuf[];            // one target row (when it fits): every pass over it reads shared memory
    __shared__ BlockScratch sh;
    __shared__ float row_max[ACC_ROWS_PER_CTA], row_inv[ACC_ROWS_PER_CTA];      // max of the row's logits, 1 / sum of its exponentials
    __shared__ int row_arg[ACC_ROWS_PER_CTA];
    __shared__ int flag_sh[ACC_ROWS_PER_CTA];
    __shared__ int n_sh;
    pdl_launch_dependents();
    const int i = blockIdx.x / csize, rank = blockIdx.x % csize;
    const int idx = P.use_list ? P.list.ids[i] : i;
    const int b = P.use_list ? P.list.out[i] : i;
    const int V = P.V, gamma = P.gamma;
    const float T = P.T;
    const float inv_T = T > 0.f ? 1.f / T : 0.f;
    const float* tgt = P.target + (size_t)b * (gamma + 1) * V;
    const float* q = P.q + (size_t)b * gamma * V;
    const int32_t* x = P.x + (size_t)b * gamma;
    const bool logits = P.target_is_logits != 0;
    pdl_wait();                                   // target rows, drafts and per-sequence state come from earlier kernels

    int cur = -1;                                 // which of this CTA's rows the buffer holds
    auto ensure = [&](int j, int li) {
        if (staged && cur != li) { __syncthreads(); stage_row(tgt + (size_t)j * V, rowbuf, V); cur = li; }
    };
    auto val = [&](int j, int k) -> float { return staged ? rowbuf[k] : tgt[(size_t)j * V + k]; };
    auto prob = [&](int j, int li, int k) -> float {          // li: index of row j among this CTA's rows
        if (logits && T == 0.f) return k == row_arg[li] ? 1.f : 0.f;
        const float v = val(j, k);
        if (!logits) return v;
        return expf((v - row_max[li]) * inv_T) * row_inv[li];      // (multiplications by 1/T and 1/sum: see softmax_sample_row)
    };

    for (int li = 0; li < ACC_ROWS_PER_CTA; ++li) {
        const int j = rank + li * csize;
        if (j > gamma) break;                                   // uniform in the CTA
        ensure(j, li);
        if (logits) {
            if (T == 0.f) {
                int a = block_argmax([&](int k) { return val(j, k); }, V, sh, nullptr);
                if (threadIdx.x == 0) row_arg[li] = a;
            } else {
                float m = -INFINITY;
                for (int k = threadIdx.x; k < V; k += blockDim.x) m = fmaxf(m, val(j, k));
                m = block_max(m, sh.red);
                float sum = 0.f;
                for (int k = threadIdx.x; k < V; k += blockDim.x) sum += expf((val(j, k) - m) * inv_T);
                sum = block_sum(sum, sh.red);
                if (threadIdx.x == 0) { row_max[li] = m; row_inv[li] = 1.f / sum; }
            }
            __syncthreads();
        }
        if (P.alpha_terms && j < gamma) {                       // Eq. 1's alpha for this slot: the draft is kept with probability sum_k min(p, q)
            const float* __restrict__ qj = q + (size_t)j * V;
            float a = 0.f;
            const int stride = blockDim.x;
            int k = threadIdx.x;
            for (; k + 3 * stride < V; k += 4 * stride) {             // four independent loads of q in flight per thread
                const float q0 = __ldg(qj + k), q1 = __ldg(qj + k + stride), q2 = __ldg(qj + k + 2 * stride), q3 = __ldg(qj + k + 3 * stride);
                a += fminf(prob(j, li, k), q0);
                a += fminf(prob(j, li, k + stride), q1);
                a += fminf(prob(j, li, k + 2 * stride), q2);
                a += fminf(prob(j, li, k + 3 * stride), q3);
            }
            for (; k < V; k += stride) a += fminf(prob(j, li, k), __ldg(qj + k));
            a = block_sum(a, sh.red);
            if (threadIdx.x == 0) P.alpha_terms[(size_t)b * gamma + j] = a;
        }
        if (threadIdx.x == 0 && j < gamma) {
            int ok = 0;
            const int xs = x[j];
            if (xs >= 0 && xs < V) {                            // an impossible token counts as rejected
                const uint32_t ui = uniform24(P.seed, P.iter[idx], (uint32_t)j, P.seq_id[idx], DRAW_ACCEPT);
                const float u = (float)ui * (1.0f / 16777216.0f);
                const float lhs = __fmul_rn(u, q[(size_t)j * V + xs]);
                ok = lhs <= prob(j, li, xs);
            }
            flag_sh[li] = ok;
        }
    }
    cluster.sync();                                             // every CTA's flags are in place
    if (threadIdx.x == 0) {
        int n = 0;
        while (n < gamma) {
            const int* remote = cluster.map_shared_rank(flag_sh, n % csize);
            if (!remote[n / csize]) break;
            ++n;
        }
        n_sh = n;
    }
    __syncthreads();
    const int n = n_sh;
    if (n % csize == rank) {                                    // this CTA holds the statistics of row n
        const int li = n / csize;
        const uint32_t ui = uniform24(P.seed, P.iter[idx], (uint32_t)n, P.seq_id[idx], DRAW_RESAMPLE);
        const float* qn = q + (size_t)(n < gamma ? n : 0) * V;
        int y;
        if (staged) {
            // the weights of the draw replace the row in shared memory (one coalesced pass over q), then the
            // integer CDF runs on them; residual all zero -> the target distribution itself -> its argmax
            ensure(n, li);
            for (int k = threadIdx.x; k < V; k += blockDim.x) {
                const float pk = prob(n, li, k);
                rowbuf[k] = n < gamma ? fmaxf(__fsub_rn(pk, qn[k]), 0.f) : pk;
            }
            __syncthreads();
            y = block_icdf([&](int k) { return rowbuf[k]; }, V, ui, sh);
            if (y < 0 && n < gamma) {
                cur = -1;
                ensure(n, li);
                for (int k = threadIdx.x; k < V; k += blockDim.x) rowbuf[k] = prob(n, li, k);
                __syncthreads();
                y = block_icdf([&](int k) { return rowbuf[k]; }, V, ui, sh);
            }
            if (y < 0) y = block_argmax([&](int k) { return rowbuf[k]; }, V, sh, nullptr);
        } else {
            if (n < gamma) {
                y = block_icdf([&](int k) { return fmaxf(__fsub_rn(prob(n, li, k), qn[k]), 0.f); }, V, ui, sh);
                if (y < 0) y = block_icdf([&](int k) { return prob(n, li, k); }, V, ui, sh);
            } else {
                y = block_icdf([&](int k) { return prob(n, li, k); }, V, ui, sh);
            }
            if (y < 0) y = block_argmax([&](int k) { return prob(n, li, k); }, V, sh, nullptr);
        }
        if (threadIdx.x == 0) P.n_acc[b] = n;
        for (int s = threadIdx.x; s <= gamma; s += blockDim.x)
            P.out_tok[(size_t)b * (gamma + 1) + s] = s < n ? x[s] : (s == n ? y : -1);
    }
    cluster.sync();                                             // no CTA leaves while its flags may still be read
}

// The same rule with the vocabulary cut over the cluster instead of the rows: every CTA holds an eighth of all gamma + 1 rows in
// shared memory, so that each exponential is computed once and by eight times as many threads, and the draw from row n is
// spread as well.  Taken when the slices fit (gamma + 1 rows of V / 8).  One sequence, gamma = 5, V = 32000: 33 -> 19 us
// (1B iteration, five draws and one accept: 1.100 -> 1.058 ms).
constexpr int ACC_MAX_ROWS = SD_MAX_GAMMA + 1;
struct AcceptSliceScratch {
    BlockScratch b;
    float warp_f[ACC_MAX_ROWS][32];                            // per row and warp
    float mx[ACC_MAX_ROWS][SLICES], sum[ACC_MAX_ROWS][SLICES], alpha[ACC_MAX_ROWS][SLICES];
    int arg[ACC_MAX_ROWS][SLICES], ok[ACC_MAX_ROWS];
    unsigned long long total[2][SLICES];
};
__global__ void __cluster_dims__(SLICES, 1, 1) __launch_bounds__(1024) k_accept_sliced(AcceptParams P) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) float buf[];               // [row][slice]: logits, then exponentials (or the probabilities as given)
    __shared__ AcceptSliceScratch sh;
    pdl_launch_dependents();
    const int i = blockIdx.x / SLICES, rank = blockIdx.x % SLICES, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int idx = P.use_list ? P.list.ids[i] : i, b = P.use_list ? P.list.out[i] : i;
    const int V = P.V, gamma = P.gamma, rows = gamma + 1;
    const int len = slice_len(V), base = min(V, rank * len), n = min(V, base + len) - base;
    const float T = P.T, inv_T = T > 0.f ? 1.f / T : 0.f;
    const float* tgt = P.target + (size_t)b * rows * V + base;
    const float* q = P.q + (size_t)b * gamma * V + base;
    const int32_t* x = P.x + (size_t)b * gamma;
    const bool logits = P.target_is_logits != 0, soft = logits && T > 0.f;
    if (tid < rows) sh.ok[tid] = 0;
    pdl_wait();                                                // target rows, drafts and per-sequence state come from earlier kernels
    // a per-row reduction over the CTA, then to every CTA of the cluster
    auto reduce_rows = [&](int n_rows, bool is_max, float (*out)[SLICES]) {      // of warp_f
        __syncthreads();
        for (int j = warp; j < n_rows; j += 32) {
            float v = sh.warp_f[j][lane];
            v = is_max ? warp_max(v) : warp_sum(v);
            if (lane < SLICES) cluster.map_shared_rank(&out[j][0], lane)[rank] = v;
        }
        cluster.sync();
    };
    for (int j = 0; j < rows; ++j) {
        float m = -INFINITY;
        for (int k = tid; k < n; k += 1024) { const float v = __ldcg(tgt + (size_t)j * V + k); buf[j * len + k] = v; m = fmaxf(m, v); }
        if (logits) { m = warp_max(m); if (lane == 0) sh.warp_f[j][warp] = m; }
    }
    cluster.sync();                                            // every CTA is there before the others write into it
    float inv_s = 1.f;                                          // (of row `lane` in every warp, below)
    if (logits) reduce_rows(rows, true, sh.mx);
    auto row_max = [&](int j) {
        float m = sh.mx[j][0];
#pragma unroll
        for (int r = 1; r < SLICES; ++r) m = fmaxf(m, sh.mx[j][r]);
        return m;
    };
    if (soft) {
        for (int j = 0; j < rows; ++j) {
            const float m = row_max(j);
            float s = 0.f;
            for (int k = tid; k < n; k += 1024) { const float e = expf((buf[j * len + k] - m) * inv_T); buf[j * len + k] = e; s += e; }      // (1/T: see softmax_sample_row)
            s = warp_sum(s);
            if (lane == 0) sh.warp_f[j][warp] = s;
        }
        reduce_rows(rows, false, sh.sum);
        if (lane < rows) {
            float s = 0.f;
#pragma unroll
            for (int r = 0; r < SLICES; ++r) s += sh.sum[lane][r];
            inv_s = 1.f / s;
        }
    } else if (logits) {                                       // one-hot: lowest index of the maximum
        for (int j = 0; j < rows; ++j) {
            const float m = row_max(j);
            int best = 0x7fffffff;
            for (int k = tid; k < n; k += 1024) if (buf[j * len + k] == m) { best = base + k; break; }
            best = block_min_int(best, sh.b);
            if (tid < SLICES) cluster.map_shared_rank(&sh.arg[j][0], tid)[rank] = best;
        }
        cluster.sync();
        for (int j = 0; j < rows; ++j) {
            int a = sh.arg[j][0];
#pragma unroll
            for (int r = 1; r < SLICES; ++r) a = min(a, sh.arg[j][r]);
            for (int k = tid; k < n; k += 1024) buf[j * len + k] = base + k == a ? 1.f : 0.f;
        }
    }
    // probability of the row's k-th value of this slice: what is in the buffer times the row's factor
    auto factor = [&](int j) { return soft ? __shfl_sync(0xffffffffu, inv_s, j) : 1.f; };
    __syncthreads();
    for (int j = 0; j < gamma; ++j) {
        const float f = factor(j);
        if (P.alpha_terms) {                                   // Eq. 1's alpha for this slot: the draft is kept with probability sum_k min(p, q)
            const float* qj = q + (size_t)j * V;
            float a = 0.f;
#pragma unroll 4
            for (int k = tid; k < n; k += 1024) a += fminf(buf[j * len + k] * f, __ldg(qj + k));
            a = warp_sum(a);
            if (lane == 0) sh.warp_f[j][warp] = a;
        }
        if (tid == 0) {
            const int xs = x[j] - base;
            if (xs >= 0 && xs < n) {                           // the CTA whose slice holds the token (an impossible token stays rejected)
                const uint32_t ui = uniform24(P.seed, P.iter[idx], (uint32_t)j, P.seq_id[idx], DRAW_ACCEPT);
                const float u = (float)ui * (1.0f / 16777216.0f);
                const int ok = __fmul_rn(u, q[(size_t)j * V + xs]) <= buf[j * len + xs] * f;
                for (int r = 0; r < SLICES; ++r) cluster.map_shared_rank(sh.ok, r)[j] = ok;
            }
        }
    }
    if (P.alpha_terms && gamma > 0) reduce_rows(gamma, false, sh.alpha); else cluster.sync();
    if (P.alpha_terms && rank == 0 && tid < gamma) {
        float a = 0.f;
#pragma unroll
        for (int r = 0; r < SLICES; ++r) a += sh.alpha[tid][r];
        P.alpha_terms[(size_t)b * gamma + tid] = a;
    }
    int nacc = 0;
    while (nacc < gamma && sh.ok[nacc]) ++nacc;
    // the draw: residual max(0, p_n - q_n), or p_gamma itself; all of it zero -> the target distribution -> its largest value
    float* w = buf + nacc * len;
    const float fn = factor(nacc);
    const float* qn = q + (size_t)(nacc < gamma ? nacc : 0) * V;
    const uint32_t ui = uniform24(P.seed, P.iter[idx], (uint32_t)nacc, P.seq_id[idx], DRAW_RESAMPLE);
    int y = 0, owner = -1;                                     // the CTA that writes the result, and (there) the token
    for (int attempt = nacc < gamma ? 0 : 1; attempt < 2 && owner < 0; ++attempt) {
        auto weight = [&](int k) { const float p = w[k] * fn; return attempt == 0 ? fmaxf(__fsub_rn(p, __ldg(qn + k)), 0.f) : p; };
        unsigned long long mine;
        const unsigned long long local = slice_weight(weight, n, &mine, sh.b);
        if (tid < SLICES) cluster.map_shared_rank(&sh.total[attempt][0], tid)[rank] = mine;
        cluster.sync();
        const SliceDraw d = slice_draw(sh.total[attempt], ui);
        owner = d.owner;
        if (owner == rank) y = base + max(slice_pick(weight, n, d.before, d.thr, local, sh.b), 0);
    }
    if (owner < 0) {                                           // the largest probability, lowest index on ties
        float pm = -INFINITY;
        for (int k = tid; k < n; k += 1024) pm = fmaxf(pm, w[k] * fn);
        pm = block_max(pm, sh.b.red);
        if (tid < SLICES) cluster.map_shared_rank(&sh.mx[0][0], tid)[rank] = pm;
        cluster.sync();
        pm = row_max(0);
        int best = 0x7fffffff;
        for (int k = tid; k < n; k += 1024) if (w[k] * fn == pm) { best = base + k; break; }
        best = block_min_int(best, sh.b);
        if (tid < SLICES) cluster.map_shared_rank(&sh.arg[0][0], tid)[rank] = best;
        cluster.sync();
        y = sh.arg[0][0];
#pragma unroll
        for (int r = 1; r < SLICES; ++r) y = min(y, sh.arg[0][r]);
        owner = 0;
    }
    if (owner == rank) {
        if (tid == 0) P.n_acc[b] = nacc;
        if (tid <= gamma) P.out_tok[(size_t)b * rows + tid] = tid < nacc ? x[tid] : (tid == nacc ? y : -1);
    }
    cluster.sync();                                            // no CTA leaves while the others may still write into it
}

// Where that is the faster form, by what both take: a wave of slices costs its barriers, a barrier or two per row, and a little per value; a
// wave of CTAs with a row each costs its row's length, twice from nine rows on.  Coefficients (us, rows, values) for logits with a
// temperature, greedy logits and probabilities as given, from 1,000...50,000 values, 1...16 rows, 1...64 sequences.  One wave, 12288 / 32000
// values, sliced and a CTA per row: with a temperature 2 rows 11.8 / 12.6 and 17.6 / 33.3, 6 rows 18.6 / 19.0 and 17.1 / 32.8, 9 rows 23.4 / 24.0
// and 22.4 / 41.9, 16 rows 34.5 / 37 (24000) and 26.7 / 41; greedy 2 rows 12.2 / 12.7 and 14.3 / 24.0, 6 rows 20.6 / 21.0 and 14.1 / 24.3, 10 rows
// 28.4 / 28.9 and 20.5 / 34.9; as given 6 rows 13.4 / 14.4 and 11.6 / 18.5, 10 rows 16.4 / 16.4 and 14.4 / 22.1.
struct AcceptCost { double wave, row, row_value, one, one_value, some, some_value, two, two_value; };      // sliced; a row per CTA: one row in all, up to 8, more
static bool accept_sliced(int V, int rows, int n, bool logits, bool greedy) {
    static const AcceptCost SOFT = {8.5, 1.32, 2.1e-5, 7.0, 3.9e-4, 8.2, 7.7e-4, 10.7, 9.8e-4}, GREEDY = {8.0, 1.68, 1.5e-5, 7.0, 3.0e-4, 8.0, 5.1e-4, 11.2, 7.4e-4},
                            GIVEN = {9.2, 0.6, 0.5e-5, 7.5, 1.5e-4, 8.6, 2.3e-4, 10.5, 2.7e-4};
    if ((size_t)slice_len(V) * rows * sizeof(float) > (size_t)STAGE_MAX_BYTES || rows > ACC_MAX_ROWS) return false;
    if (!row_stage_bytes(V)) return true;                      // (64000 values, 3 rows, with a temperature: 18 against 120)
    const AcceptCost& c = !logits ? GIVEN : greedy ? GREEDY : SOFT;
    const int more = std::min(std::max(rows - 9, 0), 3);       // (up to twelve rows more and more CTAs have two)
    const double row = rows == 1 ? c.one + c.one_value * V : rows <= 8 ? c.some + c.some_value * V : c.two + 0.33 * more + c.two_value * (1 + 0.07 * more) * V;
    const int side_by_side = rows > 4 ? SLICED_WAVE : rows > 2 ? 36 : 148;       // clusters of eight, four, and fewer CTAs
    return sliced_waves(n) * (c.wave + rows * (c.row + c.row_value * V)) < (n + side_by_side - 1) / side_by_side * row;
}

cudaError_t launch_accept(const AcceptParams& p, int dependent, cudaStream_t st) {
    if (p.B <= 0) return cudaSuccess;
    const size_t slices = (size_t)slice_len(p.V) * (p.gamma + 1) * sizeof(float);
    if (accept_sliced(p.V, p.gamma + 1, p.B, p.target_is_logits != 0, p.T == 0.f)) {
        cudaError_t e = cudaFuncSetAttribute(k_accept_sliced, cudaFuncAttributeMaxDynamicSharedMemorySize, STAGE_MAX_BYTES);
        if (e != cudaSuccess) return e;
        return launch_pdl(k_accept_sliced, dim3(p.B * SLICES), dim3(1024), slices, st, dependent, p);
    }
    int csize = 1;
    while (csize < p.gamma + 1 && csize < 8) csize <<= 1;      // portable cluster sizes only
    if (csize * ACC_ROWS_PER_CTA < p.gamma + 1) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    const size_t smem = row_stage_bytes(p.V);
    cudaError_t e = cudaFuncSetAttribute(k_accept, cudaFuncAttributeMaxDynamicSharedMemorySize, STAGE_MAX_BYTES);
    if (e != cudaSuccess) return e;
    cfg.gridDim = dim3(p.B * csize); cfg.blockDim = dim3(1024); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = csize; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = dependent ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, k_accept, p, csize, (int)(smem > 0));
}

}  // namespace sd
