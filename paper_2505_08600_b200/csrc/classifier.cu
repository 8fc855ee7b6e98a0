// Prompt classifier, MLP variant (embedding, two fully connected layers, softmax -> argmax):
// routes each prompt to one of the heterogeneous draft models.
#include <cooperative_groups.h>

#include "kernels.h"

namespace sd {

constexpr int CLF_CTAS = 8, CLF_WARPS = 16;
constexpr int CLF_PART_BYTES = CLF_WARPS * 256 * 4, CLF_MAX_SMEM = 227 * 1024 - CLF_PART_BYTES;      // static, and the dynamic shared memory left

// Eight consecutive columns of an embedding row, added to acc.
__device__ __forceinline__ void add_cols(const bf16* p, float (&acc)[8]) {
    const uint4 raw = __ldg(reinterpret_cast<const uint4*>(p));
    const __nv_bfloat162* v = reinterpret_cast<const __nv_bfloat162*>(&raw);
#pragma unroll
    for (int i = 0; i < 4; ++i) { const float2 f = __bfloat1622float2(v[i]); acc[2 * i] += f.x; acc[2 * i + 1] += f.y; }
}
__device__ __forceinline__ void add_cols(const float* p, float (&acc)[8]) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(p)), b = __ldg(reinterpret_cast<const float4*>(p) + 1);
    acc[0] += a.x; acc[1] += a.y; acc[2] += a.z; acc[3] += a.w; acc[4] += b.x; acc[5] += b.y; acc[6] += b.z; acc[7] += b.w;
}

// Bound: latency of the embedding rows (n d values; a prompt of 480 tokens at d = 2048 is 2 MB) and of w1.  A cluster of eight
// CTAs per sequence: each pools an eighth of the columns (warp = every 16th token, lane = 8 columns), hands its part of the
// mean to all eight, and takes an eighth of the hidden layer; the first CTA finishes.  Five prompts of 37...480 tokens, 1B
// target: 18 us (one CTA per sequence with a thread per column and the tokens one after the other: 826 us).
template <typename T>
__global__ void __cluster_dims__(CLF_CTAS, 1, 1) __launch_bounds__(32 * CLF_WARPS)
k_classifier(SeqState S, SeqList list, SeqList forced, const T* __restrict__ embed, int d, int vocab, const float* __restrict__ w1,
             const float* __restrict__ b1, int dh, const float* __restrict__ w2, const float* __restrict__ b2, int nc) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) float sm[];
    float* e = sm;                               // [d] mean-pooled prompt embedding (d is a multiple of 8)
    float* z = sm + d;                           // [dh] hidden activations (first CTA)
    float* o = z + dh;                           // [nc] class scores (first CTA)
    __shared__ float part[CLF_WARPS][256];
    const int i = blockIdx.x / CLF_CTAS, rank = blockIdx.x % CLF_CTAS, slot = list.ids[i];
    if (forced.ids[i] >= 0) {                    // task type given with the request: no classification (uniform in the cluster)
        if (rank == 0 && threadIdx.x == 0) S.draft_id[slot] = min(forced.ids[i], nc - 1);
        return;
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n = S.n_prompt[slot];
    const int32_t* toks = S.tokens + (size_t)slot * S.tok_stride;
    const int per = (d / 8 + CLF_CTAS - 1) / CLF_CTAS * 8, k0 = min(d, rank * per), k1 = min(d, k0 + per);
    cluster.sync();                              // every CTA of the cluster is there before the others write into it
    for (int kb = k0; kb < k1; kb += 256) {
        float acc[8] = {};
        const int k = kb + 8 * lane;
        if (k < k1) {
#pragma unroll 4
            for (int t = warp; t < n; t += CLF_WARPS) {
                int tok = __ldg(toks + t);
                tok = (tok < 0 || tok >= vocab) ? 0 : tok;
                add_cols(embed + (size_t)tok * d + k, acc);
            }
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) part[warp][8 * lane + c] = acc[c];
        __syncthreads();
        if (threadIdx.x < 256 && kb + (int)threadIdx.x < k1) {
            float sum = 0.f;
#pragma unroll
            for (int w = 0; w < CLF_WARPS; ++w) sum += part[w][threadIdx.x];
            const float mean = sum / (float)n;
            for (int r = 0; r < CLF_CTAS; ++r) cluster.map_shared_rank(e, r)[kb + threadIdx.x] = mean;
        }
        __syncthreads();
    }
    cluster.sync();
    float* z0 = cluster.map_shared_rank(z, 0);
    for (int j = rank * CLF_WARPS + warp; j < dh; j += CLF_CTAS * CLF_WARPS) {
        const float4* w = reinterpret_cast<const float4*>(w1 + (size_t)j * d);
        float acc = 0.f;
#pragma unroll 4
        for (int k = lane; k < d / 4; k += 32) {
            const float4 a = __ldg(w + k), b = reinterpret_cast<const float4*>(e)[k];
            acc = fmaf(a.x, b.x, acc); acc = fmaf(a.y, b.y, acc); acc = fmaf(a.z, b.z, acc); acc = fmaf(a.w, b.w, acc);
        }
        acc = warp_sum(acc);
        if (lane == 0) z0[j] = fmaxf(acc + b1[j], 0.f);
    }
    cluster.sync();
    if (rank != 0) return;
    for (int c = warp; c < nc; c += CLF_WARPS) {
        float acc = 0.f;
        for (int j = lane; j < dh; j += 32) acc = fmaf(w2[(size_t)c * dh + j], z[j], acc);
        acc = warp_sum(acc);
        if (lane == 0) o[c] = acc + b2[c];
    }
    __syncthreads();
    if (threadIdx.x == 0) {                      // softmax is monotone: its argmax is the argmax of the scores
        int best = 0;
        for (int c = 1; c < nc; ++c) if (o[c] > o[best]) best = c;
        S.draft_id[slot] = best;
    }
}

cudaError_t launch_classifier(const SeqState& S, const SeqList& list, const SeqList& forced,
                              const void* embed, int dtype, int d, int vocab,
                              const float* w1, const float* b1, int d_hidden, const float* w2, const float* b2,
                              int n_classes, cudaStream_t st) {
    if (list.n <= 0) return cudaSuccess;
    size_t smem = sizeof(float) * (size_t)(d + d_hidden + n_classes);
    if (smem > (size_t)CLF_MAX_SMEM) return cudaErrorInvalidValue;
    // (always the largest, not this call's: another context's call on another thread must not lower it before the launch)
    const cudaError_t err = dtype == SD_BF16 ? cudaFuncSetAttribute(k_classifier<bf16>, cudaFuncAttributeMaxDynamicSharedMemorySize, CLF_MAX_SMEM)
                                             : cudaFuncSetAttribute(k_classifier<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, CLF_MAX_SMEM);
    if (err != cudaSuccess) return err;
    if (dtype == SD_BF16) k_classifier<bf16><<<list.n * CLF_CTAS, 32 * CLF_WARPS, smem, st>>>(S, list, forced, (const bf16*)embed, d, vocab, w1, b1, d_hidden, w2, b2, n_classes);
    else k_classifier<float><<<list.n * CLF_CTAS, 32 * CLF_WARPS, smem, st>>>(S, list, forced, (const float*)embed, d, vocab, w1, b1, d_hidden, w2, b2, n_classes);
    return cudaGetLastError();
}

}  // namespace sd
