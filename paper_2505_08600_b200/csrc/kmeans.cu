// One Lloyd iteration of K-means over dense fp32 vectors (the offline task-partitioning step, Section 3.2:
// 384-dimensional sentence vectors, a handful of clusters).
//
// With K <= 8 centroids the step is a single pass over the points and is bound by that pass (4 K flop per loaded
// byte-quad: far below the ALU ridge), so the kernel is a streaming one, not a tensor-core contraction: a warp takes
// whole points, every lane owns dim / 32 columns (float4 loads, one coalesced row per warp), the centroids sit in
// shared memory, squared distances are summed in fp32 and reduced with shuffles.  The same pass accumulates, per warp
// and in registers, the sum of the points of every cluster; warps of a block are added in warp order, blocks in block
// order by a second small kernel: the new centroids, the counts and the inertia are identical from run to run.
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/sd.h"
#include "f32x2.cuh"

namespace sd {
namespace {

constexpr int KM_MAX_K = 8;
// Points of a warp that its ring holds, warps of a CTA and CTAs of an SM, for 128 nv components and up to km clusters.  Two points at a
// time with four centroids in registers take 160 registers at 384 components: one CTA of twelve warps; 512: eight warps; fewer
// components, or two centroids: two CTAs of eight (rings of six points at 512, so that two fit the shared memory).
constexpr __host__ __device__ int km_depth(int nv, int km) { return km == 8 || (km == 2 && nv == 4) ? 6 : 8; }
constexpr __host__ __device__ int km_warps(int nv, int km) { return km == 4 && nv == 3 ? 12 : 8; }
constexpr __host__ __device__ int km_per_sm(int nv, int km) { return km == 4 && nv >= 3 ? 1 : 2; }
constexpr int KM_RUN = 128;            // points in one run of fp32 sums, where a warp keeps runs

template <int NV, int KM>          // KM: compiled cluster bound (2, 4 or 8); up to 4 the centroids are kept in registers
__global__ void __launch_bounds__(32 * km_warps(NV, KM), KM == 8 ? 1 : km_per_sm(NV, KM))
k_kmeans_assign(const float* __restrict__ pts, long long n, int k, const float* __restrict__ cent, int32_t* __restrict__ labels,
                float* __restrict__ part_sums, long long* __restrict__ part_counts, double* __restrict__ part_inertia) {
    constexpr int DIM = 128 * NV, KM_WARPS = km_warps(NV, KM), KM_DEPTH = km_depth(NV, KM);
    extern __shared__ __align__(16) float km_smem[];
    float* cs = km_smem;                       // [k][DIM] centroids
    float* acc_s = km_smem + KM * DIM;         // [k][DIM] the block's sums
    __shared__ long long cnt_s[KM];
    __shared__ double inertia_s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < k * DIM; i += blockDim.x) cs[i] = cent[i];
    __syncthreads();

    // Up to four centroids: every lane keeps its columns of them in registers (shared memory could not feed four
    // centroid reads per point at the rate the points arrive); more: read from shared memory.
    constexpr bool CREG = KM <= 4;
    ulonglong2 creg[CREG ? KM : 1][CREG ? NV : 1];
    if (CREG) {
#pragma unroll
        for (int kk = 0; kk < KM; ++kk)
#pragma unroll
            for (int v = 0; v < NV; ++v)
                creg[CREG ? kk : 0][CREG ? v : 0] = kk < k ? *reinterpret_cast<const ulonglong2*>(cs + kk * DIM + (v * 32 + lane) * 4) : make_ulonglong2(0ull, 0ull);
    }
    ulonglong2 acc[KM][NV];                     // (the bit pattern 0 is +0.0f twice)
#pragma unroll
    for (int kk = 0; kk < KM; ++kk)
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[kk][v] = make_ulonglong2(0ull, 0ull);
    int cnt = 0;                                // lane kk: points of this warp in cluster kk (a warp sees n / (KM_WARPS * blocks) points)
    double inertia = 0.0;

    // Every lane copies its own columns of its warp's next points (KM_DEPTH - 1 of them, KM_DEPTH - 2 two at a time) into shared memory
    // with asynchronous 16-byte copies and reads back only what it copied itself: no barrier, and enough bytes in flight per SM
    // (warps x depth x row) to cover the memory latency at full bandwidth.
    const long long total_warps = (long long)gridDim.x * KM_WARPS;
    const long long i0 = (long long)blockIdx.x * KM_WARPS + warp;
    float* ring = acc_s + KM * DIM + (size_t)warp * KM_DEPTH * DIM + lane * 4;     // [KM_DEPTH][DIM] of this warp, this lane's first column
    const uint32_t ring_sa = (uint32_t)__cvta_generic_to_shared(ring);
    const float* src_next = pts + i0 * DIM + lane * 4;                            // the next point to request and its index
    long long idx_next = i0;
    const long long src_step = total_warps * DIM;
    int slot_next = 0;
    auto stage = [&]() {
        if (idx_next < n) {
#pragma unroll
            for (int v = 0; v < NV; ++v)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(ring_sa + (uint32_t)(slot_next * DIM + v * 128) * 4u), "l"(src_next + v * 128) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");                      // (an empty group past the end keeps the count uniform)
        idx_next += total_warps; src_next += src_step;
        slot_next = slot_next + 1 == KM_DEPTH ? 0 : slot_next + 1;
    };
    // One CTA per SM has fewer warps than two, and so more points in each warp's fp32 sums: there a lane moves its sums to shared memory
    // every KM_RUN points and begins anew (no other lane reads them: no barrier).  Error against 64 bits of the centroid of a million copies
    // of one 512-component point: 0.9e-6; 6.1e-6 without; two CTAs per SM: 3.0e-6.  2,000,003 x 384, 4 clusters: 616 -> 622 us
    // (every 256 points: 621).
    constexpr bool RUNS = km_per_sm(NV, KM) == 1 && KM == 4;
    // [KM][DIM] of this warp, this lane's first column: behind the rings; the first warp's where the block's sums will be, which it writes first
    float* runs = (warp == 0 ? acc_s : acc_s + KM * DIM + KM_WARPS * KM_DEPTH * DIM + (warp - 1) * KM * DIM) + lane * 4;
    bool moved = false;
    auto move_sums = [&]() {
#pragma unroll
        for (int kk = 0; kk < KM; ++kk)
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                ulonglong2* dst = reinterpret_cast<ulonglong2*>(runs + kk * DIM + v * 128);
                if (moved) { const ulonglong2 s = *dst; acc[kk][v].x = f2_add(s.x, acc[kk][v].x); acc[kk][v].y = f2_add(s.y, acc[kk][v].y); }
                *dst = acc[kk][v];
                acc[kk][v] = make_ulonglong2(0ull, 0ull);
            }
        moved = true;
    };
    int slot = 0;
    auto ring_at = [&](int sl, int v) { return *reinterpret_cast<const ulonglong2*>(ring + sl * DIM + v * 128); };
    auto partial = [&](const ulonglong2 (&x)[NV], int kk) {                       // this lane's share of a squared distance
        f32x2 d2 = 0ull;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const ulonglong2 c = creg[CREG ? kk : 0][CREG ? v : 0];
            const f32x2 a = f2_sub(x[v].x, c.x), b = f2_sub(x[v].y, c.y);
            d2 = f2_fma(a, a, d2); d2 = f2_fma(b, b, d2);
        }
        return f2_hsum(d2);
    };
    auto count = [&](const ulonglong2 (&x)[NV], int label) {                      // label: uniform
        cnt += label == lane ? 1 : 0;
#pragma unroll
        for (int kk = 0; kk < KM; ++kk) {
            if (kk == label) {
#pragma unroll
                for (int v = 0; v < NV; ++v) { acc[kk][v].x = f2_add(acc[kk][v].x, x[v].x); acc[kk][v].y = f2_add(acc[kk][v].y, x[v].y); }
            }
        }
    };
    if (KM <= 4) {
        // Two points at a time (four clusters): their eight sums over the warp cost nine shuffles (halves of the warp trade one point for the other,
        // then clusters), the smallest of four per half four more, and the two chains of latencies run side by side; the distances are
        // added in the same order as one by one.  2,000,003 x 384, 4 clusters: 636 us one point at a time (16 warps per SM of 128
        // registers), 579 with two points, twelve warps of 168 registers (at 128 registers they spill: 1,100); 4,000,000 x 128:
        // 691 and 564; 1,000,000 x 512: 429 and 408.  A ring of ten points is no faster than one of eight.
        // One or two clusters have a form of their own (1,000,003 x 256 and 512, two clusters: 223 and 429 us one point at a time, 234 and
        // 449 with four sums for two, 192 and 354 with two).
        constexpr int AHEAD = KM_DEPTH - 2;
        for (int t = 0; t < AHEAD; ++t) stage();
        for (long long i = i0; i < n;) {
            const long long i_end = RUNS ? min(n, i + KM_RUN * total_warps) : n;
            for (; i < i_end; i += 2 * total_warps) {
                stage(); stage();
                asm volatile("cp.async.wait_group %0;" ::"n"(AHEAD) : "memory");       // these two points have landed
                const int slot1 = slot + 1 == KM_DEPTH ? 0 : slot + 1;
                const bool both = i + total_warps < n;                                // uniform
                float d[2][KM];
                ulonglong2 x0[NV], x1[NV];
#pragma unroll
                for (int v = 0; v < NV; ++v) { x0[v] = ring_at(slot, v); x1[v] = ring_at(slot1, v); }
#pragma unroll
                for (int kk = 0; kk < KM; ++kk) {                                     // (centroids past k are zeros and drop out below)
                    d[0][kk] = partial(x0, CREG ? kk : 0);
                    d[1][kk] = partial(x1, CREG ? kk : 0);
                }
                const bool hi16 = lane & 16, hi8 = lane & 8, hi4 = lane & 4;
                float a[KM];
#pragma unroll
                for (int kk = 0; kk < KM; ++kk) a[kk] = (hi16 ? d[1][kk] : d[0][kk]) + __shfl_xor_sync(0xffffffffu, hi16 ? d[0][kk] : d[1][kk], 16);
                float e;
                if (KM == 2) {
                    e = (hi8 ? a[1] : a[0]) + __shfl_xor_sync(0xffffffffu, hi8 ? a[0] : a[1], 8);
                    e += __shfl_xor_sync(0xffffffffu, e, 4);
                } else {
                    constexpr int K2 = KM > 2 ? 2 : 0, K3 = KM > 2 ? 3 : 0;
                    const float b0 = (hi8 ? a[K2] : a[0]) + __shfl_xor_sync(0xffffffffu, hi8 ? a[0] : a[K2], 8);
                    const float b1 = (hi8 ? a[K3] : a[1]) + __shfl_xor_sync(0xffffffffu, hi8 ? a[1] : a[K3], 8);
                    e = (hi4 ? b1 : b0) + __shfl_xor_sync(0xffffffffu, hi4 ? b0 : b1, 4);
                }
                e += __shfl_xor_sync(0xffffffffu, e, 2);
                e += __shfl_xor_sync(0xffffffffu, e, 1);
                // a lane's bit 4 is the point, bits 3 and 2 are the cluster (two clusters: bit 3); the smallest wins, the lowest index on ties
                int label = KM == 2 ? (hi8 ? 1 : 0) : (hi8 ? 2 : 0) + (hi4 ? 1 : 0);
                if (label >= k || !(e == e)) e = INFINITY;
#pragma unroll
                for (int o = KM == 2 ? 8 : 4; o <= 8; o <<= 1) {
                    const float e2 = __shfl_xor_sync(0xffffffffu, e, o);
                    const int l2 = __shfl_xor_sync(0xffffffffu, label, o);
                    if (e2 < e || (e2 == e && l2 < label)) { e = e2; label = l2; }
                }
                if (!hi16 || both) {
                    inertia += (double)e;                                             // (the lower half sums the first points, the upper half the second ones)
                    if ((lane & 15) == 0) labels[hi16 ? i + total_warps : i] = label;
                }
                const int label0 = __shfl_sync(0xffffffffu, label, 0), label1 = __shfl_sync(0xffffffffu, label, 16);
                count(x0, label0);
                if (both) count(x1, label1);
                slot = slot1 + 1 == KM_DEPTH ? 0 : slot1 + 1;
            }
            if (RUNS && i < n) move_sums();
        }
        inertia += __shfl_sync(0xffffffffu, inertia, 16);                         // (what lane 0 writes)
    } else {
        for (int t = 0; t < KM_DEPTH - 1; ++t) stage();
        for (long long i = i0; i < n; i += total_warps) {
            stage();
            asm volatile("cp.async.wait_group %0;" ::"n"(KM_DEPTH - 1) : "memory");    // this point has landed
            ulonglong2 x[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) x[v] = ring_at(slot, v);
            float dk[KM];                                                         // this lane's share of every squared distance
#pragma unroll
            for (int kk = 0; kk < KM; ++kk) {
                dk[kk] = 0.f;
                if (kk < k) {                                                     // uniform
                    f32x2 d2 = 0ull;
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        const ulonglong2 c = *reinterpret_cast<const ulonglong2*>(cs + kk * DIM + (v * 32 + lane) * 4);
                        const f32x2 a = f2_sub(x[v].x, c.x), b = f2_sub(x[v].y, c.y);
                        d2 = f2_fma(a, a, d2); d2 = f2_fma(b, b, d2);
                    }
                    dk[kk] = f2_hsum(d2);
                }
            }
#pragma unroll
            for (int kk = 0; kk < KM; ++kk)
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) dk[kk] += __shfl_xor_sync(0xffffffffu, dk[kk], o);      // every lane ends with the same sums
            float best = INFINITY;
            int label = 0;
#pragma unroll
            for (int kk = 0; kk < KM; ++kk)
                if (kk < k && dk[kk] < best) { best = dk[kk]; label = kk; }        // a later centroid must be strictly closer
            if (lane == 0) labels[i] = label;
            inertia += (double)best;
            count(x, label);
            slot = slot + 1 == KM_DEPTH ? 0 : slot + 1;
        }
    }

    if (RUNS && moved) {
#pragma unroll
        for (int kk = 0; kk < KM; ++kk)
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const ulonglong2 s = *reinterpret_cast<const ulonglong2*>(runs + kk * DIM + v * 128);
                acc[kk][v].x = f2_add(s.x, acc[kk][v].x); acc[kk][v].y = f2_add(s.y, acc[kk][v].y);
            }
    }

    // the block's sums: its warps in warp order
    for (int w = 0; w < KM_WARPS; ++w) {
        if (warp == w) {
#pragma unroll
            for (int kk = 0; kk < KM; ++kk) {
                if (kk < k) {
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        ulonglong2* dst = reinterpret_cast<ulonglong2*>(acc_s + kk * DIM + (v * 32 + lane) * 4);
                        ulonglong2 s = w == 0 ? make_ulonglong2(0ull, 0ull) : *dst;
                        s.x = f2_add(s.x, acc[kk][v].x); s.y = f2_add(s.y, acc[kk][v].y);
                        *dst = s;
                    }
                    if (lane == kk) cnt_s[kk] = (w == 0 ? 0 : cnt_s[kk]) + (long long)cnt;
                }
            }
            if (lane == 0) inertia_s = (w == 0 ? 0.0 : inertia_s) + inertia;
        }
        __syncthreads();
    }
    for (int i = threadIdx.x; i < k * DIM; i += blockDim.x) part_sums[(size_t)blockIdx.x * k * DIM + i] = acc_s[i];
    if (threadIdx.x < k) part_counts[(size_t)blockIdx.x * k + threadIdx.x] = cnt_s[threadIdx.x];
    if (threadIdx.x == 0) part_inertia[blockIdx.x] = inertia_s;
}

// New centroids = (sum over blocks) / count; a cluster without points keeps its centroid.  One CTA per (cluster, 32
// columns): eight threads per column each add a contiguous run of the blocks' partial sums in block order (independent
// loads, several in flight), and the eight runs are added in run order: a fixed order, in double.
__global__ void __launch_bounds__(256)
k_kmeans_reduce(const float* __restrict__ part_sums, const long long* __restrict__ part_counts,
                const double* __restrict__ part_inertia, int n_blocks, int k, int dim,
                const float* __restrict__ cent, float* __restrict__ cent_out, long long* __restrict__ counts_out,
                double* __restrict__ inertia_out) {
    __shared__ double run_sum[8][32];
    __shared__ long long run_cnt[8];
    __shared__ double run_in[8];
    const int kk = blockIdx.x, d = blockIdx.y * 32 + (threadIdx.x & 31), run = threadIdx.x >> 5;
    const int per = (n_blocks + 7) / 8, b0 = run * per, b1 = min(n_blocks, b0 + per);
    double s = 0.0;
    if (d < dim) {
#pragma unroll 8
        for (int b = b0; b < b1; ++b) s += (double)__ldcg(part_sums + ((size_t)b * k + kk) * dim + d);
    }
    run_sum[run][threadIdx.x & 31] = s;
    {   // the run's counts and inertia: a lane per block, then a fixed tree over the lanes
        long long c = 0;
        double in = 0.0;
        for (int b = b0 + (int)(threadIdx.x & 31); b < b1; b += 32) { c += part_counts[(size_t)b * k + kk]; in += part_inertia[b]; }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { c += __shfl_xor_sync(0xffffffffu, c, o); in += __shfl_xor_sync(0xffffffffu, in, o); }
        if ((threadIdx.x & 31) == 0) { run_cnt[run] = c; run_in[run] = in; }
    }
    __syncthreads();
    if (run != 0) return;
    long long c = 0;
    double tot = 0.0, in = 0.0;
    for (int r = 0; r < 8; ++r) { c += run_cnt[r]; tot += run_sum[r][threadIdx.x]; in += run_in[r]; }
    if (d < dim && cent_out) cent_out[(size_t)kk * dim + d] = c > 0 ? (float)(tot / (double)c) : cent[(size_t)kk * dim + d];
    if (threadIdx.x == 0 && blockIdx.y == 0) {
        if (counts_out) counts_out[kk] = c;
        if (kk == 0 && inertia_out) *inertia_out = in;
    }
}

int km_blocks() {
    int dev = 0, n_sm = 148;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    return 2 * n_sm;
}

size_t km_align(size_t v) { return (v + 255) & ~(size_t)255; }

}  // namespace
}  // namespace sd

extern "C" size_t sd_kmeans_workspace(int dim, int k) {
    if (dim < 1 || k < 1) return 0;
    const size_t b = (size_t)sd::km_blocks();
    return sd::km_align(b * k * dim * sizeof(float)) + sd::km_align(b * k * sizeof(long long)) + sd::km_align(b * sizeof(double));
}

extern "C" sd_status sd_kmeans_step(const float* points, int64_t n, int dim, const float* centroids, int k, int32_t* labels,
                                    float* centroids_out, int64_t* counts_out, double* inertia_out, void* workspace,
                                    size_t workspace_bytes, void* cuda_stream) {
    using namespace sd;
    if (!centroids || n < 0 || k < 1 || dim < 1 || (n > 0 && (!points || !labels))) return SD_ERR_INVALID_ARG;
    if (k > KM_MAX_K || (dim % 128) || dim > 512) return SD_ERR_UNSUPPORTED;
    if (((uintptr_t)points & 15) || ((uintptr_t)centroids & 15)) return SD_ERR_INVALID_ARG;
    if (!workspace || workspace_bytes < sd_kmeans_workspace(dim, k)) return SD_ERR_CAPACITY;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const int km = k <= 2 ? 2 : k <= 4 ? 4 : KM_MAX_K;
    // (two clusters of few long vectors: one CTA per SM as well, whose set-up and partial sums are half as many.  3,000 x 384: 18.5 us, with
    // two 22.6; 512: 18.5 and 23.4)
    const bool few = km == 2 && dim >= 384 && n < 16 * km_warps(dim / 128, km) * (km_blocks() / 2);
    const int blocks = km_blocks() / (few ? 2 : 2 / km_per_sm(dim / 128, km));
    char* w = (char*)workspace;
    float* part_sums = (float*)w;              w += km_align((size_t)blocks * k * dim * sizeof(float));
    long long* part_counts = (long long*)w;    w += km_align((size_t)blocks * k * sizeof(long long));
    double* part_inertia = (double*)w;
    const int warps = km_warps(dim / 128, km), runs = km == 4 && km_per_sm(dim / 128, km) == 1 ? (warps - 1) * km : 0;
    const size_t smem = ((size_t)2 * km + (size_t)warps * km_depth(dim / 128, km) + runs) * dim * sizeof(float);
    cudaError_t e = cudaSuccess;
#define KM_LAUNCH(NV, KM)                                                                                                        \
    do {                                                                                                                     \
        e = cudaFuncSetAttribute(k_kmeans_assign<NV, KM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);           \
        if (e == cudaSuccess) k_kmeans_assign<NV, KM><<<blocks, 32 * km_warps(NV, KM), smem, st>>>(points, n, k, centroids, labels, part_sums, part_counts, part_inertia); \
    } while (0)
    switch (dim / 128) {
    case 1: if (km == 2) KM_LAUNCH(1, 2); else if (km == 4) KM_LAUNCH(1, 4); else KM_LAUNCH(1, 8); break;
    case 2: if (km == 2) KM_LAUNCH(2, 2); else if (km == 4) KM_LAUNCH(2, 4); else KM_LAUNCH(2, 8); break;
    case 3: if (km == 2) KM_LAUNCH(3, 2); else if (km == 4) KM_LAUNCH(3, 4); else KM_LAUNCH(3, 8); break;
    default: if (km == 2) KM_LAUNCH(4, 2); else if (km == 4) KM_LAUNCH(4, 4); else KM_LAUNCH(4, 8); break;
    }
#undef KM_LAUNCH
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return SD_ERR_CUDA;
    k_kmeans_reduce<<<dim3(k, (dim + 31) / 32), 256, 0, st>>>(part_sums, part_counts, part_inertia, blocks, k, dim, centroids, centroids_out,
                                       (long long*)counts_out, inertia_out);
    return cudaGetLastError() == cudaSuccess ? SD_OK : SD_ERR_CUDA;
}
