// The layers of an fp32 model over a few token rows: every matrix and the step that follows it as one kernel.
//
// Such models are small and a pass over a few rows is a chain of launches (thirteen per layer on the plain path, 1.3-3 us each,
// for matrices that L2 delivers in far less): norm, matrix and step are one kernel here, five launches per layer, each a
// programmatic dependent of the one before with its weights in registers before the wait.  A warp owns a unit of two output
// features that the step needs together (a rotary pair, gate and up, or just two rows) and the whole reduction.  RMSNorm is
// folded around the product: the rows enter as h * gain, and the warp that reads all of a row has its sum of squares as well.
// Everything in fp32.  Bound by the chain of launches and one memory latency each.  (Iteration of the tiny fp32 pair, 2 + 2 layers
// of d 128 to 256, K = 4: 204 us through the plain kernels, 156 with the rows read from L2 by every warp, 154 with the rows
// fetched into shared memory once per CTA.)
#include "gemm_tc.h"
#include <algorithm>
#include <type_traits>

#include "plain_steps.h"

namespace sd {
namespace {

constexpr int PS_ROW_BYTES = 96 * 1024;                // shared memory for the rows
constexpr int PS_WARPS = 8, PS_VECS = 6;                  // float4 of a weight row per lane and round: 768 elements

template <int MODE, int M>
__global__ void __launch_bounds__(32 * PS_WARPS) k_plain_step(const __grid_constant__ PlainStep p) {
    constexpr bool NORM = MODE == PS_QKV || MODE == PS_GU || MODE == PS_LM;
    extern __shared__ __align__(16) float x_sm[];          // [rows][K]: fetched in one round of loads by the whole CTA
    pdl_launch_dependents();
    const int lane = threadIdx.x & 31, u = blockIdx.x * PS_WARPS + (threadIdx.x >> 5);
    const int units = MODE == PS_GU ? p.F : (p.n_out + 1) / 2, half = p.hd >> 1;
    const bool live = u < units;
    const int f0 = MODE == PS_QKV ? u / half * p.hd + u % half : u;
    const int f1 = MODE == PS_QKV ? f0 + half : MODE == PS_GU ? p.F + u : u + units;
    const bool live1 = live && f1 < p.n_out;
    const int K4 = p.K >> 2;
    const float4* w0 = reinterpret_cast<const float4*>(p.w + (size_t)f0 * p.K);
    const float4* w1 = reinterpret_cast<const float4*>(p.w + (size_t)f1 * p.K);
    const float4* gn = reinterpret_cast<const float4*>(p.gain);
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 a[PS_VECS], b[PS_VECS], g[NORM ? PS_VECS : 1];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int i = 0; i < PS_VECS; ++i) {
            const int k = k0 + lane + 32 * i;
            a[i] = live && k < K4 ? __ldg(w0 + k) : zero;
            b[i] = live1 && k < K4 ? __ldg(w1 + k) : zero;
            if (NORM) g[NORM ? i : 0] = k < K4 ? __ldg(gn + k) : zero;
        }
    };
    fetch(0);
    pdl_wait();                                           // rows, residual stream and row plan come from the kernels before
    float4* xs = reinterpret_cast<float4*>(x_sm);
    for (int m = 0; m < p.rows; ++m) {
        const int r = MODE == PS_LM ? m * p.row_stride + p.row_offset : m;
        for (int k = threadIdx.x; k < K4; k += 32 * PS_WARPS) xs[m * K4 + k] = __ldcg(reinterpret_cast<const float4*>(p.x + (size_t)r * p.K) + k);
    }
    __syncthreads();
    float s0[M], s1[M], ss[M];
#pragma unroll
    for (int m = 0; m < M; ++m) s0[m] = s1[m] = ss[m] = 0.f;
    for (int k0 = 0; k0 < K4; k0 += 32 * PS_VECS) {
        if (k0) fetch(k0);
#pragma unroll
        for (int i = 0; i < PS_VECS; ++i) {
            const int k = k0 + lane + 32 * i;
            if (k0 + 32 * i >= K4) break;
#pragma unroll
            for (int m = 0; m < M; ++m) {
                float4 x = m < p.rows && k < K4 ? xs[m * K4 + k] : zero;
                if (NORM) {
                    ss[m] = fmaf(x.x, x.x, ss[m]); ss[m] = fmaf(x.y, x.y, ss[m]); ss[m] = fmaf(x.z, x.z, ss[m]); ss[m] = fmaf(x.w, x.w, ss[m]);
                    const float4 q = g[NORM ? i : 0];
                    x.x *= q.x; x.y *= q.y; x.z *= q.z; x.w *= q.w;
                }
                s0[m] = fmaf(a[i].x, x.x, s0[m]); s0[m] = fmaf(a[i].y, x.y, s0[m]); s0[m] = fmaf(a[i].z, x.z, s0[m]); s0[m] = fmaf(a[i].w, x.w, s0[m]);
                s1[m] = fmaf(b[i].x, x.x, s1[m]); s1[m] = fmaf(b[i].y, x.y, s1[m]); s1[m] = fmaf(b[i].z, x.z, s1[m]); s1[m] = fmaf(b[i].w, x.w, s1[m]);
            }
        }
    }
    float v0 = 0.f, v1 = 0.f;                             // lane m finishes row m
#pragma unroll
    for (int m = 0; m < M; ++m) {
        const float x0 = warp_sum(s0[m]), x1 = warp_sum(s1[m]);
        const float inv = NORM ? rsqrtf(warp_sum(ss[m]) / (float)p.K + p.eps) : 1.f;
        if (lane == m) { v0 = x0 * inv; v1 = x1 * inv; }
    }
    if (!live || lane >= p.rows || lane >= M) return;
    const int m = lane;
    if (MODE == PS_QKV) {
        const int pos = __ldcg(p.row_pos + m), head = u / half, e = u % half;
        if (pos < 0) return;
        if (head < p.H + p.Hkv) {
            const float c = __ldg(p.rcos + (size_t)pos * half + e), s = __ldg(p.rsin + (size_t)pos * half + e);
            const float ra = v0 * c - v1 * s, rb = v0 * s + v1 * c;
            v0 = ra; v1 = rb;
        }
        float* dst;
        if (head < p.H) dst = p.q + ((size_t)m * p.H + head) * p.hd + e;
        else {
            const bool is_v = head >= p.H + p.Hkv;
            dst = (is_v ? p.vc : p.kc) + (((size_t)__ldcg(p.row_slot + m) * p.Hkv + head - p.H - (is_v ? p.Hkv : 0)) * p.max_ctx + pos) * p.hd + e;
        }
        dst[0] = v0; dst[half] = v1;
    } else if (MODE == PS_RESIDUAL) {
        float* h = p.y + (size_t)m * p.n_out;
        h[f0] = __ldcg(h + f0) + v0;
        if (live1) h[f1] = __ldcg(h + f1) + v1;
    } else if (MODE == PS_GU) {
        p.y[(size_t)m * p.F + u] = v0 / (1.f + expf(-v0)) * v1;
    } else {
        float* y = p.y + (size_t)m * p.n_out;
        y[f0] = v0;
        if (live1) y[f1] = v1;
    }
}

// Attention of a few fp32 rows: a CTA per (row, query head), four lanes per key for the scores, as many groups of hd threads as
// there are for the values.  The scores of the whole context sit in shared memory.  Bound: latency of the loads, so PA_KEYS keys per
// lane (one up to 64 positions, with four parts of it) and PA_VALUES values per thread are on their way at a time, and the four lanes of a key
// read whole sectors.  (Verify pass of a 2-layer, 256-
// and 768-wide model, 5 rows, 8,000 positions: 614 and 928 us; one key and four values at a time, a quarter of a key per lane: 1,011 and 2,603;
// the plain kernels 686 and 1,486.  64 positions, 256 wide: 57.6; 59.5; 61.5.)
constexpr int PA_KEYS = 4, PA_VALUES = 16;
__global__ void __launch_bounds__(256) k_plain_attention(const float* __restrict__ q, const float* __restrict__ kc, const float* __restrict__ vc, float* __restrict__ out,
                                                         const int32_t* __restrict__ row_slot, const int32_t* __restrict__ row_pos, int H, int Hkv, int hd, int max_ctx) {
    extern __shared__ __align__(16) float sm[];
    __shared__ float red[32];
    __shared__ float acc_s[256];
    float* qs = sm;                                       // [hd]
    float* sc = sm + hd;                                  // [n_ctx]
    pdl_launch_dependents();
    const int r = blockIdx.x, h = blockIdx.y, t = threadIdx.x;
    pdl_wait();
    const int pos = __ldcg(row_pos + r), slot = __ldcg(row_slot + r);
    float* o = out + ((size_t)r * H + h) * hd;
    if (pos < 0) { for (int i = t; i < hd; i += 256) o[i] = 0.f; return; }
    const int n = pos + 1;
    const size_t base = ((size_t)slot * Hkv + h / (H / Hkv)) * (size_t)max_ctx * hd;
    const float* K = kc + base;
    const float* V = vc + base;
    const float scale = rsqrtf((float)hd);
    for (int i = t; i < hd; i += 256) qs[i] = __ldcg(q + ((size_t)r * H + h) * hd + i) * scale;
    __syncthreads();
    float mx = -INFINITY;
    const int part = t & 3;
    const float4* q4 = reinterpret_cast<const float4*>(qs);
    auto scores = [&](auto keys) {
        constexpr int KEYS = decltype(keys)::value;
        for (int p0 = t >> 2; p0 < n; p0 += 64 * KEYS) {  // (the four lanes of a key stay together)
            float sk[KEYS];
#pragma unroll
            for (int u = 0; u < KEYS; ++u) sk[u] = 0.f;
#pragma unroll 4
            for (int i = part; i < hd >> 2; i += 4) {     // hd is a multiple of 16
                float4 k[KEYS];
#pragma unroll
                for (int u = 0; u < KEYS; ++u) {
                    const int p = p0 + 64 * u;
                    k[u] = p < n ? __ldcg(reinterpret_cast<const float4*>(K + (size_t)p * hd) + i) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
                const float4 b = q4[i];
#pragma unroll
                for (int u = 0; u < KEYS; ++u) {
                    sk[u] = fmaf(k[u].x, b.x, sk[u]); sk[u] = fmaf(k[u].y, b.y, sk[u]); sk[u] = fmaf(k[u].z, b.z, sk[u]); sk[u] = fmaf(k[u].w, b.w, sk[u]);
                }
            }
            const unsigned four = 0xfu << (t & 28);
#pragma unroll
            for (int u = 0; u < KEYS; ++u) {
                sk[u] += __shfl_xor_sync(four, sk[u], 1);
                sk[u] += __shfl_xor_sync(four, sk[u], 2);
                const int p = p0 + 64 * u;
                if (p < n) { if (part == 0) sc[p] = sk[u]; mx = fmaxf(mx, sk[u]); }
            }
        }
    };
    // (up to 64 positions a lane has one key: four would only wait for parts of it; iteration of the tiny pair at 33 positions 157 us with four, 151)
    if (n <= 64) scores(std::integral_constant<int, 1>()); else scores(std::integral_constant<int, PA_KEYS>());
    mx = block_max(mx, red);
    float den = 0.f;
    for (int p = t; p < n; p += 256) { const float e = expf(sc[p] - mx); sc[p] = e; den += e; }
    den = block_sum(den, red);
    const int groups = 256 / hd, grp = t / hd, e = t % hd;
    float acc = 0.f;
    if (grp < groups) {
        for (int p0 = grp; p0 < n; p0 += groups * PA_VALUES) {
            float v[PA_VALUES];
#pragma unroll
            for (int u = 0; u < PA_VALUES; ++u) { const int p = p0 + groups * u; v[u] = p < n ? __ldcg(V + (size_t)p * hd + e) : 0.f; }
#pragma unroll
            for (int u = 0; u < PA_VALUES; ++u) { const int p = p0 + groups * u; if (p < n) acc = fmaf(sc[p], v[u], acc); }
        }
    }
    acc_s[t] = acc;
    __syncthreads();
    if (t < hd) {
        for (int i = 1; i < groups; ++i) acc += acc_s[i * hd + t];
        o[t] = acc * (1.f / den);
    }
}

template <int MODE>
cudaError_t launch_mode(const PlainStep& p, cudaStream_t st) {
    const int units = MODE == PS_GU ? p.F : (p.n_out + 1) / 2;
    const dim3 grid((units + PS_WARPS - 1) / PS_WARPS), block(32 * PS_WARPS);
    void (*kern)(const PlainStep) = p.rows <= 1 ? k_plain_step<MODE, 1> : p.rows <= 2 ? k_plain_step<MODE, 2> : p.rows <= 5 ? k_plain_step<MODE, 5> : k_plain_step<MODE, PS_MAX_ROWS>;
    const size_t smem = (size_t)p.rows * p.K * sizeof(float);
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, PS_ROW_BYTES);
    if (e != cudaSuccess) return e;
    return launch_pdl(kern, grid, block, smem, st, 1, p);
}

}  // namespace

// Up to five rows, each with two accumulators per unit in registers, up to eight where the largest matrix has 8 MB or more; that matrix at
// most 16 MB, so that L2 holds the model and launches, not bytes, are the bound (larger fp32 models keep the plain kernels).  A pass,
// plain / here, us: largest matrix 1.4 MB 1 row 55 / 39, 5 rows 66 / 61, 6 rows 67.6 / 71.6; 5.6 MB 127 / 80, 150 / 143, 163 / 165; 12.6 MB
// 210 / 146, 231 / 208, 248 / 242, 8 rows 273 / 259; 16.8 MB 229 / 165, 263 / 235, 284 / 278, 315 / 295; beyond the line, 32.8 MB: 249 / 182, 285 / 274,
// 304 / 317.
// Rows and scores have to fit in shared memory; head_dim % 16 == 0 for the float4 reads of a quarter of a key.
bool plain_steps_fit(const sd_model_desc& m, int rows, int max_ctx) {
    const size_t d = m.d_model, dq = (size_t)m.n_heads * m.head_dim, n_qkv = dq + 2 * (size_t)m.n_kv_heads * m.head_dim, F = m.d_ffn, V = m.vocab;
    const size_t largest = std::max(std::max(n_qkv * d, d * dq), std::max(2 * F * d, V * d)) * sizeof(float);
    return m.dtype == SD_F32 && rows >= 1 && rows <= (largest >= ((size_t)8 << 20) ? PS_MAX_ROWS : 5) && m.head_dim % 16 == 0 && m.d_model % 4 == 0 && m.d_ffn % 4 == 0 &&
           largest <= ((size_t)16 << 20) && (size_t)rows * std::max(std::max(d, dq), F) * sizeof(float) <= (size_t)PS_ROW_BYTES && (size_t)(m.head_dim + max_ctx) * sizeof(float) <= 40 * 1024;
}

cudaError_t launch_plain_step(const PlainStep& p, cudaStream_t st) {
    if (p.rows < 1 || p.rows > PS_MAX_ROWS || (p.K & 3) || (size_t)p.rows * p.K * sizeof(float) > (size_t)PS_ROW_BYTES) return cudaErrorInvalidValue;
    switch (p.mode) {
        case PS_QKV: return launch_mode<PS_QKV>(p, st);
        case PS_RESIDUAL: return launch_mode<PS_RESIDUAL>(p, st);
        case PS_GU: return launch_mode<PS_GU>(p, st);
        case PS_LM: return launch_mode<PS_LM>(p, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_plain_attention(const float* q, const float* kc, const float* vc, float* out, const int32_t* row_slot, const int32_t* row_pos, int n_rows,
                                   int H, int Hkv, int hd, int max_ctx, cudaStream_t st) {
    return launch_pdl(k_plain_attention, dim3(n_rows, H), dim3(256), sizeof(float) * (size_t)(hd + max_ctx), st, 1, q, kc, vc, out, row_slot, row_pos, H, Hkv, hd, max_ctx);
}

}  // namespace sd
