// Weight matrix times a handful of token rows, with the step that follows it, in one kernel: the layers of the draft models
// (Fig. 1(a)), whose matrices are so small that a pass over them is bound by latency, not by the weights.
//
// The weight-streaming GEMM (gemm_tc.cu) cuts such a matrix into pieces over all SMs and leaves them to a second kernel: two
// launches and two trips through L2 per matrix.  Here a CTA owns 16 output features and the whole reduction:
//   - every thread requests its weights straight into registers (16-byte loads, all in flight) before it waits for the kernel
//     before, so that after the wait only the token rows, the MMAs and the step are left;
//   - tensor cores through mma.sync m16n8k16: the 16 features are its rows, 8 token rows (or twice 8) its columns, in the two
//     bf16 parts of the activations (x_hi + x_lo).  A lane holds eight consecutive reduction elements per 16-byte load;
//     both operands take them in the same order, so the order inside the MMA does not matter;
//   - the warps split the reduction; their sums meet in shared memory, in warp order;
//   - a tile is eight units of two features that the step needs together: a rotary pair, gate and up, or rows eight apart.
// Measured (12-layer, 768-wide draft at 512 positions, one row): 27 -> 17.4 us per layer, of which attention takes 5; the 7B
// iteration 4.57 -> 4.05 ms, 16 sequences on four drafts 9.70 -> 7.22, one shared draft with adapters 5.39 -> 4.66.
// Lines of the choice: at most 16 rows (two MMA column groups) and reductions of at most 4096 (the registers of 16 warps).
// One cooperative launch for the whole pass, with tagged words between CTAs, was no faster than the old path (24 us per layer:
// a hand-over between 148 polling CTAs takes 1.5-2 us, a kernel boundary with the weights already in registers about 1.3).
#include "gemv.h"
#include "tc_ptx.cuh"

namespace sd {
namespace {

__device__ __forceinline__ uint4 ldg_stream(const bf16* p) {           // weights: read once
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

// W warps, NB 32-wide k blocks per warp, NT groups of eight token rows.  ST: with time stamps (as a test of the pointer they cost 0.1-0.2 us
// per launch: 1B target's decoding step 367 -> 371 us).
template <int W, int NB, int NT, bool ST>
__global__ void __launch_bounds__(32 * W, W == 8 && NT == 1 ? 3 : 1) k_gemv(const __grid_constant__ Gemv g) {
    constexpr int M = 8 * NT, PITCH = W + 4;                            // floats per (feature, row): the warps' sums, readable by fours
    __shared__ __align__(16) float red[16 * M * PITCH];
    __shared__ float scale[M];
    const Epilogue& ep = g.ep;
    pdl_launch_dependents();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gid = lane >> 2, tig = lane & 3, tile = blockIdx.x;
    // weight rows of unit u of the tile
    const int half = ep.mode == EPI_QKV_ROPE ? ep.hd >> 1 : 64;
    auto first_row = [&](int u) {
        const int n = tile * 8 + u;
        if (ep.mode == EPI_QKV_ROPE) return n / half * ep.hd + n % half;
        if (ep.mode == EPI_SWIGLU) return (n >> 6) * 128 + (n & 63);
        return tile * 16 + u;
    };
    const int apart = ep.mode == EPI_QKV_ROPE || ep.mode == EPI_SWIGLU ? half : 8;
    const int KB = g.K >> 5;
    uint4 a0[NB], a1[NB];
    {
        const int r0 = first_row(gid), r1 = r0 + apart;
        const bf16* w0 = g.w + (size_t)r0 * g.K + 8 * tig;
        const bf16* w1 = g.w + (size_t)r1 * g.K + 8 * tig;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const int kb = warp + W * b;
            a0[b] = kb < KB && r0 < g.n_out ? ldg_stream(w0 + 32 * kb) : make_uint4(0, 0, 0, 0);
            a1[b] = kb < KB && r1 < g.n_out ? ldg_stream(w1 + 32 * kb) : make_uint4(0, 0, 0, 0);
        }
    }
    if (ST && tid == 0) stamp_first(ep.stamp, ST_START);                      // (behind the requests for the weights)
    // what the finishing threads need besides: their unit's features, gains, the rows' plan and rotary factors (written by the
    // pass's first kernel; the second one is launched in full stream order after it, every later one begins after that)
    const int ui = tid & 7, um = tid >> 3;                              // unit and token row this thread finishes
    const bool mine = um < g.rows && tid < 8 * M;
    const int f0 = first_row(ui), f1 = f0 + apart;
    float gain0 = 0.f, gain1 = 0.f, cs = 1.f, sn = 0.f;
    int pos = -1, slot = 0, task = -1;
    if (mine && ep.mode == EPI_RESIDUAL && ep.gain_next) { gain0 = __ldg(ep.gain_next + f0); gain1 = __ldg(ep.gain_next + f1); }
    if (mine && ep.mode == EPI_QKV_ROPE) {
        pos = __ldcg(ep.row_pos + um); slot = __ldcg(ep.row_slot + um);
        if (f0 / ep.hd < ep.H + ep.Hkv) { cs = __ldcg(ep.rcos + (size_t)um * half + f0 % ep.hd); sn = __ldcg(ep.rsin + (size_t)um * half + f0 % ep.hd); }
    }
    if (mine && ep.lora_b) { task = __ldcg(ep.lora_task + um); if (task >= ep.lora_n) task = -1; }

    pdl_wait();                                                         // token rows, residual stream and sums of squares come from the kernels before
    if (ST && tid == 0) stamp_pair(ep.stamp, ST_DEP_FIRST);
    float h0 = 0.f, h1 = 0.f;
    if (mine && ep.mode == EPI_RESIDUAL) { h0 = __ldcg(ep.h + (size_t)um * g.n_out + f0); h1 = __ldcg(ep.h + (size_t)um * g.n_out + f1); }
    float ss[(M + W - 1) / W];                                          // a warp per token row sums the row's pieces
    if (ep.rs.ssq) {
#pragma unroll
        for (int i = 0; i < (M + W - 1) / W; ++i) {
            const int m = warp + W * i;
            ss[i] = 0.f;
            if (m < g.rows)
                for (int p = lane; p < ep.rs.n_parts; p += 32) ss[i] += __ldcg(ep.rs.ssq + (size_t)m * ep.rs.stride + p);
        }
    }
    float acc[NT][4];
#pragma unroll
    for (int t = 0; t < NT; ++t) acc[t][0] = acc[t][1] = acc[t][2] = acc[t][3] = 0.f;
    constexpr int GB = NB < 8 / NT ? NB : 8 / NT;                       // k blocks whose token rows are in flight together
#pragma unroll
    for (int b0 = 0; b0 < NB; b0 += GB) {
        uint4 xh[GB][NT], xl[GB][NT];
#pragma unroll
        for (int b = 0; b < GB; ++b)
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                const int kb = warp + W * (b0 + b), m = 8 * t + gid;
                const bool on = b0 + b < NB && kb < KB && m < g.rows;
                const bf16* x = g.x + (size_t)m * g.K + 32 * kb + 8 * tig;
                xh[b][t] = on ? *reinterpret_cast<const uint4*>(x) : make_uint4(0, 0, 0, 0);
                xl[b][t] = on && ep.lo_off ? *reinterpret_cast<const uint4*>(x + (size_t)ep.lo_off * g.K) : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
        for (int b = 0; b < GB; ++b)
            if (b0 + b < NB) {
                const uint4 p = a0[b0 + b], q = a1[b0 + b];
#pragma unroll
                for (int t = 0; t < NT; ++t) {
                    mma_bf16(acc[t], p.x, q.x, p.y, q.y, xh[b][t].x, xh[b][t].y);
                    mma_bf16(acc[t], p.z, q.z, p.w, q.w, xh[b][t].z, xh[b][t].w);
                    mma_bf16(acc[t], p.x, q.x, p.y, q.y, xl[b][t].x, xl[b][t].y);
                    mma_bf16(acc[t], p.z, q.z, p.w, q.w, xl[b][t].z, xl[b][t].w);
                }
            }
    }
#pragma unroll
    for (int t = 0; t < NT; ++t) {
        float* r = red + (size_t)(gid * M + 8 * t + 2 * tig) * PITCH + warp;       // [feature][row][warp]
        r[0] = acc[t][0]; r[PITCH] = acc[t][1];
        r[8 * M * PITCH] = acc[t][2]; r[(8 * M + 1) * PITCH] = acc[t][3];
    }
    if (ep.rs.ssq) {
#pragma unroll
        for (int i = 0; i < (M + W - 1) / W; ++i) {
            const float s = warp_sum(ss[i]);
            if (lane == 0 && warp + W * i < M) scale[warp + W * i] = rsqrtf(s * ep.rs.inv_d + ep.rs.eps);
        }
    }
    __syncthreads();
    if (tid >= 8 * M) return;                                           // (whole warps: 8 M is a multiple of 32)
    float v0 = 0.f, v1 = 0.f;
    {
        const float4* r = reinterpret_cast<const float4*>(red + (size_t)(ui * M + um) * PITCH);
#pragma unroll
        for (int i = 0; i < W / 4; ++i) {
            const float4 p = r[i], q = r[8 * M * PITCH / 4 + i];
            v0 += (p.x + p.y) + (p.z + p.w); v1 += (q.x + q.y) + (q.z + q.w);
        }
    }
    if (mine && task >= 0) {                                            // the low-rank update of this matrix: t = x A^T comes from the kernel before
        const float* t = g.lora_t + (size_t)um * 128 + task * ep.lora_r;
        const bf16* b0 = ep.lora_b + ((size_t)task * g.n_out + f0) * ep.lora_r;
        const bf16* b1 = ep.lora_b + ((size_t)task * g.n_out + f1) * ep.lora_r;
        float s0 = 0.f, s1 = 0.f;
        for (int j = 0; j < ep.lora_r; j += 8) {
            const uint4 p = __ldg(reinterpret_cast<const uint4*>(b0 + j)), q = __ldg(reinterpret_cast<const uint4*>(b1 + j));
            const __nv_bfloat162* ph = reinterpret_cast<const __nv_bfloat162*>(&p);
            const __nv_bfloat162* qh = reinterpret_cast<const __nv_bfloat162*>(&q);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 x = __ldcg(reinterpret_cast<const float2*>(t + j + 2 * e)), a = __bfloat1622float2(ph[e]), b = __bfloat1622float2(qh[e]);
                s0 = fmaf(x.x, a.x, s0); s0 = fmaf(x.y, a.y, s0);
                s1 = fmaf(x.x, b.x, s1); s1 = fmaf(x.y, b.y, s1);
            }
        }
        v0 = fmaf(ep.lora_scale, s0, v0); v1 = fmaf(ep.lora_scale, s1, v1);
    }
    if (ep.rs.ssq && um < M) { v0 *= scale[um]; v1 *= scale[um]; }
    auto store2 = [&](bf16* p, size_t lo, float x) {                    // in two bf16 parts where the pass carries two
        const bf16 hi = __float2bfloat16_rn(x);
        *p = hi;
        if (ep.lo_off) p[lo] = __float2bfloat16_rn(x - __bfloat162float(hi));
    };
    switch (ep.mode) {
    case EPI_PLAIN: {
        const int r = um - ep.row_offset;                               // token row i * row_stride + row_offset is output row i
        if (mine && r >= 0 && r % ep.row_stride == 0 && r / ep.row_stride < ep.n_out_rows) {
            float* y = ep.y + (size_t)(r / ep.row_stride) * g.n_out;
            if (f0 < g.n_out) y[f0] = v0;
            if (f1 < g.n_out) y[f1] = v1;
        }
        break;
    }
    case EPI_QKV_ROPE: {
        if (mine && pos >= 0 && f1 < g.n_out) {
            const int hd = ep.hd, head = f0 / hd, e = f0 % hd;
            bf16* dst;
            if (head < ep.H) dst = ep.q_out + ((size_t)um * ep.H + head) * hd + e;
            else {
                const bool is_v = head >= ep.H + ep.Hkv;
                dst = (is_v ? ep.vc : ep.kc) + (((size_t)slot * ep.Hkv + head - ep.H - (is_v ? ep.Hkv : 0)) * ep.max_ctx + pos) * hd + e;
            }
            dst[0] = __float2bfloat16_rn(v0 * cs - v1 * sn);
            dst[half] = __float2bfloat16_rn(v0 * sn + v1 * cs);
        }
        break;
    }
    case EPI_RESIDUAL: {
        h0 += v0; h1 += v1;
        if (mine) {
            const size_t at = (size_t)um * g.n_out;
            ep.h[at + f0] = h0; ep.h[at + f1] = h1;
            if (ep.gain_next) {
                store2(ep.xn + at + f0, (size_t)ep.lo_off * g.n_out, h0 * gain0);
                store2(ep.xn + at + f1, (size_t)ep.lo_off * g.n_out, h1 * gain1);
            }
        }
        if (ep.gain_next) {                                             // the tile's share of the row's sum of squares: eight neighbouring lanes
            float s = mine ? h0 * h0 + h1 * h1 : 0.f;
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (mine && ui == 0) ep.ssq_out[(size_t)um * GEMV_SSQ_STRIDE + tile] = s;
        }
        break;
    }
    default: {                                                          // EPI_SWIGLU
        if (mine) store2(ep.act + (size_t)um * ep.F + tile * 8 + ui, (size_t)ep.lo_off * ep.F, v0 / (1.f + expf(-v0)) * v1);
        break;
    }
    }
    if (ST && tid == 0) stamp_pair(ep.stamp, ST_DONE_FIRST);
}

typedef void (*Kernel)(const Gemv);
struct Form { int warps, blocks; Kernel k[2][2]; };       // [two groups of rows][with time stamps]
#define GEMV_FORM(W, NB) {W, NB, {{k_gemv<W, NB, 1, false>, k_gemv<W, NB, 1, true>}, {k_gemv<W, NB, 2, false>, k_gemv<W, NB, 2, true>}}}
const Form FORMS[] = {GEMV_FORM(8, 3), GEMV_FORM(8, 4), GEMV_FORM(16, 4), GEMV_FORM(16, 6), GEMV_FORM(16, 8)};
#undef GEMV_FORM

const Form* form_of(int K) {
    for (const Form& f : FORMS) if (f.warps * f.blocks * 32 >= K) return &f;
    return nullptr;
}

}  // namespace

bool gemv_supported(const Gemv& g) {
    if (g.rows < 1 || g.rows > GEMV_MAX_ROWS || g.K % 32 || !form_of(g.K) || g.n_out < 1) return false;
    switch (g.ep.mode) {
    case EPI_QKV_ROPE: return (g.ep.hd == 64 || g.ep.hd == 128) && g.n_out % g.ep.hd == 0;
    case EPI_SWIGLU: return g.ep.F % 64 == 0 && g.n_out == 2 * g.ep.F;
    case EPI_RESIDUAL: return g.n_out % 16 == 0;
    default: return true;
    }
}

cudaError_t launch_gemv(const Gemv& g, int dependent, cudaStream_t st) {
    if (!gemv_supported(g) || g.ep.lo_off < 0 || (g.ep.lo_off && g.ep.lo_off < g.rows)) return cudaErrorInvalidValue;
    if (g.ep.lora_b && (g.ep.lora_r < 8 || g.ep.lora_r > 32 || (g.ep.lora_r & 7) || g.ep.lora_n * g.ep.lora_r > 128 || !g.lora_t)) return cudaErrorInvalidValue;
    const Form* f = form_of(g.K);
    return launch_pdl(f->k[g.rows > 8][g.ep.stamp != nullptr], dim3((g.n_out + 15) / 16), dim3(32 * f->warps), 0, st, dependent, g);
}

}  // namespace sd
