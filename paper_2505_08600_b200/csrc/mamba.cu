// The Mamba-based prompt classifier (Section 2.4, Section 3.3.3): embedding -> one selective state-space layer ->
// average pooling over the prompt -> fully connected layer -> argmax.  Everything is fp32.
//
// The layer's recurrence h_t = a_t * h_{t-1} + b_t is linear in h, so a prompt is cut into chunks of MB_CHUNK tokens that are
// scanned side by side, once, from a zero state: with P_t the product of a chunk's decays up to token t and s the state the
// chunk starts from, h_t = h_t(zero) + P_t s, so what a chunk adds to the pooled sum of g_t = (C_t h_t + D v_t) silu(z_t) is
//   sum_t (C_t h_t(zero) + D v_t) silu(z_t)  +  s . sum_t silu(z_t) C_t P_t,
// both sums of the one scan.  The states s follow from the chunks' end states and decays in a short serial pass per prompt.
// The pooled vector is the mean over tokens of W_out g_t, which is W_out applied to the mean of g_t: the kernels sum
// g_t per channel (chunks in order) and apply W_out and the classification layer once per prompt.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "../../include/sd.h"
#include "f32x2.cuh"

namespace sd {
namespace {

constexpr int MB_CHUNK = 64;         // tokens per chunk of the scan
constexpr int MB_MAX_N = 16;         // state size kept in registers
constexpr int MB_MAX_CONV = 8;
constexpr int MB_MAX_DI = 1024, MB_MAX_D = 512, MB_MAX_X = 256, MB_MAX_K = 64;      // largest d_inner, d_model, r + B + C, classes

struct MambaDims { int V, D, Di, N, R, Kc, K; };

struct ChunkRec { int32_t prompt, tok0, n_tok, pos0; };      // tok0: index into the flattened token list; pos0: position of the chunk's first token in its prompt

__device__ __forceinline__ float silu_f(float x) { return x / (1.f + expf(-x)); }
__device__ __forceinline__ float softplus_f(float x) { return x > 20.f ? x : log1pf(expf(x)); }

// What the host knows of up to NP prompts, handed over as a kernel parameter: no copy that the call would have to wait for.
template <int NP> struct PromptTable { int64_t start[NP]; int32_t len[NP], tok0[NP], chunk0[NP]; };
constexpr int MT_FEW = 32, MT_MANY = 1024, MT_ROWS = 32;      // (parameters of 640 bytes and of 20 KB; CTAs that share a prompt's chunks)

// The chunks of every prompt, and where every flattened token's projected row is: its own, or its token's when the whole vocabulary was projected.
template <int NP>
__global__ void k_mamba_tables(const __grid_constant__ PromptTable<NP> t, int first, int n_all, const int32_t* __restrict__ tokens, int V, int by_token,
                               ChunkRec* __restrict__ chunks, int32_t* __restrict__ prompt_chunk0, int32_t* __restrict__ lens,
                               int32_t* __restrict__ tok_id, int32_t* __restrict__ tok_row) {
    const int p = blockIdx.x, len = t.len[p], tok0 = t.tok0[p], chunk0 = t.chunk0[p], n_chunks = (len + MB_CHUNK - 1) / MB_CHUNK;
    const int32_t* src = tokens + t.start[p];
    if (blockIdx.y == 0 && threadIdx.x == 0) {
        prompt_chunk0[first + p] = chunk0;
        if (first + p + 1 == n_all) prompt_chunk0[n_all] = chunk0 + n_chunks;
        lens[first + p] = len;
    }
    for (int k = blockIdx.y; k < n_chunks; k += gridDim.y) {
        const int pos0 = k * MB_CHUNK, n = min(MB_CHUNK, len - pos0);
        if (threadIdx.x == 0) chunks[chunk0 + k] = ChunkRec{first + p, tok0 + pos0, n, pos0};
        for (int i = pos0 + threadIdx.x; i < pos0 + n; i += blockDim.x) {
            const int tok = min(max(src[i], 0), V - 1);
            tok_id[tok0 + i] = tok;
            tok_row[tok0 + i] = by_token ? tok : tok0 + i;
        }
    }
}

// u, gate = split(W_in E[row]), the gate behind its SiLU, for every row: token by token, or, when the prompts hold more tokens than the vocabulary has, once per
// token of the vocabulary (the projection depends on nothing else).  Bound: fp32 multiply-adds (21,128 rows: 76 us; 109,096 token
// by token, a thread per feature, 757).  64 x 128 tiles of 256 threads, 4 x 8 sums each in register pairs, 16-deep slices of both operands
// through two buffers (128 x 128 tiles of 8 x 8 leave a third wave of 664 CTAs that is a quarter full: 80 us with the gates, 76 so; one prompt of 300
// tokens, whole call: 94 and 89).
constexpr int MI_TILE = 128, MI_ROWS = 64, MI_K = 16, MI_PITCH = MI_TILE + 4, MI_RPITCH = MI_ROWS + 4;
__global__ void __launch_bounds__(256, 3)
k_mamba_in(MambaDims m, const int32_t* __restrict__ tok_id /*nullptr: row = token*/, int rows, const float* __restrict__ embed,
           const float* __restrict__ w_in, float* __restrict__ u, float* __restrict__ gate) {
    __shared__ __align__(16) float as[2][MI_K][MI_RPITCH], bs[2][MI_K][MI_PITCH];
    const int tid = threadIdx.x, r0 = blockIdx.x * MI_ROWS, j0 = blockIdx.y * MI_TILE;
    const int lr = tid >> 2, lk = (tid & 3) * 4;                        // this thread loads row lr, features lr and lr + 64, columns lk ... lk + 3
    const float* b_src[2];
    const float* a_src = r0 + lr < rows ? embed + (size_t)(tok_id ? tok_id[r0 + lr] : r0 + lr) * m.D : nullptr;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int j = j0 + lr + 64 * i;
        b_src[i] = j < 2 * m.Di ? w_in + (size_t)j * m.D : nullptr;
    }
    const bool vec = (m.D & 3) == 0 && (((uintptr_t)embed | (uintptr_t)w_in) & 15) == 0;
    const bool vec_out = (m.Di & 3) == 0 && (((uintptr_t)u | (uintptr_t)gate) & 15) == 0;      // (the workspace may begin at any multiple of 8)
    auto get = [&](const float* src, int k) {
        if (!src) return make_float4(0.f, 0.f, 0.f, 0.f);
        if (vec) return k < m.D ? __ldg(reinterpret_cast<const float4*>(src + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
        return make_float4(k < m.D ? src[k] : 0.f, k + 1 < m.D ? src[k + 1] : 0.f, k + 2 < m.D ? src[k + 2] : 0.f, k + 3 < m.D ? src[k + 3] : 0.f);
    };
    float4 a_next, b_next[2];
    auto fetch = [&](int k0) {
        a_next = get(a_src, k0 + lk);
#pragma unroll
        for (int i = 0; i < 2; ++i) b_next[i] = get(b_src[i], k0 + lk);
    };
    auto stash = [&](int buf) {
        float* a = &as[buf][lk][lr];
        a[0] = a_next.x; a[MI_RPITCH] = a_next.y; a[2 * MI_RPITCH] = a_next.z; a[3 * MI_RPITCH] = a_next.w;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            float* b = &bs[buf][lk][lr + 64 * i];
            b[0] = b_next[i].x; b[MI_PITCH] = b_next[i].y; b[2 * MI_PITCH] = b_next[i].z; b[3 * MI_PITCH] = b_next[i].w;
        }
    };
    const int tx = tid & 15, ty = tid >> 4;                             // rows 4 ty ...; features 4 tx ..., 64 + 4 tx ...
    f32x2 acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
    fetch(0);
    stash(0);
    __syncthreads();
    for (int k0 = 0, buf = 0; k0 < m.D; k0 += MI_K, buf ^= 1) {
        if (k0 + MI_K < m.D) fetch(k0 + MI_K);
#pragma unroll
        for (int k = 0; k < MI_K; ++k) {
            float av[4];
            *reinterpret_cast<float4*>(av) = *reinterpret_cast<const float4*>(&as[buf][k][4 * ty]);
            const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(&bs[buf][k][4 * tx]), b1 = *reinterpret_cast<const ulonglong2*>(&bs[buf][k][64 + 4 * tx]);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const f32x2 a2 = f2_pack(av[i], av[i]);
                acc[i][0] = f2_fma(a2, b0.x, acc[i][0]); acc[i][1] = f2_fma(a2, b0.y, acc[i][1]);
                acc[i][2] = f2_fma(a2, b1.x, acc[i][2]); acc[i][3] = f2_fma(a2, b1.y, acc[i][3]);
            }
        }
        if (k0 + MI_K < m.D) { stash(buf ^ 1); __syncthreads(); }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = r0 + 4 * ty + i;
        if (r >= rows) continue;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = j0 + 64 * h + 4 * tx;
            const float2 p = f2_unpack(acc[i][2 * h]), q = f2_unpack(acc[i][2 * h + 1]);
            float v[4] = {p.x, p.y, q.x, q.y};
#pragma unroll
            for (int e = 0; e < 4; ++e) if (j + e >= m.Di) v[e] = silu_f(v[e]);
            if (vec_out) {                                              // (a group of four lies in one of the halves)
                if (j < 2 * m.Di) *reinterpret_cast<float4*>((j < m.Di ? u + (size_t)r * m.Di + j : gate + (size_t)r * m.Di + j - m.Di)) = make_float4(v[0], v[1], v[2], v[3]);
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (j + e < 2 * m.Di) (j + e < m.Di ? u[(size_t)r * m.Di + j + e] : gate[(size_t)r * m.Di + j + e - m.Di]) = v[e];
            }
        }
    }
}

// Everything of one chunk between the input projection and the pooled sum.  Bound: issue slots (exponentials, d_state of them per token
// and channel, and the multiply-adds around them; 57 % of the slots are taken, at sixteen warps of 128 registers per SM).  A chunk is
// walked MC_TILE tokens at a time, a thread per channel but for the projections:
//   1. convolution + SiLU into shared memory;
//   2. the projections (r, B, C): a thread takes four tokens, three outputs and half of the channels, twelve sums per seven 16-byte reads;
//   3. step sizes into shared memory (no token's waits for the one before: in the scan each would);
//   4. the scan goes on over these tokens, its state in registers: recurrence from a zero state, and the chunk's sum.  Only chunks that
//      are not their prompt's first keep the products of decays and the sum they are weighted with (see the top of the file): three of
//      seven packed operations per pair of states.
// 400 prompts of 109,096 tokens: 694 -> 391 us (some 290 instructions per token and 32 channels, 356 with the convolution in 2 and again in 4, the
// step size and the SiLU of the gate in the scan, half of the states' results stored four bytes at a time); whole call 815 -> 512,
// one prompt of 8 / 64 / 300 tokens 77 / 128 / 141 -> 54 / 81 / 91.  Two threads per channel with half of its states each, 32 warps of 64
// registers, spill: 720...795.  Rank 8 as a compiled form: 539 -> 512, one prompt of 300 96 -> 91.
//   More than MC_CHANNELS channels: a cluster of up to four CTAs per chunk with as many channels each.  A CTA projects its own channels;
//   the parts of r, B, C meet through distributed shared memory (each CTA adds a share of them, parts in the CTAs' order), tile by tile, before: once
//   per chunk.  1,024 channels: one prompt of 300 tokens 459 -> 418 us, 400 prompts 14.9 -> 14.5 ms, but one of 4,000 858 -> 884; 512: 434 -> 387, 7.2 -> 6.9 ms.
constexpr int MC_TILE = 32, MC_CHANNELS = 256, MC_THREADS = MC_CHANNELS, MC_STAGED = 40 * 1024;      // W_x is staged up to this size, with which two CTAs fit an SM
// (256 channels of rank 16, 48 KB: staged 400 prompts take 1,171 us, read from L2 1,018; one prompt of 300 tokens 133 and 137)
constexpr int MC_GROUP = 16 /*tokens of the convolution on their way at a time*/, MC_PITCH = MC_CHANNELS + 4, MC_AHEAD = 2 /*gates on their way during the scan*/;
constexpr int MC_PARTS = MC_THREADS / 128, MC_OUT = 48;              // parts the channels of a projection are cut into; outputs of one round of it
constexpr int MC_PART = MC_TILE * (MC_OUT + 1);          // floats of one part's sums, in the place of the step sizes
static_assert(MC_PARTS * MC_PART <= MC_TILE * MC_PITCH, "the parts' sums fit where the step sizes will be");
// Most dynamic shared memory a launch takes: B, C and r of a tile, its v and step sizes, and the staged W_x at their largest.
constexpr int MC_MAX_SMEM = (MC_TILE * MB_MAX_X + 2 * MC_TILE * MC_PITCH) * 4 + MC_STAGED;
constexpr int MH_THREADS = 512;
constexpr int MH_MAX_SMEM = (MB_MAX_DI * MB_MAX_N + MB_MAX_DI + MB_MAX_D + MB_MAX_K) * 4;

template <int NS /*states: 16, or any up to MB_MAX_N as 0*/, int KC /*taps: 4, or any up to four as -4, or up to MB_MAX_CONV as 0*/, int RS /*rank of the step size: 8, or any as 0*/,
          bool CL /*several CTAs per chunk*/, bool CARRY /*some prompt has more than one chunk*/>
__global__ void __launch_bounds__(MC_THREADS, 2)
k_mamba_chunk(MambaDims m, const ChunkRec* __restrict__ chunks, const int32_t* __restrict__ tok_row, const float* __restrict__ u, const float* __restrict__ gate,
              const float* __restrict__ w_conv, const float* __restrict__ b_conv, const float* __restrict__ w_x, const float* __restrict__ w_dt,
              const float* __restrict__ b_dt, const float* __restrict__ a_log, const float* __restrict__ d_skip,
              float* __restrict__ end_state, float* __restrict__ decay, float* __restrict__ carry_gain /*all [chunk][N][Di]*/, double* __restrict__ chunk_sum /*[chunk][Di]*/, int w_staged, int n_cta, int per_cta) {
    extern __shared__ __align__(16) float sm[];
    const int per = CL ? per_cta : (m.Di + 3) & ~3;        // channels of a CTA, padded to a multiple of 4
    const int N = NS ? NS : m.N, R = RS ? RS : m.R, n_x = R + 2 * N, xp = (n_x + 3) & ~3;
    float* xd_s = sm;                                      // [MC_TILE][xp]: B, C, r of every token
    float* v_s = sm + MC_TILE * xp;                        // [MC_TILE][MC_PITCH]
    float* dt_s = v_s + MC_TILE * MC_PITCH;                // [MC_TILE][MC_PITCH]; before that the parts' sums
    float* wx_s = dt_s + MC_TILE * MC_PITCH;               // this CTA's columns of W_x, [n_x][n_c], if they were given room
    // where the rows of the taps in front of a tile's tokens (-1: before the prompt) and of its tokens begin; this tile's and the next one's
    __shared__ long long row_s[2][MB_MAX_CONV + MC_TILE + MC_AHEAD];
    const int tid = threadIdx.x;
    const int chunk = CL ? blockIdx.x / n_cta : blockIdx.x, c_lo = CL ? (int)(blockIdx.x % n_cta) * per : 0, n_c = CL ? min(m.Di - c_lo, per) : m.Di;
    const ChunkRec ch = chunks[chunk];
    constexpr int KM = KC > 0 ? KC : KC < 0 ? -KC : MB_MAX_CONV;
    const int Kc = KC > 0 ? KC : m.Kc, back = Kc - 1;
    auto load_rows = [&](int t0) {                         // (past the chunk's end: any row)
        if (tid < back + MC_TILE + MC_AHEAD) {
            const int t = min(t0 + tid - back, ch.n_tok - 1);
            row_s[(t0 / MC_TILE) & 1][tid] = ch.pos0 + t >= 0 ? (long long)tok_row[ch.tok0 + t] * m.Di : -1;
        }
    };
    load_rows(0);
    if (w_staged) for (int i = tid; i < n_x * n_c; i += MC_THREADS) wx_s[i] = __ldg(CL ? w_x + (size_t)(i / n_c) * m.Di + c_lo + i % n_c : w_x + i);
    const bool vec = (m.Di & 3) == 0 && (w_staged || ((uintptr_t)w_x & 15) == 0);      // (then n_c is a multiple of 4 as well)

    const bool on = tid < n_c;                             // this thread's channel
    const int c = c_lo + min(tid, n_c - 1);
    f32x2 A[MB_MAX_N / 2], h[MB_MAX_N / 2], P[CARRY ? MB_MAX_N / 2 : 1], G[CARRY ? MB_MAX_N / 2 : 1];
#pragma unroll
    for (int i = 0; i < MB_MAX_N / 2; ++i) {               // (decays as powers of two; an unused state: decay one, input zero)
        const int n = 2 * i;
        const float a0 = n < N ? -expf(__ldg(a_log + (size_t)c * m.N + n)) * 1.4426950408889634f : 0.f;
        const float a1 = n + 1 < N ? -expf(__ldg(a_log + (size_t)c * m.N + n + 1)) * 1.4426950408889634f : 0.f;
        A[i] = f2_pack(a0, a1);
        h[i] = 0ull;
        if (CARRY) { P[CARRY ? i : 0] = f2_pack(1.f, 1.f); G[CARRY ? i : 0] = 0ull; }
    }
    const float* uc = u + c; const float* gc = gate + c;
    double sum = 0.0;                                      // (in double here and over the chunks: the sum's rounding would be the largest of all)
    const bool carried = CARRY && ch.pos0 > 0;
    __syncthreads();

    for (int t0 = 0; t0 < ch.n_tok; t0 += MC_TILE) {
        const int nt = min(MC_TILE, ch.n_tok - t0), cur = (t0 / MC_TILE) & 1;
        // (a channel's few weights are read again for every tile: in registers they would be in the way of the other steps)
        {
            float w[KM];
            const float b = __ldg(b_conv + c);
#pragma unroll
            for (int j = 0; j < KM; ++j) w[j] = j < Kc ? __ldg(w_conv + (size_t)c * Kc + j) : 0.f;
#pragma unroll 1
            for (int tb = 0; tb < nt; tb += MC_GROUP) {
                float nu[KM - 1 + MC_GROUP];               // the tokens under the taps (in the order of the sum)
#pragma unroll
                for (int i = 0; i < KM - 1 + MC_GROUP; ++i) {      // (past the chunk's end: any token's, of which nothing is used)
                    const long long at = KC > 0 || i < back + MC_GROUP ? row_s[cur][tb + i] : -1;
                    nu[i] = i >= KM - 1 && KC > 0 ? __ldg(uc + at) : at >= 0 ? __ldg(uc + at) : 0.f;
                }
#pragma unroll
                for (int t = 0; t < MC_GROUP; ++t) {
                    float acc = b;
#pragma unroll
                    for (int j = 0; j < KM; ++j) if (j < Kc) acc = fmaf(w[j], nu[t + j], acc);
                    v_s[(tb + t) * MC_PITCH + tid] = silu_f(acc);
                }
            }
        }
        __syncthreads();
        if (t0 + MC_TILE < ch.n_tok) load_rows(t0 + MC_TILE);
        const int tg = tid & 7, og = (tid >> 3) & 15, pt = tid >> 7;                       // tokens tg, tg + 8 ...; outputs og, og + ns, og + 2 ns
        const int kq = ((n_c + 4 * MC_PARTS - 1) / (4 * MC_PARTS)) * 4, k0 = min(n_c, pt * kq), k1 = min(n_c, k0 + kq);
        const float* v0 = v_s + tg * MC_PITCH;
        for (int o0 = 0; o0 < n_x; o0 += MC_OUT) {
            const int n_o = min(MC_OUT, n_x - o0), ns = (n_o + 2) / 3;
            float s[3][4];
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int t = 0; t < 4; ++t) s[i][t] = 0.f;
            auto project = [&](const float* wx, int w_ld) {      // (called with shared and with global memory: two loops, each of which knows which it reads)
                const float* w0 = wx + (size_t)min(o0 + og, n_x - 1) * w_ld;
                const float* w1 = wx + (size_t)min(o0 + og + ns, n_x - 1) * w_ld;
                const float* w2 = wx + (size_t)min(o0 + og + 2 * ns, n_x - 1) * w_ld;
                if (vec) {
#pragma unroll 2
                    for (int k = k0; k < k1; k += 4) {
                        float4 a[4];
#pragma unroll
                        for (int t = 0; t < 4; ++t) a[t] = *reinterpret_cast<const float4*>(v0 + 8 * t * MC_PITCH + k);
#pragma unroll
                        for (int i = 0; i < 3; ++i) {
                            const float4 p = *reinterpret_cast<const float4*>((i == 0 ? w0 : i == 1 ? w1 : w2) + k);
#pragma unroll
                            for (int t = 0; t < 4; ++t) {
                                s[i][t] = fmaf(p.x, a[t].x, s[i][t]); s[i][t] = fmaf(p.y, a[t].y, s[i][t]);
                                s[i][t] = fmaf(p.z, a[t].z, s[i][t]); s[i][t] = fmaf(p.w, a[t].w, s[i][t]);
                            }
                        }
                    }
                } else {
                    for (int k = k0; k < k1; ++k)
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            const float a = v0[8 * t * MC_PITCH + k];
                            s[0][t] = fmaf(w0[k], a, s[0][t]); s[1][t] = fmaf(w1[k], a, s[1][t]); s[2][t] = fmaf(w2[k], a, s[2][t]);
                        }
                }
            };
            if (og < ns) {
                if (w_staged) project(wx_s, CL ? n_c : m.Di); else project(w_x + c_lo, m.Di);
                float* part = dt_s + pt * MC_PART + tg * (MC_OUT + 1) + og;
#pragma unroll
                for (int i = 0; i < 3; ++i)
                    if (og + i * ns < n_o)
#pragma unroll
                        for (int t = 0; t < 4; ++t) part[8 * t * (MC_OUT + 1) + i * ns] = s[i][t];
            }
            __syncthreads();
            // kept as [B | C | r], so that a token's B and C can be read by fours; eight threads per token
            for (int j = tid & 7; j < n_o; j += 8) {
                const int t = tid >> 3, o = o0 + j;
                const float* q = dt_s + t * (MC_OUT + 1) + j;
                xd_s[t * xp + (o < R ? 2 * N + o : o - R)] = q[0] + q[MC_PART];
            }
            __syncthreads();
        }
        if (CL) {                                          // the other CTAs' channels: every value is added by one CTA, which hands the sum to all
            namespace cg = cooperative_groups;
            cg::cluster_group cluster = cg::this_cluster();
            cluster.sync();
            const int n = MC_TILE * xp, share = (n + n_cta - 1) / n_cta, i0 = (int)(blockIdx.x % n_cta) * share;
            for (int i = i0 + tid; i < min(n, i0 + share); i += MC_THREADS) {
                float v[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) v[r] = r < n_cta ? cluster.map_shared_rank(xd_s, r)[i] : 0.f;
                const float all = ((v[0] + v[1]) + v[2]) + v[3];
#pragma unroll
                for (int r = 0; r < 4; ++r) if (r < n_cta) cluster.map_shared_rank(xd_s, r)[i] = all;
            }
            cluster.sync();                                // (no CTA touches another's shared memory from here to the next tile's first cluster barrier)
        }
        float ng[MC_AHEAD];
#pragma unroll
        for (int i = 0; i < MC_AHEAD; ++i) ng[i] = __ldg(gc + row_s[cur][back + i]);
        {
            const float bdt = __ldg(b_dt + c);
            float wd[RS ? RS : 8];                         // the first eight columns of the channel's row of W_dt (the rest, if any, is read as needed)
#pragma unroll
            for (int r = 0; r < 8; ++r) wd[r] = r < R ? __ldg(w_dt + (size_t)c * m.R + r) : 0.f;
#pragma unroll 4
            for (int t = 0; t < nt; ++t) {
                const float* xr = xd_s + t * xp + 2 * N;
                float dt = bdt;
                if (NS && RS) {                            // (2 N and the pitch are multiples of four)
                    const float4 a = *reinterpret_cast<const float4*>(xr), b = *reinterpret_cast<const float4*>(xr + 4);
                    dt = fmaf(wd[0], a.x, dt); dt = fmaf(wd[1], a.y, dt); dt = fmaf(wd[2], a.z, dt); dt = fmaf(wd[3], a.w, dt);
                    dt = fmaf(wd[4], b.x, dt); dt = fmaf(wd[5], b.y, dt); dt = fmaf(wd[6], b.z, dt); dt = fmaf(wd[7], b.w, dt);
                } else {
#pragma unroll
                    for (int r = 0; r < 8; ++r) if (r < R) dt = fmaf(wd[r], xr[r], dt);
                    for (int r = 8; r < R; ++r) dt = fmaf(__ldg(w_dt + (size_t)c * m.R + r), xr[r], dt);
                }
                dt_s[t * MC_PITCH + tid] = softplus_f(dt);
            }
        }
        __syncthreads();
        auto scan = [&](auto with_carry) {
            constexpr bool WITH = decltype(with_carry)::value;
            const float dsk = __ldg(d_skip + c);
            for (int t1 = 0; t1 < nt; t1 += MC_AHEAD) {
                float now[MC_AHEAD];
#pragma unroll
                for (int i = 0; i < MC_AHEAD; ++i) {       // the next tokens' gates are on their way during these
                    now[i] = ng[i];
                    ng[i] = __ldg(gc + row_s[cur][back + t1 + MC_AHEAD + i]);
                }
#pragma unroll
                for (int i = 0; i < MC_AHEAD; ++i) {
                    if (t1 + i >= nt) break;               // uniform
                    const float* xb = xd_s + (t1 + i) * xp;
                    const float v = v_s[(t1 + i) * MC_PITCH + tid], dt = dt_s[(t1 + i) * MC_PITCH + tid], g = now[i], dx = dt * v;
                    const f32x2 dt2 = f2_pack(dt, dt), dx2 = f2_pack(dx, dx), g2 = f2_pack(g, g);
                    f32x2 y2 = 0ull;
#pragma unroll
                    for (int k = 0; k < MB_MAX_N / 2; k += 2) {
                        if (2 * k >= N) break;
                        f32x2 B[2], C[2];
                        if (NS) {
                            const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(xb + 2 * k), cc = *reinterpret_cast<const ulonglong2*>(xb + NS + 2 * k);
                            B[0] = b.x; B[1] = b.y; C[0] = cc.x; C[1] = cc.y;
                        } else {
#pragma unroll
                            for (int j = 0; j < 2; ++j) {
                                const int n = 2 * (k + j), e = n;
                                B[j] = f2_pack(n < N ? xb[e] : 0.f, n + 1 < N ? xb[e + 1] : 0.f);
                                C[j] = f2_pack(n < N ? xb[m.N + e] : 0.f, n + 1 < N ? xb[m.N + e + 1] : 0.f);
                            }
                        }
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            const float2 e = f2_unpack(f2_mul(dt2, A[k + j]));
                            const f32x2 a = f2_pack(exp2_ftz(e.x), exp2_ftz(e.y));
                            h[k + j] = f2_fma(a, h[k + j], f2_mul(dx2, B[j]));
                            y2 = f2_fma(h[k + j], C[j], y2);
                            if (WITH) {
                                P[CARRY ? k + j : 0] = f2_mul(P[CARRY ? k + j : 0], a);
                                G[CARRY ? k + j : 0] = f2_fma(f2_mul(g2, C[j]), P[CARRY ? k + j : 0], G[CARRY ? k + j : 0]);
                            }
                        }
                    }
                    const float2 y = f2_unpack(y2);
                    sum += (double)(fmaf(dsk, v, y.x + y.y) * g);
                }
            }
        };
        if (on) { if (carried) scan(std::integral_constant<bool, CARRY>()); else scan(std::false_type()); }
        __syncthreads();                                   // the tile's v, step sizes, B, C, r have been read, the next one's rows are there
    }
    if (!on) return;
    chunk_sum[(size_t)chunk * m.Di + c] = sum;
    if (!CARRY) return;
#pragma unroll
    for (int k = 0; k < MB_MAX_N / 2; ++k) {
        const float2 hv = f2_unpack(h[k]), pv = f2_unpack(P[CARRY ? k : 0]), gv = f2_unpack(G[CARRY ? k : 0]);
        const int n = 2 * k;
        const size_t at = ((size_t)chunk * m.N + n) * m.Di + c;      // (of a prompt's first chunk only the end state is read)
        if (n < N) { end_state[at] = hv.x; decay[at] = pv.x; carry_gain[at] = gv.x; }
        if (n + 1 < N) { end_state[at + m.Di] = hv.y; decay[at + m.Di] = pv.y; carry_gain[at + m.Di] = gv.y; }
    }
}

// The pooled sums of long prompts: what the chunks' starting states add and the chunks' own sums, a thread per (channel, state) and a CTA
// per eight channels instead of the head's one CTA per prompt, with the coefficients of eight chunks on their way at a time.  Bound: latency
// of the chain over chunks.  One prompt of 1,000 / 4,000 / 30,000 / 200,000 tokens, whole call: 90 / 102 / 281 / 1,214 us,
// in the head 100 / 160 / 806 / 8,003.  From eight chunks on a queue of shorter prompts is the slower for the launch (100 / 400 prompts of
// 32...512 tokens: 244 / 521 against 239 / 512).
constexpr int MB_LONG = 16;                              // chunks from which on a prompt is long
constexpr int CARRY_CH = 8, CARRY_BATCH = 8;
__global__ void __launch_bounds__(CARRY_CH * MB_MAX_N)
k_mamba_carry(MambaDims m, const int32_t* __restrict__ prompt_chunk0, const double* __restrict__ chunk_sum, const float* __restrict__ end_state,
              const float* __restrict__ decay, const float* __restrict__ carry_gain, double* __restrict__ g_sum /*[prompt][Di]*/) {
    const int c0 = prompt_chunk0[blockIdx.x], c1 = prompt_chunk0[blockIdx.x + 1];
    if (c1 - c0 < MB_LONG) return;
    const int c = blockIdx.y * CARRY_CH + threadIdx.x % CARRY_CH, n = threadIdx.x / CARRY_CH;
    const bool on = c < m.Di && n < m.N;
    const size_t per = (size_t)m.Di * m.N, i = (size_t)min(n, m.N - 1) * m.Di + min(c, m.Di - 1);
    float s = on ? __ldg(end_state + c0 * per + i) : 0.f, add = 0.f;
    for (int ch = c0 + 1; ch < c1; ch += CARRY_BATCH) {
        float e[CARRY_BATCH], p[CARRY_BATCH], g[CARRY_BATCH];
#pragma unroll
        for (int b = 0; b < CARRY_BATCH; ++b) {
            const bool in = on && ch + b < c1;
            const size_t at = (size_t)(ch + b) * per + i;
            e[b] = in ? __ldg(end_state + at) : 0.f; p[b] = in ? __ldg(decay + at) : 0.f; g[b] = in ? __ldg(carry_gain + at) : 0.f;
        }
#pragma unroll
        for (int b = 0; b < CARRY_BATCH; ++b)
            if (ch + b < c1) { add = fmaf(g[b], s, add); s = fmaf(p[b], s, e[b]); }
    }
    double sum = 0.0;
    if (c < m.Di) {
#pragma unroll 8
        for (int ch = c0 + n; ch < c1; ch += MB_MAX_N) sum += __ldg(chunk_sum + (size_t)ch * m.Di + c);
    }
    sum += on ? (double)add : 0.0;
    __shared__ double part[MB_MAX_N][CARRY_CH];
    part[n][threadIdx.x % CARRY_CH] = sum;
    __syncthreads();
    if (n == 0 && c < m.Di) {
        for (int k = 1; k < MB_MAX_N; ++k) sum += part[k][threadIdx.x];
        g_sum[(size_t)blockIdx.x * m.Di + c] = sum;
    }
}

// Per prompt: the states its chunks start from (serial, a thread per channel and state), mean over tokens of the gated outputs
// (chunks in order), W_out, the classification layer, argmax.
__global__ void k_mamba_head(MambaDims m, const int32_t* __restrict__ prompt_chunk0, const int32_t* __restrict__ lens,
                             const double* __restrict__ chunk_sum, const float* __restrict__ end_state, const float* __restrict__ decay,
                             const float* __restrict__ carry_gain, const double* __restrict__ g_sum /*of long prompts*/, const float* __restrict__ w_out, const float* __restrict__ w_fc,
                             const float* __restrict__ b_fc, float* __restrict__ scores, int32_t* __restrict__ labels) {
    extern __shared__ float hs[];                        // per (state, channel) what the starting states add [N Di], g mean [Di], pooled [D], scores [K]
    float* c_s = hs;                                     // [N][Di]
    float* g_s = c_s + m.Di * m.N;
    float* o_s = g_s + m.Di;
    float* sc_s = o_s + m.D;
    const int pr = blockIdx.x;
    const int c0 = prompt_chunk0[pr], c1 = prompt_chunk0[pr + 1];
    const float inv = 1.f / (float)lens[pr];
    const size_t per = (size_t)m.Di * m.N;
    const bool is_long = c1 - c0 >= MB_LONG;
    if (c1 - c0 > 1 && !is_long)
        for (int i = 2 * threadIdx.x; i < m.Di * m.N; i += 2 * blockDim.x) {      // two neighbours at a time (the workspace begins at a multiple of eight bytes)
            const bool two = (per & 1) == 0;
            auto get = [&](const float* p) { return two ? __ldg(reinterpret_cast<const float2*>(p)) : make_float2(__ldg(p), (size_t)i + 1 < per ? __ldg(p + 1) : 0.f); };
            float2 s = get(end_state + c0 * per + i), add = make_float2(0.f, 0.f);
#pragma unroll 4
            for (int ch = c0 + 1; ch < c1; ++ch) {
                const size_t at = ch * per + i;
                const float2 g = get(carry_gain + at), p = get(decay + at), e = get(end_state + at);
                add.x = fmaf(g.x, s.x, add.x); add.y = fmaf(g.y, s.y, add.y);
                s.x = fmaf(p.x, s.x, e.x); s.y = fmaf(p.y, s.y, e.y);
            }
            c_s[i] = add.x;
            if ((size_t)i + 1 < per) c_s[i + 1] = add.y;
        }
    __syncthreads();
    for (int c = threadIdx.x; c < m.Di; c += blockDim.x) {
        double s = 0.0;
        if (is_long) s = g_sum[(size_t)pr * m.Di + c];
        else for (int ch = c0; ch < c1; ++ch) s += chunk_sum[(size_t)ch * m.Di + c];
        if (c1 - c0 > 1 && !is_long) for (int n = 0; n < m.N; ++n) s += (double)c_s[n * m.Di + c];
        g_s[c] = (float)s * inv;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    for (int d = warp; d < m.D; d += n_warps) {
        float acc = 0.f;
        for (int c = lane; c < m.Di; c += 32) acc = fmaf(w_out[(size_t)d * m.Di + c], g_s[c], acc);
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, s);
        if (lane == 0) o_s[d] = acc;
    }
    __syncthreads();
    for (int k = warp; k < m.K; k += n_warps) {
        float acc = 0.f;
        for (int d = lane; d < m.D; d += 32) acc = fmaf(w_fc[(size_t)k * m.D + d], o_s[d], acc);
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, s);
        if (lane == 0) { acc += b_fc[k]; sc_s[k] = acc; if (scores) scores[(size_t)pr * m.K + k] = acc; }
    }
    __syncthreads();
    if (threadIdx.x == 0 && labels) {
        int best = 0;
        for (int k = 1; k < m.K; ++k) if (sc_s[k] > sc_s[best]) best = k;        // lowest index on ties
        labels[pr] = best;
    }
}

size_t al(size_t v) { return (v + 255) & ~(size_t)255; }

bool dims_ok(const sd_mamba_desc* d, MambaDims& m) {
    if (!d || d->vocab < 1 || d->d_model < 1 || d->d_state < 1 || d->d_conv < 1 || d->expand < 1 || d->n_classes < 1 || d->dt_rank < 1) return false;
    m = MambaDims{d->vocab, d->d_model, d->expand * d->d_model, d->d_state, d->dt_rank, d->d_conv, d->n_classes};
    return true;
}

struct Layout { size_t u, gate, end_state, decay, carry_gain, chunk_sum, tok_id, tok_row, chunks, prompt_chunk0, lens, total; };

Layout layout(const MambaDims& m, int64_t T, int64_t n_chunks, int n_prompts) {
    Layout L;
    size_t o = 0;
    auto take = [&](size_t bytes) { const size_t at = o; o += al(bytes); return at; };
    L.u = take((size_t)T * m.Di * 4); L.gate = take((size_t)T * m.Di * 4);      // (with more tokens than the vocabulary has, one row per token of it: fewer)
    L.end_state = take((size_t)n_chunks * m.Di * m.N * 4); L.decay = take((size_t)n_chunks * m.Di * m.N * 4);
    L.carry_gain = take((size_t)n_chunks * m.Di * m.N * 4);
    L.chunk_sum = take((size_t)n_chunks * m.Di * 8);
    L.tok_id = take((size_t)T * 4); L.tok_row = take((size_t)T * 4);
    L.chunks = take((size_t)n_chunks * sizeof(ChunkRec));
    L.prompt_chunk0 = take((size_t)(n_prompts + 1) * 4); L.lens = take((size_t)n_prompts * 4);
    L.total = o;
    return L;
}

}  // namespace
}  // namespace sd

extern "C" size_t sd_mamba_workspace(const sd_mamba_desc* desc, int64_t total_tokens, int n_prompts) {
    sd::MambaDims m;
    if (!sd::dims_ok(desc, m) || total_tokens < 0 || n_prompts < 0) return 0;
    // every prompt may end with a partly filled chunk
    const int64_t n_chunks = total_tokens / sd::MB_CHUNK + n_prompts;
    return sd::layout(m, total_tokens, n_chunks, n_prompts).total;
}

extern "C" sd_status sd_mamba_classify(const sd_mamba_desc* desc, const sd_mamba_weights* w, const int32_t* tokens_dev,
                                       const int64_t* starts_host, const int32_t* lens_host, int n_prompts, float* scores_dev,
                                       int32_t* labels_dev, void* workspace_dev, size_t workspace_bytes, void* cuda_stream) {
    using namespace sd;
    MambaDims m;
    if (!dims_ok(desc, m) || !w || !tokens_dev || !starts_host || !lens_host || n_prompts < 0 || (!scores_dev && !labels_dev)) return SD_ERR_INVALID_ARG;
    if (!w->embed || !w->w_in || !w->w_conv || !w->b_conv || !w->w_x || !w->w_dt || !w->b_dt || !w->a_log || !w->d_skip || !w->w_out || !w->w_fc || !w->b_fc)
        return SD_ERR_INVALID_ARG;
    if (m.N > MB_MAX_N || m.Kc > MB_MAX_CONV || m.Di > MB_MAX_DI || m.D > MB_MAX_D || m.R + 2 * m.N > MB_MAX_X || m.K > MB_MAX_K) return SD_ERR_UNSUPPORTED;
    if (n_prompts == 0) return SD_OK;
    int64_t T = 0;
    for (int i = 0; i < n_prompts; ++i) {
        if (lens_host[i] < 1 || starts_host[i] < 0) return SD_ERR_INVALID_ARG;
        T += lens_host[i];
    }
    if (T > (int64_t)1 << 30) return SD_ERR_CAPACITY;
    if (!workspace_dev || workspace_bytes < sd_mamba_workspace(desc, T, n_prompts)) return SD_ERR_CAPACITY;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;      // (not in a capture: its replays would see this call's prompts)
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) return SD_ERR_CUDA;
    int longest = 0;                                         // chunks of a prompt
    int64_t n_chunks = 0;
    for (int i = 0; i < n_prompts; ++i) {
        const int n = (lens_host[i] - 1) / MB_CHUNK + 1;
        n_chunks += n;
        longest = std::max(longest, n);
    }
    const Layout L = layout(m, T, T / MB_CHUNK + n_prompts, n_prompts);
    char* base = (char*)workspace_dev;
    float* u = (float*)(base + L.u); float* gate = (float*)(base + L.gate);
    ChunkRec* chunks_d = (ChunkRec*)(base + L.chunks);
    int32_t* pc0 = (int32_t*)(base + L.prompt_chunk0); int32_t* lens_d = (int32_t*)(base + L.lens);
    int32_t* tok_id = (int32_t*)(base + L.tok_id); int32_t* tok_row = (int32_t*)(base + L.tok_row);

    // 400 prompts of 109,096 tokens over 21,128: the projection is a fifth of the work token by token
    const bool by_token = T >= m.V;
    const int rows = by_token ? m.V : (int)T;
    int32_t tok0 = 0, chunk0 = 0;
    auto tables = [&](auto& t, int first, int n) {
        int rows_y = 1;
        for (int i = 0; i < n; ++i) {
            const int len = lens_host[first + i], k = (len - 1) / MB_CHUNK + 1;
            t.start[i] = starts_host[first + i]; t.len[i] = len; t.tok0[i] = tok0; t.chunk0[i] = chunk0;
            tok0 += len; chunk0 += k;
            rows_y = std::max(rows_y, std::min(k, MT_ROWS));
        }
        k_mamba_tables<<<dim3((unsigned)n, (unsigned)rows_y), 64, 0, st>>>(t, first, n_prompts, tokens_dev, m.V, by_token ? 1 : 0, chunks_d, pc0, lens_d, tok_id, tok_row);
    };
    if (n_prompts <= MT_FEW) { PromptTable<MT_FEW> t; tables(t, 0, n_prompts); }
    else for (int i = 0; i < n_prompts; i += MT_MANY) { PromptTable<MT_MANY> t; tables(t, i, std::min(MT_MANY, n_prompts - i)); }
    k_mamba_in<<<dim3((unsigned)((rows + MI_ROWS - 1) / MI_ROWS), (unsigned)((2 * m.Di + MI_TILE - 1) / MI_TILE)), 256, 0, st>>>(
        m, by_token ? nullptr : tok_id, rows, w->embed, w->w_in, u, gate);
    const int n_cta = (m.Di + MC_CHANNELS - 1) / MC_CHANNELS, per = ((m.Di + n_cta - 1) / n_cta + 3) & ~3;      // (the last CTA has at least one channel)
    const size_t xp = (size_t)((m.R + 2 * m.N + 3) & ~3), wx_bytes = (size_t)(m.R + 2 * m.N) * per * 4;
    const int w_staged = wx_bytes <= MC_STAGED;
    const size_t chunk_smem = (MC_TILE * xp + (size_t)2 * MC_TILE * MC_PITCH) * 4 + (w_staged ? wx_bytes : 0);
    auto pick = [&](auto cl, auto carry) {
        constexpr bool CL = decltype(cl)::value, CARRY = decltype(carry)::value;
        if (m.N == MB_MAX_N)
            return m.Kc == 4 ? (m.R == 8 ? k_mamba_chunk<MB_MAX_N, 4, 8, CL, CARRY> : k_mamba_chunk<MB_MAX_N, 4, 0, CL, CARRY>) : k_mamba_chunk<MB_MAX_N, 0, 0, CL, CARRY>;
        return m.Kc <= 4 ? k_mamba_chunk<0, -4, 0, CL, CARRY> : k_mamba_chunk<0, 0, 0, CL, CARRY>;
    };
    const std::true_type yes;
    const std::false_type no;
    auto chunk_kernel = longest > 1 ? (n_cta > 1 ? pick(yes, yes) : pick(no, yes)) : (n_cta > 1 ? pick(yes, no) : pick(no, no));
    const size_t head_smem = ((size_t)m.Di * m.N + m.Di + m.D + m.K) * 4;
    // Always the bound over all sizes that are accepted: the attribute belongs to the kernel, and a smaller classifier's call on
    // another thread must not lower it between here and the launch.
    if (cudaFuncSetAttribute(chunk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, MC_MAX_SMEM) != cudaSuccess ||
        cudaFuncSetAttribute(k_mamba_head, cudaFuncAttributeMaxDynamicSharedMemorySize, MH_MAX_SMEM) != cudaSuccess)
        return SD_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(n_chunks * n_cta)); cfg.blockDim = dim3(MC_THREADS); cfg.dynamicSmemBytes = chunk_smem; cfg.stream = st;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)n_cta; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
    cfg.attrs = &attr; cfg.numAttrs = n_cta > 1 ? 1 : 0;
    if (cudaLaunchKernelEx(&cfg, chunk_kernel, m, (const ChunkRec*)chunks_d, (const int32_t*)tok_row, (const float*)u, (const float*)gate, w->w_conv, w->b_conv, w->w_x, w->w_dt, w->b_dt,
                           w->a_log, w->d_skip, (float*)(base + L.end_state), (float*)(base + L.decay), (float*)(base + L.carry_gain),
                           (double*)(base + L.chunk_sum), w_staged, n_cta, per) != cudaSuccess)
        return SD_ERR_CUDA;
    // (u and the gates are not read any more; their place, eight bytes per token and channel, holds eight per prompt and channel)
    double* g_sum = (double*)(base + L.u);
    if (longest >= MB_LONG)
        k_mamba_carry<<<dim3((unsigned)n_prompts, (unsigned)((m.Di + CARRY_CH - 1) / CARRY_CH)), CARRY_CH * MB_MAX_N, 0, st>>>(
            m, (const int32_t*)pc0, (const double*)(base + L.chunk_sum), (const float*)(base + L.end_state), (const float*)(base + L.decay),
            (const float*)(base + L.carry_gain), g_sum);
    k_mamba_head<<<(unsigned)n_prompts, MH_THREADS, head_smem, st>>>(
        m, (const int32_t*)pc0, (const int32_t*)lens_d, (const double*)(base + L.chunk_sum), (const float*)(base + L.end_state), (const float*)(base + L.decay),
        (const float*)(base + L.carry_gain), g_sum, w->w_out, w->w_fc, w->b_fc, scores_dev, labels_dev);
    return cudaGetLastError() == cudaSuccess ? SD_OK : SD_ERR_CUDA;
}
