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
#include <string.h>

#include <algorithm>
#include <type_traits>
#include <vector>

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

// Where every flattened token's projected row is: its own, or its token's when whole vocabulary was projected (one CTA per chunk).
__global__ void k_mamba_tables(const ChunkRec* __restrict__ chunks, const int64_t* __restrict__ starts, const int32_t* __restrict__ tokens, int V, int by_token,
                               int32_t* __restrict__ tok_id, int32_t* __restrict__ tok_row) {
    const ChunkRec ch = chunks[blockIdx.x];
    for (int i = threadIdx.x; i < ch.n_tok; i += blockDim.x) {
        const int tok = min(max(tokens[starts[ch.prompt] + ch.pos0 + i], 0), V - 1);
        tok_id[ch.tok0 + i] = tok;
        tok_row[ch.tok0 + i] = by_token ? tok : ch.tok0 + i;
    }
}

// u, z = split(W_in E[row]) for every row: token by token, or, when the prompts hold more tokens than the vocabulary has, once per
// token of the vocabulary (the projection depends on nothing else).  Bound: fp32 multiply-adds (21,128 rows: 69 us; 109,096 token
// by token, a thread per feature, 757).  128 x 128 tiles of 256
// threads, 8 x 8 sums each in register pairs, 16-deep slices of both operands through two buffers.
constexpr int MI_TILE = 128, MI_K = 16, MI_PITCH = MI_TILE + 4;
__global__ void __launch_bounds__(256, 2)
k_mamba_in(MambaDims m, const int32_t* __restrict__ tok_id /*nullptr: row = token*/, int rows, const float* __restrict__ embed,
           const float* __restrict__ w_in, float* __restrict__ u, float* __restrict__ z) {
    __shared__ __align__(16) float as[2][MI_K][MI_PITCH], bs[2][MI_K][MI_PITCH];
    const int tid = threadIdx.x, r0 = blockIdx.x * MI_TILE, j0 = blockIdx.y * MI_TILE;
    const int lr = tid >> 2, lk = (tid & 3) * 4;                        // this thread loads rows lr and lr + 64, columns lk ... lk + 3
    const float* a_src[2]; const float* b_src[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int r = r0 + lr + 64 * i, j = j0 + lr + 64 * i;
        a_src[i] = r < rows ? embed + (size_t)(tok_id ? tok_id[r] : r) * m.D : nullptr;
        b_src[i] = j < 2 * m.Di ? w_in + (size_t)j * m.D : nullptr;
    }
    const bool vec = (m.D & 3) == 0 && (((uintptr_t)embed | (uintptr_t)w_in) & 15) == 0;
    const bool vec_out = (m.Di & 3) == 0 && (((uintptr_t)u | (uintptr_t)z) & 15) == 0;      // (the workspace may begin at any multiple of 8)
    auto get = [&](const float* src, int k) {
        if (!src) return make_float4(0.f, 0.f, 0.f, 0.f);
        if (vec) return k < m.D ? __ldg(reinterpret_cast<const float4*>(src + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
        return make_float4(k < m.D ? src[k] : 0.f, k + 1 < m.D ? src[k + 1] : 0.f, k + 2 < m.D ? src[k + 2] : 0.f, k + 3 < m.D ? src[k + 3] : 0.f);
    };
    float4 a_next[2], b_next[2];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int i = 0; i < 2; ++i) { a_next[i] = get(a_src[i], k0 + lk); b_next[i] = get(b_src[i], k0 + lk); }
    };
    auto stash = [&](int buf) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            float* a = &as[buf][lk][lr + 64 * i]; float* b = &bs[buf][lk][lr + 64 * i];
            a[0] = a_next[i].x; a[MI_PITCH] = a_next[i].y; a[2 * MI_PITCH] = a_next[i].z; a[3 * MI_PITCH] = a_next[i].w;
            b[0] = b_next[i].x; b[MI_PITCH] = b_next[i].y; b[2 * MI_PITCH] = b_next[i].z; b[3 * MI_PITCH] = b_next[i].w;
        }
    };
    const int tx = tid & 15, ty = tid >> 4;                             // rows 4 ty ..., 64 + 4 ty ...; features 4 tx ..., 64 + 4 tx ...
    f32x2 acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
    fetch(0);
    stash(0);
    __syncthreads();
    for (int k0 = 0, buf = 0; k0 < m.D; k0 += MI_K, buf ^= 1) {
        if (k0 + MI_K < m.D) fetch(k0 + MI_K);
#pragma unroll
        for (int k = 0; k < MI_K; ++k) {
            float av[8];
            *reinterpret_cast<float4*>(av) = *reinterpret_cast<const float4*>(&as[buf][k][4 * ty]);
            *reinterpret_cast<float4*>(av + 4) = *reinterpret_cast<const float4*>(&as[buf][k][64 + 4 * ty]);
            const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(&bs[buf][k][4 * tx]), b1 = *reinterpret_cast<const ulonglong2*>(&bs[buf][k][64 + 4 * tx]);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const f32x2 a2 = f2_pack(av[i], av[i]);
                acc[i][0] = f2_fma(a2, b0.x, acc[i][0]); acc[i][1] = f2_fma(a2, b0.y, acc[i][1]);
                acc[i][2] = f2_fma(a2, b1.x, acc[i][2]); acc[i][3] = f2_fma(a2, b1.y, acc[i][3]);
            }
        }
        if (k0 + MI_K < m.D) { stash(buf ^ 1); __syncthreads(); }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int r = r0 + (i < 4 ? 4 * ty + i : 60 + 4 * ty + i);
        if (r >= rows) continue;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = j0 + 64 * h + 4 * tx;
            const float2 p = f2_unpack(acc[i][2 * h]), q = f2_unpack(acc[i][2 * h + 1]);
            const float v[4] = {p.x, p.y, q.x, q.y};
            if (vec_out) {                                              // (a group of four lies in one of the halves)
                if (j < 2 * m.Di) *reinterpret_cast<float4*>((j < m.Di ? u + (size_t)r * m.Di + j : z + (size_t)r * m.Di + j - m.Di)) = make_float4(v[0], v[1], v[2], v[3]);
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (j + e < 2 * m.Di) (j + e < m.Di ? u[(size_t)r * m.Di + j + e] : z[(size_t)r * m.Di + j + e - m.Di]) = v[e];
            }
        }
    }
}

// Everything of one chunk between the input projection and the pooled sum.  Bound: exponentials (d_state of them per token and
// channel) and the multiply-adds around them.  400 prompts of 109,096 tokens: 0.72 ms (convolution and projections 0.73 ms, two
// scans 0.80 ms as kernels of their own, v, dt, B and C through memory in between); the whole call 2.28 -> 0.81 ms, the error of
// its scores against 64 bits 1.8e-7 -> 1.7e-7.
//   1. convolution + SiLU for MC_TILE tokens at a time into shared memory, from there the projections (r, B, C): a thread takes
//      two tokens and every 16th output, three at a time;
//   2. a thread per channel scans the chunk: convolution again (four multiply-adds are less than a trip through memory), step
//      size, recurrence from a zero state, and the two sums of the chunk (see the top of the file).
//   More than MC_CHANNELS channels: a cluster of up to four CTAs per chunk with as many channels each.  A CTA projects its own channels;
//   the parts of r, B, C meet through distributed shared memory (each CTA adds a share of them, parts in the CTAs' order).  1,024
//   channels, whole call: one prompt of 64 tokens 425 us (1,329 with one CTA for all channels, 904 as kernels of their own), four of
//   100...300 462 (1,378, 999), 400 of 32...512 15.3 ms (17.0, 32.2); 512 channels, one prompt of 64: 172 us (256, 303).
constexpr int MC_TILE = 32, MC_THREADS = 256, MC_CHANNELS = 256, MC_STAGED = 48 * 1024;      // W_x is staged up to this size: two CTAs of the usual sizes still fit an SM
// Most dynamic shared memory a launch takes: B, C, r of a chunk, a tile of v and the staged W_x at their largest.
constexpr int MC_MAX_SMEM = (MB_CHUNK * MB_MAX_X + MC_TILE * (MC_CHANNELS + 4)) * 4 + MC_STAGED;
constexpr int MH_MAX_SMEM = (MB_MAX_DI * MB_MAX_N + MB_MAX_DI + MB_MAX_D + MB_MAX_K) * 4;
template <int NS /*states: 16, or any up to MB_MAX_N as 0*/, int KC /*taps: 4, or any up to four as -4, or up to MB_MAX_CONV as 0*/, bool CL /*several CTAs per chunk*/>
__global__ void __launch_bounds__(MC_THREADS, 2)
k_mamba_chunk(MambaDims m, const ChunkRec* __restrict__ chunks, const int32_t* __restrict__ tok_row, const float* __restrict__ u, const float* __restrict__ z,
              const float* __restrict__ w_conv, const float* __restrict__ b_conv, const float* __restrict__ w_x, const float* __restrict__ w_dt,
              const float* __restrict__ b_dt, const float* __restrict__ a_log, const float* __restrict__ d_skip,
              float* __restrict__ end_state, float* __restrict__ decay, float* __restrict__ carry_gain /*all [chunk][Di][N]*/, double* __restrict__ chunk_sum /*[chunk][Di]*/, int w_staged, int n_cta, int per_cta) {
    extern __shared__ __align__(16) float sm[];
    const int Dp = (m.Di + 3) & ~3, per = CL ? per_cta : Dp;                             // channels of a CTA, padded to a multiple of 4
    const int N = NS ? NS : m.N, n_x = m.R + 2 * m.N, xp = (n_x + 3) & ~3;
    float* xd_s = sm;                                      // [MB_CHUNK][xp]: B, C, r of every token
    float* v_s = sm + MB_CHUNK * xp;                       // [MC_TILE][vp]
    float* wx_s = v_s + MC_TILE * (per + 4);               // this CTA's columns of W_x, [n_x][n_c], if they were given room
    __shared__ int row_s[MB_CHUNK + MB_MAX_CONV];          // rows of the chunk's tokens and of the taps in front of them (-1: before the prompt)
    const int tid = threadIdx.x, vp = per + 4;
    const int chunk = CL ? blockIdx.x / n_cta : blockIdx.x, c_lo = CL ? (int)(blockIdx.x % n_cta) * per : 0, n_c = CL ? min(m.Di - c_lo, per) : m.Di;
    const ChunkRec ch = chunks[chunk];
    constexpr int KM = KC > 0 ? KC : KC < 0 ? -KC : MB_MAX_CONV;
    const int Kc = KC > 0 ? KC : m.Kc, back = Kc - 1;
    for (int i = tid; i < ch.n_tok + back; i += MC_THREADS) row_s[i] = ch.pos0 + i - back >= 0 ? tok_row[ch.tok0 + i - back] : -1;
    if (w_staged) for (int i = tid; i < n_x * n_c; i += MC_THREADS) wx_s[i] = __ldg(CL ? w_x + (size_t)(i / n_c) * m.Di + c_lo + i % n_c : w_x + i);
    const float* wx = w_staged ? wx_s : w_x + c_lo;
    const int w_ld = CL && w_staged ? n_c : m.Di;
    __syncthreads();
    // SiLU(convolution) of channel c at token t; the taps come in the order of the sum
    auto conv = [&](const float (&w)[KM], float b, const float (&x)[KM]) {
        float acc = b;
#pragma unroll
        for (int j = 0; j < KM; ++j) if (j < Kc) acc = fmaf(w[j], x[j], acc);
        return silu_f(acc);
    };
    const bool vec = (m.Di & 3) == 0 && (w_staged || ((uintptr_t)w_x & 15) == 0);      // (then n_c is a multiple of 4 as well)
    for (int t0 = 0; t0 < ch.n_tok; t0 += MC_TILE) {
        const int nt = min(MC_TILE, ch.n_tok - t0);
        for (int i = tid; i < per; i += MC_THREADS) {
            float w[KM], x[KM];
            const int c = c_lo + i;
            const bool on = i < n_c;
#pragma unroll
            for (int j = 0; j < KM; ++j) {
                w[j] = on && j < Kc ? __ldg(w_conv + (size_t)c * Kc + j) : 0.f;
                x[j] = 0.f;
                if (on && j < back) { const int r = row_s[t0 + j]; x[j] = r >= 0 ? __ldg(u + (size_t)r * m.Di + c) : 0.f; }
            }
            const float b = on ? __ldg(b_conv + c) : 0.f;
#pragma unroll 4
            for (int t = 0; t < MC_TILE; ++t) {
                const float nu = on && t < nt ? __ldg(u + (size_t)row_s[t0 + t + back] * m.Di + c) : 0.f;
#pragma unroll
                for (int j = 0; j < KM; ++j) if (j == back) x[j] = nu;
                v_s[t * vp + i] = on && t < nt ? conv(w, b, x) : 0.f;
#pragma unroll
                for (int j = 0; j + 1 < KM; ++j) if (j < back) x[j] = x[j + 1];
            }
        }
        __syncthreads();
        const int t = tid & 15, og = tid >> 4;
        const float* v0 = v_s + t * vp;
        const float* v1 = v0 + 16 * vp;
        for (int o0 = og; o0 < n_x; o0 += 48) {
            const int o1 = o0 + 16, o2 = o0 + 32;
            float s[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            const float* w0 = wx + (size_t)o0 * w_ld;
            const float* w1 = wx + (size_t)min(o1, n_x - 1) * w_ld;
            const float* w2 = wx + (size_t)min(o2, n_x - 1) * w_ld;
            if (vec) {
#pragma unroll 2
                for (int c = 0; c < n_c; c += 4) {
                    const float4 a = *reinterpret_cast<const float4*>(v0 + c), b = *reinterpret_cast<const float4*>(v1 + c);
                    const float4 p = *reinterpret_cast<const float4*>(w0 + c), q = *reinterpret_cast<const float4*>(w1 + c), r = *reinterpret_cast<const float4*>(w2 + c);
                    s[0] = fmaf(p.x, a.x, s[0]); s[0] = fmaf(p.y, a.y, s[0]); s[0] = fmaf(p.z, a.z, s[0]); s[0] = fmaf(p.w, a.w, s[0]);
                    s[1] = fmaf(p.x, b.x, s[1]); s[1] = fmaf(p.y, b.y, s[1]); s[1] = fmaf(p.z, b.z, s[1]); s[1] = fmaf(p.w, b.w, s[1]);
                    s[2] = fmaf(q.x, a.x, s[2]); s[2] = fmaf(q.y, a.y, s[2]); s[2] = fmaf(q.z, a.z, s[2]); s[2] = fmaf(q.w, a.w, s[2]);
                    s[3] = fmaf(q.x, b.x, s[3]); s[3] = fmaf(q.y, b.y, s[3]); s[3] = fmaf(q.z, b.z, s[3]); s[3] = fmaf(q.w, b.w, s[3]);
                    s[4] = fmaf(r.x, a.x, s[4]); s[4] = fmaf(r.y, a.y, s[4]); s[4] = fmaf(r.z, a.z, s[4]); s[4] = fmaf(r.w, a.w, s[4]);
                    s[5] = fmaf(r.x, b.x, s[5]); s[5] = fmaf(r.y, b.y, s[5]); s[5] = fmaf(r.z, b.z, s[5]); s[5] = fmaf(r.w, b.w, s[5]);
                }
            } else {
                for (int c = 0; c < n_c; ++c) {
                    const float a = v0[c], b = v1[c], p = w0[c], q = w1[c], r = w2[c];
                    s[0] = fmaf(p, a, s[0]); s[1] = fmaf(p, b, s[1]); s[2] = fmaf(q, a, s[2]); s[3] = fmaf(q, b, s[3]); s[4] = fmaf(r, a, s[4]); s[5] = fmaf(r, b, s[5]);
                }
            }
            // kept as [B | C | r], so that a token's B and C can be read by fours
            auto at = [&](int o) { return o < m.R ? 2 * m.N + o : o - m.R; };
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int o = o0 + 16 * i;
                if (o < n_x) {
                    if (t < nt) xd_s[(t0 + t) * xp + at(o)] = s[2 * i];
                    if (t + 16 < nt) xd_s[(t0 + t + 16) * xp + at(o)] = s[2 * i + 1];
                }
            }
        }
        __syncthreads();
    }
    if (CL) {                                              // the other CTAs' channels: every value is added by one CTA, which hands the sum to all
        namespace cg = cooperative_groups;
        cg::cluster_group cluster = cg::this_cluster();
        cluster.sync();
        const int n = ch.n_tok * xp, share = (n + n_cta - 1) / n_cta, i0 = (int)(blockIdx.x % n_cta) * share;
        for (int i = i0 + tid; i < min(n, i0 + share); i += MC_THREADS) {
            float v[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) v[r] = r < n_cta ? cluster.map_shared_rank(xd_s, r)[i] : 0.f;
            const float sum = ((v[0] + v[1]) + v[2]) + v[3];
#pragma unroll
            for (int r = 0; r < 4; ++r) if (r < n_cta) cluster.map_shared_rank(xd_s, r)[i] = sum;
        }
        cluster.sync();                                    // (no CTA touches another's shared memory from here on)
    }
    for (int c = c_lo + tid; c < c_lo + n_c; c += MC_THREADS) {
        float w[KM], x[KM];
#pragma unroll
        for (int j = 0; j < KM; ++j) {
            w[j] = j < Kc ? __ldg(w_conv + (size_t)c * Kc + j) : 0.f;
            x[j] = 0.f;
            if (j < back) { const int r = row_s[j]; x[j] = r >= 0 ? __ldg(u + (size_t)r * m.Di + c) : 0.f; }
        }
        const float b = __ldg(b_conv + c), bdt = __ldg(b_dt + c), dsk = __ldg(d_skip + c);
        float wd[8];                                       // the first eight columns of the channel's row of W_dt (the rest, if any, is read as needed)
#pragma unroll
        for (int r = 0; r < 8; ++r) wd[r] = r < m.R ? __ldg(w_dt + (size_t)c * m.R + r) : 0.f;
        float A[MB_MAX_N];
        f32x2 h[MB_MAX_N / 2], P[MB_MAX_N / 2], G[MB_MAX_N / 2];
#pragma unroll
        for (int n = 0; n < MB_MAX_N; ++n) A[n] = n < N ? -expf(__ldg(a_log + (size_t)c * m.N + n)) * 1.4426950408889634f : 0.f;      // (decays as powers of two)
#pragma unroll
        for (int n = 0; n < MB_MAX_N / 2; ++n) { h[n] = 0ull; P[n] = f2_pack(1.f, 1.f); G[n] = 0ull; }
        double sum = 0.0;                                  // (in double here and over the chunks: the sum's rounding would be the largest of all)
        float nu = __ldg(u + (size_t)row_s[back] * m.Di + c), nz = __ldg(z + (size_t)row_s[back] * m.Di + c);
        for (int t = 0; t < ch.n_tok; ++t) {
            const float zt = nz;
#pragma unroll
            for (int j = 0; j < KM; ++j) if (j == back) x[j] = nu;
            if (t + 1 < ch.n_tok) {                        // the next token's values are on their way during this one
                const size_t r = (size_t)row_s[t + 1 + back] * m.Di + c;
                nu = __ldg(u + r); nz = __ldg(z + r);
            }
            const float v = conv(w, b, x);
#pragma unroll
            for (int j = 0; j + 1 < KM; ++j) if (j < back) x[j] = x[j + 1];
            const float* xd = xd_s + t * xp;
            float dt = bdt;
#pragma unroll
            for (int r = 0; r < 8; ++r) if (r < m.R) dt = fmaf(wd[r], xd[2 * m.N + r], dt);
            for (int r = 8; r < m.R; ++r) dt = fmaf(__ldg(w_dt + (size_t)c * m.R + r), xd[2 * m.N + r], dt);
            dt = softplus_f(dt);
            const float dx = dt * v, g = silu_f(zt);
            const f32x2 dx2 = f2_pack(dx, dx), g2 = f2_pack(g, g);
            f32x2 y2 = 0ull;
#pragma unroll
            for (int n = 0; n < MB_MAX_N / 2; ++n) {
                if (2 * n < N) {
                    const bool odd = NS ? false : 2 * n + 1 >= N;      // (an unused second state: its decay is one, its input zero)
                    const f32x2 a = f2_pack(exp2f(dt * A[2 * n]), odd ? 1.f : exp2f(dt * A[2 * n + 1]));
                    const f32x2 B2 = NS ? *reinterpret_cast<const f32x2*>(xd + 2 * n) : f2_pack(xd[2 * n], odd ? 0.f : xd[2 * n + 1]);
                    const f32x2 C2 = NS ? *reinterpret_cast<const f32x2*>(xd + NS + 2 * n) : f2_pack(xd[m.N + 2 * n], odd ? 0.f : xd[m.N + 2 * n + 1]);
                    h[n] = f2_fma(a, h[n], f2_mul(dx2, B2));
                    P[n] = f2_mul(P[n], a);
                    y2 = f2_fma(h[n], C2, y2);
                    G[n] = f2_fma(f2_mul(g2, C2), P[n], G[n]);
                }
            }
            const float2 y = f2_unpack(y2);
            sum += (double)(fmaf(dsk, v, y.x + y.y) * g);
        }
        chunk_sum[(size_t)chunk * m.Di + c] = sum;
        const size_t at = ((size_t)chunk * m.Di + c) * m.N;
#pragma unroll
        for (int n = 0; n < MB_MAX_N / 2; ++n) {
            if (2 * n < N) {
                const float2 hv = f2_unpack(h[n]), pv = f2_unpack(P[n]), gv = f2_unpack(G[n]);
                end_state[at + 2 * n] = hv.x; decay[at + 2 * n] = pv.x; carry_gain[at + 2 * n] = gv.x;
                if (NS || 2 * n + 1 < N) { end_state[at + 2 * n + 1] = hv.y; decay[at + 2 * n + 1] = pv.y; carry_gain[at + 2 * n + 1] = gv.y; }
            }
        }
    }
}

// The pooled sums of long prompts: what the chunks' starting states add and the chunks' own sums, a thread per (channel, state) and a CTA
// per eight channels instead of the head's one CTA per prompt, with the coefficients of eight chunks on their way at a time.  Bound: latency
// of the chain over chunks.  One prompt of 4,000 / 30,000 / 200,000 tokens, whole call: 140 / 366 / 1,628 us,
// in the head 203 / 869 / 6,758 (as kernels of their own, before: 275 / 802 / 4,757).  From eight chunks on a queue of shorter prompts is the slower
// for the launch (100 prompts of 32...512 tokens: 323 against 319).
constexpr int MB_LONG = 16;                              // chunks from which on a prompt is long
constexpr int CARRY_CH = 8, CARRY_BATCH = 8;
__global__ void __launch_bounds__(CARRY_CH * MB_MAX_N)
k_mamba_carry(MambaDims m, const int32_t* __restrict__ prompt_chunk0, const double* __restrict__ chunk_sum, const float* __restrict__ end_state,
              const float* __restrict__ decay, const float* __restrict__ carry_gain, double* __restrict__ g_sum /*[prompt][Di]*/) {
    const int c0 = prompt_chunk0[blockIdx.x], c1 = prompt_chunk0[blockIdx.x + 1];
    if (c1 - c0 < MB_LONG) return;
    const int n = threadIdx.x % MB_MAX_N, c = blockIdx.y * CARRY_CH + threadIdx.x / MB_MAX_N;
    const bool on = c < m.Di && n < m.N;
    const size_t per = (size_t)m.Di * m.N, i = (size_t)min(c, m.Di - 1) * m.N + min(n, m.N - 1);
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
#pragma unroll
    for (int o = MB_MAX_N / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (n == 0 && c < m.Di) g_sum[(size_t)blockIdx.x * m.Di + c] = sum;
}

// Per prompt: the states its chunks start from (serial, a thread per channel and state), mean over tokens of the gated outputs
// (chunks in order), W_out, the classification layer, argmax.
__global__ void k_mamba_head(MambaDims m, const int32_t* __restrict__ prompt_chunk0, const int32_t* __restrict__ lens,
                             const double* __restrict__ chunk_sum, const float* __restrict__ end_state, const float* __restrict__ decay,
                             const float* __restrict__ carry_gain, const double* __restrict__ g_sum /*of long prompts*/, const float* __restrict__ w_out, const float* __restrict__ w_fc,
                             const float* __restrict__ b_fc, float* __restrict__ scores, int32_t* __restrict__ labels) {
    extern __shared__ float hs[];                        // per (channel, state) what the starting states add [Di N], g mean [Di], pooled [D], scores [K]
    float* c_s = hs;
    float* g_s = c_s + m.Di * m.N;
    float* o_s = g_s + m.Di;
    float* sc_s = o_s + m.D;
    const int pr = blockIdx.x;
    const int c0 = prompt_chunk0[pr], c1 = prompt_chunk0[pr + 1];
    const float inv = 1.f / (float)lens[pr];
    const size_t per = (size_t)m.Di * m.N;
    const bool is_long = c1 - c0 >= MB_LONG;
    if (c1 - c0 > 1 && !is_long)
        for (int i = threadIdx.x; i < m.Di * m.N; i += blockDim.x) {
            float s = end_state[c0 * per + i], add = 0.f;
#pragma unroll 4
            for (int ch = c0 + 1; ch < c1; ++ch) {
                const size_t at = ch * per + i;
                add = fmaf(carry_gain[at], s, add);
                s = fmaf(decay[at], s, end_state[at]);
            }
            c_s[i] = add;
        }
    __syncthreads();
    for (int c = threadIdx.x; c < m.Di; c += blockDim.x) {
        double s = 0.0;
        if (is_long) s = g_sum[(size_t)pr * m.Di + c];
        else for (int ch = c0; ch < c1; ++ch) s += chunk_sum[(size_t)ch * m.Di + c];
        if (c1 - c0 > 1 && !is_long) for (int n = 0; n < m.N; ++n) s += (double)c_s[c * m.N + n];
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

struct Layout { size_t u, z, end_state, decay, carry_gain, chunk_sum, tok_id, tok_row, chunks, prompt_chunk0, lens, starts, total; };

Layout layout(const MambaDims& m, int64_t T, int64_t n_chunks, int n_prompts) {
    Layout L;
    size_t o = 0;
    auto take = [&](size_t bytes) { const size_t at = o; o += al(bytes); return at; };
    L.u = take((size_t)T * m.Di * 4); L.z = take((size_t)T * m.Di * 4);      // (with more tokens than the vocabulary has, one row per token of it: fewer)
    L.end_state = take((size_t)n_chunks * m.Di * m.N * 4); L.decay = take((size_t)n_chunks * m.Di * m.N * 4);
    L.carry_gain = take((size_t)n_chunks * m.Di * m.N * 4);
    L.chunk_sum = take((size_t)n_chunks * m.Di * 8);
    L.tok_id = take((size_t)T * 4); L.tok_row = take((size_t)T * 4);
    L.chunks = take((size_t)n_chunks * sizeof(ChunkRec));                    // from here on: uploaded in one copy
    L.prompt_chunk0 = take((size_t)(n_prompts + 1) * 4); L.lens = take((size_t)n_prompts * 4); L.starts = take((size_t)n_prompts * 8);
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
    // host tables: the chunks of every prompt (the per-token tables are filled on the device from them)
    std::vector<int32_t> prompt_chunk0((size_t)n_prompts + 1);
    std::vector<ChunkRec> chunks;
    int64_t t = 0;
    for (int i = 0; i < n_prompts; ++i) {
        prompt_chunk0[i] = (int32_t)chunks.size();
        for (int p = 0; p < lens_host[i]; p += MB_CHUNK) {
            const int n = lens_host[i] - p < MB_CHUNK ? lens_host[i] - p : MB_CHUNK;
            chunks.push_back(ChunkRec{i, (int32_t)t, n, p});
            t += n;
        }
    }
    prompt_chunk0[n_prompts] = (int32_t)chunks.size();
    int longest = 0;                                         // chunks of a prompt
    for (int i = 0; i < n_prompts; ++i) longest = std::max(longest, prompt_chunk0[i + 1] - prompt_chunk0[i]);
    const int64_t n_chunks = (int64_t)chunks.size();
    const Layout L = layout(m, T, T / MB_CHUNK + n_prompts, n_prompts);
    char* base = (char*)workspace_dev;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    std::vector<char> host(L.starts + (size_t)n_prompts * 8 - L.chunks);
    memcpy(host.data(), chunks.data(), (size_t)n_chunks * sizeof(ChunkRec));
    memcpy(host.data() + (L.prompt_chunk0 - L.chunks), prompt_chunk0.data(), (size_t)(n_prompts + 1) * 4);
    memcpy(host.data() + (L.lens - L.chunks), lens_host, (size_t)n_prompts * 4);
    memcpy(host.data() + (L.starts - L.chunks), starts_host, (size_t)n_prompts * 8);
    if (cudaMemcpyAsync(base + L.chunks, host.data(), host.size(), cudaMemcpyHostToDevice, st) != cudaSuccess) return SD_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return SD_ERR_CUDA;      // the host tables above go out of scope
    float* u = (float*)(base + L.u); float* z = (float*)(base + L.z);
    const ChunkRec* chunks_d = (const ChunkRec*)(base + L.chunks);
    const int32_t* pc0 = (const int32_t*)(base + L.prompt_chunk0);
    int32_t* tok_id = (int32_t*)(base + L.tok_id); int32_t* tok_row = (int32_t*)(base + L.tok_row);

    // 400 prompts of 109,096 tokens over 21,128: the projection is a fifth of the work token by token
    const bool by_token = T >= m.V;
    const int rows = by_token ? m.V : (int)T;
    k_mamba_tables<<<(unsigned)n_chunks, 64, 0, st>>>(chunks_d, (const int64_t*)(base + L.starts), tokens_dev, m.V, by_token ? 1 : 0, tok_id, tok_row);
    k_mamba_in<<<dim3((unsigned)((rows + MI_TILE - 1) / MI_TILE), (unsigned)((2 * m.Di + MI_TILE - 1) / MI_TILE)), 256, 0, st>>>(
        m, by_token ? nullptr : tok_id, rows, w->embed, w->w_in, u, z);
    const int n_cta = (m.Di + MC_CHANNELS - 1) / MC_CHANNELS, per = ((m.Di + n_cta - 1) / n_cta + 3) & ~3;      // (the last CTA has at least one channel)
    const size_t xp = (size_t)((m.R + 2 * m.N + 3) & ~3), wx_bytes = (size_t)(m.R + 2 * m.N) * per * 4;
    const int w_staged = wx_bytes <= MC_STAGED;
    const size_t chunk_smem = (MB_CHUNK * xp + (size_t)MC_TILE * (per + 4)) * 4 + (w_staged ? wx_bytes : 0);
    auto pick = [&](auto cl) {
        constexpr bool CL = decltype(cl)::value;
        if (m.N == MB_MAX_N) return m.Kc == 4 ? k_mamba_chunk<MB_MAX_N, 4, CL> : k_mamba_chunk<MB_MAX_N, 0, CL>;
        return m.Kc <= 4 ? k_mamba_chunk<0, -4, CL> : k_mamba_chunk<0, 0, CL>;
    };
    auto chunk_kernel = n_cta > 1 ? pick(std::true_type()) : pick(std::false_type());
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
    if (cudaLaunchKernelEx(&cfg, chunk_kernel, m, chunks_d, (const int32_t*)tok_row, (const float*)u, (const float*)z, w->w_conv, w->b_conv, w->w_x, w->w_dt, w->b_dt,
                           w->a_log, w->d_skip, (float*)(base + L.end_state), (float*)(base + L.decay), (float*)(base + L.carry_gain),
                           (double*)(base + L.chunk_sum), w_staged, n_cta, per) != cudaSuccess)
        return SD_ERR_CUDA;
    // (u and z are not read any more; their place, eight bytes per token and channel, holds eight per prompt and channel)
    double* g_sum = (double*)(base + L.u);
    if (longest >= MB_LONG)
        k_mamba_carry<<<dim3((unsigned)n_prompts, (unsigned)((m.Di + CARRY_CH - 1) / CARRY_CH)), CARRY_CH * MB_MAX_N, 0, st>>>(
            m, pc0, (const double*)(base + L.chunk_sum), (const float*)(base + L.end_state), (const float*)(base + L.decay),
            (const float*)(base + L.carry_gain), g_sum);
    k_mamba_head<<<(unsigned)n_prompts, 1024, head_smem, st>>>(
        m, pc0, (const int32_t*)(base + L.lens), (const double*)(base + L.chunk_sum), (const float*)(base + L.end_state), (const float*)(base + L.decay),
        (const float*)(base + L.carry_gain), g_sum, w->w_out, w->w_fc, w->b_fc, scores_dev, labels_dev);
    return cudaGetLastError() == cudaSuccess ? SD_OK : SD_ERR_CUDA;
}
