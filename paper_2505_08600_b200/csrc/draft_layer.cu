// A draft layer over at most eight token rows in two kernels, one for attention and one for the feed-forward part.
//
// One kernel per matrix (gemv.cu) makes five hand-overs between all SMs per layer, and with at most eight rows a hand-over (last store,
// kernel boundary, first load) costs as much as the work between two of them.  Here a layer is cut the other way, by heads and by
// feed-forward features, over clusters of four CTAs:
//   k_draft_attention  a cluster per head: the head's query, key and value rows of QKV, rotary embedding, cache append, attention over the
//                      head's cache, and the head's columns of Wo;
//   k_draft_mlp        a cluster per 128 or 192 features: their gate and up rows, SwiGLU, and their columns of the down matrix.
// Inside a cluster, CTAs hand over through distributed shared memory (a cluster barrier instead of a kernel boundary).  What a cluster
// leaves is a piece of the layer's output for all columns; the next kernel's clusters each add all pieces (in their order: the same
// sums in every cluster and from run to run), take the norm, and go on.  Weights are in registers before the wait for the kernel before
// (16-byte loads in the order of the MMA's operands, see gemv.cu), and the first tiles of the cache in shared memory.
// Activations enter the matrices in two bf16 parts, queries, keys, values and the cache in one, sums in fp32, as on the other paths.
// Bound: latency.  12 layers of 768 columns at 512 positions, one row, us after the wait: k_draft_attention 1.6 pieces added up, 0.6 barrier,
// 0.6 QKV, 0.5 rotation, 0.7 barrier, 0.8 attention, 1.3 its merge, 0.4 barrier, 0.6 Wo; k_draft_mlp 1.3, 0.5, 1.0, 0.5, 0.5, 0.7; between two
// kernels 0.5.  17.5 -> 13 us per layer, 7B iteration 4,014 -> 3,698 us, 1B (drafts of two layers) 1,058 -> 1,035.  Where they are taken: api.cu.
#include "draft_layer.h"

#include <cooperative_groups.h>

#include "tc_ptx.cuh"

namespace sd {
namespace {

namespace cg = cooperative_groups;

constexpr int RANKS = 4;                        // CTAs of a cluster
constexpr int WARPS = 16, THREADS = 32 * WARPS;
constexpr int ROWS = DL_MAX_ROWS;
constexpr int HD = 64;
constexpr int MAX_D = 1024;
// Clusters of both kernels that are resident side by side (a CTA per SM; clusters of four fill 35 or 36 places of the B200's 148 SMs when they come
// and go).  One more and the last cluster of either kernel begins when the other kernel ends: 12 + 24 clusters 18.4 us per layer.
constexpr int MAX_CLUSTERS = 32;
constexpr int ACC_COLS = MAX_D / RANKS;         // columns of the residual stream that a CTA adds up
constexpr int RED_FLOATS = WARPS * 3 * 16 * ROWS;      // largest exchange between warps (also holds WARPS x ACC_COLS)
static_assert(RED_FLOATS >= WARPS * ACC_COLS, "partial sums of the pieces fit");
constexpr int TILE_KEYS = 16, TILE_BYTES = TILE_KEYS * HD * 2, DEPTH = 2;      // a warp's tile of keys (and one of values), tiles on their way

__host__ __device__ constexpr int row_pitch(int d) { return 2 * d + 64; }      // bytes of a row in shared memory: rows 64 bytes apart modulo 128

__device__ __forceinline__ uint4 ldg_stream(const bf16* p) {           // weights: read once per pass
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ void cluster_arrive() { __syncwarp(); asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

struct Plan { int pos[ROWS], slot[ROWS], tok[ROWS]; };

// Which position and token every row stands for (the rules of the embedding kernel).  tokens: only where they are needed, behind the wait.
__device__ __forceinline__ void make_plan(const DraftLayer& p, Plan& plan, bool report) {
    const int m = threadIdx.x;
    if (m >= ROWS) return;
    int pos = -1, slot = 0, tok = 0;
    if (m < p.n_seq * p.rows_per_seq) {
        const int i = m / p.rows_per_seq, j = m % p.rows_per_seq;
        slot = p.ids[i];
        const int len = p.S.len[slot];
        if (p.rows_per_seq == 2) { pos = len - 2 + j; if (pos < p.S.dkv[slot] || pos < 0) pos = -1; }
        else pos = len - 1 + p.step;
        if (p.embed) {
            tok = p.rows_per_seq == 2 ? (pos < 0 ? 0 : p.S.tokens[(size_t)slot * p.S.tok_stride + pos]) : p.x[(size_t)p.out[i] * p.gamma + p.step - 1];
            if (tok < 0 || tok >= p.vocab) { if (report) atomicOr(p.S.status, SD_DEV_BAD_TOKEN); tok = 0; }
        }
        if (pos >= p.max_ctx) { if (report && p.embed) atomicOr(p.S.status, SD_DEV_BAD_POS); pos = -1; }
    }
    plan.pos[m] = pos; plan.slot[m] = slot; plan.tok[m] = tok;
}

// This CTA's columns of the residual stream: added up, handed to h_out (by one cluster), normed, and spread over the cluster as the
// rows of the matrix's operand; the rows' sums of squares as well.  All threads; the caller's cluster barrier makes it visible.
// AHEAD: pieces whose loads are on their way at a time.
template <int AHEAD>
__device__ __forceinline__ void rows_in(const DraftLayer& p, cg::cluster_group& cluster, int rank, bool writer, const Plan& plan, float4 gain, float* acc, uint8_t* xs,
                        float (*ssq)[ROWS][2]) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, rows = p.n_seq * p.rows_per_seq;
    const int cols = p.d / RANKS, c4n = cols / 4, base = rank * cols;
    const int row = t >> 6, c4 = t & 63;                                // two warps per row: four columns per thread
    const bool mine = row < rows && c4 < c4n;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (p.embed) {
        if (mine) {
            const uint2 raw = __ldg(reinterpret_cast<const uint2*>(p.embed + (size_t)plan.tok[row] * p.d + base + 4 * c4));
            const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.x)), b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.y));
            v = make_float4(a.x, a.y, b.x, b.y);
        }
    } else {
        const int lg = rows > 4 ? 3 : rows > 2 ? 2 : rows > 1 ? 1 : 0, groups = WARPS >> lg;     // warps that share a row's pieces
        const int wr = warp & ((1 << lg) - 1), grp = warp >> lg;
        if (wr < rows) {
            float4 s[2] = {v, v};
            if (grp == 0) {
#pragma unroll
                for (int i = 0; i < 2; ++i)
                    if (lane + 32 * i < c4n) s[i] = __ldcg(reinterpret_cast<const float4*>(p.h_in + (size_t)wr * p.d + base) + lane + 32 * i);
            }
            for (int q0 = grp; q0 < p.n_in; q0 += AHEAD * groups) {
                float4 a[AHEAD][2];
#pragma unroll
                for (int k = 0; k < AHEAD; ++k) {
                    const int q = q0 + k * groups;
#pragma unroll
                    for (int i = 0; i < 2; ++i)
                        a[k][i] = q < p.n_in && lane + 32 * i < c4n
                                      ? __ldcg(reinterpret_cast<const float4*>(p.part_in + ((size_t)q * ROWS + wr) * p.d + base) + lane + 32 * i) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
#pragma unroll
                for (int k = 0; k < AHEAD; ++k)
#pragma unroll
                    for (int i = 0; i < 2; ++i) { s[i].x += a[k][i].x; s[i].y += a[k][i].y; s[i].z += a[k][i].z; s[i].w += a[k][i].w; }
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
                if (lane + 32 * i < c4n) reinterpret_cast<float4*>(acc + warp * ACC_COLS)[lane + 32 * i] = s[i];
        }
        __syncthreads();
        if (mine)
            for (int g0 = 0; g0 < groups; g0 += 4) {
                float4 a[4];
#pragma unroll
                for (int g = 0; g < 4; ++g)
                    a[g] = g0 + g < groups ? reinterpret_cast<const float4*>(acc + (row + ((g0 + g) << lg)) * ACC_COLS)[c4] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int g = 0; g < 4; ++g) { v.x += a[g].x; v.y += a[g].y; v.z += a[g].z; v.w += a[g].w; }
            }
    }
    float ss = 0.f;
    if (mine) {
        if (writer) __stcg(reinterpret_cast<float4*>(p.h_out + (size_t)row * p.d + base) + c4, v);
        ss = (v.x * v.x + v.y * v.y) + (v.z * v.z + v.w * v.w);
        const float x[4] = {v.x * gain.x, v.y * gain.y, v.z * gain.z, v.w * gain.w};
        uint32_t hi[2], lo[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            hi[i] = pack_bf16(x[2 * i], x[2 * i + 1]);
            const float2 h = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&hi[i]));
            lo[i] = pack_bf16(x[2 * i] - h.x, x[2 * i + 1] - h.y);
        }
        const int at = row * row_pitch(p.d) + 2 * (base + 4 * c4);
#pragma unroll
        for (int r = 0; r < RANKS; ++r) {
            uint8_t* dst = cluster.map_shared_rank(xs, r) + at;
            *reinterpret_cast<uint2*>(dst) = make_uint2(hi[0], hi[1]);
            *reinterpret_cast<uint2*>(dst + ROWS * row_pitch(p.d)) = make_uint2(lo[0], lo[1]);
        }
    }
    ss = warp_sum(ss);
    if (lane < RANKS && row < rows) cluster.map_shared_rank(&ssq[0][0][0], lane)[(rank * ROWS + row) * 2 + (warp & 1)] = ss;
}

__device__ __forceinline__ float row_scale(const float (*ssq)[ROWS][2], int m, int d, float eps) {
    float s = 0.f;
#pragma unroll
    for (int r = 0; r < RANKS; ++r) s += ssq[r][m][0] + ssq[r][m][1];
    return rsqrtf(s / (float)d + eps);
}

// One 16-row tile times the rows' two parts over one 32-wide k block (a sum for each part: the MMAs of one wait for one another).
__device__ __forceinline__ void mma_block(float (&acc)[2][4], const uint4& p, const uint4& q, const uint4& hi, const uint4& lo) {
    mma_bf16(acc[0], p.x, q.x, p.y, q.y, hi.x, hi.y);
    mma_bf16(acc[1], p.x, q.x, p.y, q.y, lo.x, lo.y);
    mma_bf16(acc[0], p.z, q.z, p.w, q.w, hi.z, hi.w);
    mma_bf16(acc[1], p.z, q.z, p.w, q.w, lo.z, lo.w);
}
__device__ __forceinline__ void clear(float (&acc)[2][4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[0][i] = acc[1][i] = 0.f;
}

// Sixteen output features (tile `warp` of this CTA's quarter of them) times the rows, over 32 NK of the cluster's columns, left as a piece.
// weights(k, a, b): the operand of k block k, rows gid and gid + 8 of the tile.
template <int NK, class W>
__device__ __forceinline__ void piece_out(const DraftLayer& p, int rank, int piece, W weights, const uint8_t* xs, int pitch) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, gid = lane >> 2, tig = lane & 3, rows = p.n_seq * p.rows_per_seq;
    if (16 * warp >= p.d / RANKS) return;
    float acc[2][4];
    clear(acc);
#pragma unroll
    for (int k = 0; k < NK; ++k) {
        const uint8_t* x = xs + gid * pitch + 64 * k + 16 * tig;
        uint4 a, b;
        weights(k, a, b);
        mma_block(acc, a, b, *reinterpret_cast<const uint4*>(x), *reinterpret_cast<const uint4*>(x + ROWS * pitch));
    }
    const int n = rank * (p.d / RANKS) + 16 * warp + gid, m = 2 * tig;
    float* dst = p.part_out + ((size_t)piece * ROWS + m) * p.d + n;
    if (m < rows) { __stcg(dst, acc[0][0] + acc[1][0]); __stcg(dst + 8, acc[0][2] + acc[1][2]); }
    if (m + 1 < rows) { __stcg(dst + p.d, acc[0][1] + acc[1][1]); __stcg(dst + p.d + 8, acc[0][3] + acc[1][3]); }
}

struct AttnShared {
    Plan plan;
    float ssq[RANKS][ROWS][2];
    __align__(16) bf16 qkv[3][ROWS][HD];        // the head's new queries, keys and values
    float o[WARPS][2][HD], ml[WARPS][2][2];        // per warp and row of its sequence: output (not normalised), running max and sum
    float ro[RANKS][ROWS][HD], rml[RANKS][ROWS][2];        // the same per CTA of the cluster
    __align__(16) uint8_t xo[2 * ROWS * row_pitch(HD)];    // the head's attention output in two parts
};

// NB: 32-wide k blocks of QKV per warp.
template <int NB>
__global__ void __cluster_dims__(RANKS, 1, 1) __launch_bounds__(THREADS, 1) k_draft_attention(const __grid_constant__ DraftLayer p) {
    extern __shared__ __align__(128) uint8_t dyn[];
    __shared__ AttnShared sh;
    pdl_launch_dependents();
    cg::cluster_group cluster = cg::this_cluster();
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, gid = lane >> 2, tig = lane & 3;
    const int rank = blockIdx.x % RANKS, head = blockIdx.x / RANKS, d = p.d, H = p.n_heads, rows = p.n_seq * p.rows_per_seq;
    uint8_t* ring = dyn;                                               // [WARPS][DEPTH][keys, values]
    uint8_t* xs = dyn + WARPS * DEPTH * 2 * TILE_BYTES;                // [2][ROWS] rows of row_pitch(d) bytes
    float* red = reinterpret_cast<float*>(xs + 2 * ROWS * row_pitch(d));
    cluster_arrive();                                                  // (waited for in front of the first write into another CTA)

    // ---- weights: tile mat = 16 features, eight of the head's lower half and the eight they are rotated with
    uint4 wa[NB][3], wb[NB][3], oa[2], ob[2];
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int mat = 0; mat < 3; ++mat) {
            const int kb = warp + WARPS * b;
            const bf16* w = p.w_in + (size_t)((mat * H + head) * HD + 8 * rank + gid) * d + 32 * kb + 8 * tig;
            const bool on = 32 * kb < d;
            wa[b][mat] = on ? ldg_stream(w) : make_uint4(0, 0, 0, 0);
            wb[b][mat] = on ? ldg_stream(w + (size_t)(HD / 2) * d) : make_uint4(0, 0, 0, 0);
        }
    {
        const int n = rank * (d / RANKS) + 16 * warp + gid;
        const bool on = 16 * warp < d / RANKS;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const bf16* w = p.w_out + (size_t)n * (H * HD) + head * HD + 32 * k + 8 * tig;
            oa[k] = on ? ldg_stream(w) : make_uint4(0, 0, 0, 0);
            ob[k] = on ? ldg_stream(w + (size_t)8 * (H * HD)) : make_uint4(0, 0, 0, 0);
        }
    }
    float4 gain = make_float4(0.f, 0.f, 0.f, 0.f);
    if ((t & 63) < d / RANKS / 4) gain = __ldg(reinterpret_cast<const float4*>(p.gain + rank * (d / RANKS)) + (t & 63));
    if (t == 0) stamp_first(p.stamp, ST_START);

    // ---- row plan.  The state it comes from changes between passes only, and the pass's first kernel begins behind them; a later one
    //      may read it, and the cache positions in front of the pass's, ahead of its wait.
    if (p.embed) { pdl_wait(); if (t == 0) stamp_pair(p.stamp, ST_DEP_FIRST); }
    make_plan(p, sh.plan, head == 0 && rank == 0);
    __syncthreads();
    // this warp's sequence and its share of the sequence's tiles of 16 keys, over all warps of the cluster
    const int s = warp % p.n_seq, r0 = s * p.rows_per_seq, last = r0 + p.rows_per_seq - 1;
    const int len = max(sh.plan.pos[r0], sh.plan.pos[last]) + 1, slot = sh.plan.slot[r0];
    const int old_len = sh.plan.pos[r0] >= 0 ? sh.plan.pos[r0] : max(sh.plan.pos[last], 0);      // positions that earlier passes wrote
    const int n_sub = (WARPS - s + p.n_seq - 1) / p.n_seq, share = rank * n_sub + warp / p.n_seq, n_share = RANKS * n_sub;
    const int tiles = (len + TILE_KEYS - 1) / TILE_KEYS, t_lo = share * tiles / n_share, n_t = (share + 1) * tiles / n_share - t_lo;
    const size_t head_at = ((size_t)slot * H + head) * p.max_ctx * HD;
    uint8_t* my_ring = ring + warp * DEPTH * 2 * TILE_BYTES;
    const uint32_t ring_sa = smem_u32(my_ring);
    auto request = [&](int i) {                                        // tile i of this warp, as far as earlier passes wrote it
        const int k0 = (t_lo + i) * TILE_KEYS, nk = min(TILE_KEYS, old_len - k0);
        const uint32_t dst = ring_sa + (uint32_t)(i % DEPTH) * 2u * TILE_BYTES;
        const bf16* ks = p.kc + head_at + (size_t)k0 * HD;
        const bf16* vs = p.vc + head_at + (size_t)k0 * HD;
#pragma unroll
        for (int c = lane; c < TILE_KEYS * 8; c += 32) {
            const int key = c >> 3, ch = c & 7;
            const uint32_t off = (uint32_t)key * (HD * 2) + (uint32_t)((ch ^ (key & 7)) << 4);
            if (key < nk) { cp_async16(dst + off, ks + c * 8); cp_async16(dst + TILE_BYTES + off, vs + c * 8); }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int i = 0; i < DEPTH; ++i) if (i < n_t) request(i);
    // rotary factors of the pair this thread finishes
    const int ftok = t & 7, fe = (t >> 3) & 7, fmat = t >> 6;
    const int fpos = ftok < rows ? sh.plan.pos[ftok] : -1;
    float cs = 1.f, sn = 0.f;
    if (fmat < 2 && fpos >= 0) { cs = __ldg(p.rcos + (size_t)fpos * (HD / 2) + 8 * rank + fe); sn = __ldg(p.rsin + (size_t)fpos * (HD / 2) + 8 * rank + fe); }

    if (!p.embed) { pdl_wait(); if (t == 0) stamp_pair(p.stamp, ST_DEP_FIRST); }
    cluster_wait();                                                    // every CTA of the cluster is there
    rows_in<4>(p, cluster, rank, head == 0, sh.plan, gain, red, xs, sh.ssq);
    cluster_arrive(); cluster_wait();

    // ---- queries, keys, values
    {
        float acc[3][2][4];
#pragma unroll
        for (int mat = 0; mat < 3; ++mat) clear(acc[mat]);
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const int kb = warp + WARPS * b;
            if (32 * kb >= d) break;                                   // uniform in a warp
            const uint8_t* x = xs + gid * row_pitch(d) + 64 * kb + 16 * tig;
            const uint4 hi = *reinterpret_cast<const uint4*>(x), lo = *reinterpret_cast<const uint4*>(x + ROWS * row_pitch(d));
#pragma unroll
            for (int mat = 0; mat < 3; ++mat) mma_block(acc[mat], wa[b][mat], wb[b][mat], hi, lo);
        }
#pragma unroll
        for (int mat = 0; mat < 3; ++mat) {                            // [warp][feature][row]
            float* r = red + ((warp * 3 + mat) * 16 + gid) * ROWS + 2 * tig;
            *reinterpret_cast<float2*>(r) = make_float2(acc[mat][0][0] + acc[mat][1][0], acc[mat][0][1] + acc[mat][1][1]);
            *reinterpret_cast<float2*>(r + 8 * ROWS) = make_float2(acc[mat][0][2] + acc[mat][1][2], acc[mat][0][3] + acc[mat][1][3]);
        }
    }
    __syncthreads();
    if (fmat < 3 && ftok < rows) {
        float v0 = 0.f, v1 = 0.f;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) {
            const float* r = red + ((w * 3 + fmat) * 16 + fe) * ROWS + ftok;
            v0 += r[0]; v1 += r[8 * ROWS];
        }
        const float sc = row_scale(sh.ssq, ftok, d, p.eps);
        v0 *= sc; v1 *= sc;
        const bf16 b0 = __float2bfloat16_rn(v0 * cs - v1 * sn), b1 = __float2bfloat16_rn(v0 * sn + v1 * cs);
        const int e = 8 * rank + fe;
#pragma unroll
        for (int r = 0; r < RANKS; ++r) {
            bf16* dst = cluster.map_shared_rank(&sh.qkv[fmat][ftok][0], r) + e;
            dst[0] = b0; dst[HD / 2] = b1;
        }
        if (fmat > 0 && fpos >= 0) {
            bf16* dst = (fmat == 1 ? p.kc : p.vc) + (((size_t)sh.plan.slot[ftok] * H + head) * p.max_ctx + fpos) * HD + e;
            dst[0] = b0; dst[HD / 2] = b1;
        }
    }
    cluster_arrive(); cluster_wait();

    // ---- attention: a warp per share of a sequence's keys, one or two of the MMA's sixteen query rows in use
    {
        uint32_t a[HD / 16][2];
        const bool on = gid < p.rows_per_seq;
        const int pos = on ? sh.plan.pos[r0 + gid] : -1;
#pragma unroll
        for (int ks = 0; ks < HD / 16; ++ks) {
            const bf16* q = &sh.qkv[0][r0 + (on ? gid : 0)][16 * ks + 2 * tig];
            a[ks][0] = on ? *reinterpret_cast<const uint32_t*>(q) : 0u;
            a[ks][1] = on ? *reinterpret_cast<const uint32_t*>(q + 8) : 0u;
        }
        const float sl2 = rsqrtf((float)HD) * 1.4426950408889634f;     // softmax scale in the exp2 domain
        float m_run = -INFINITY, l_run = 0.f, O[HD / 8][4];
#pragma unroll
        for (int i = 0; i < HD / 8; ++i) O[i][0] = O[i][1] = O[i][2] = O[i][3] = 0.f;
        const int mi = lane >> 3, lr = lane & 7;
        for (int i = 0; i < n_t; ++i) {
            const int k0 = (t_lo + i) * TILE_KEYS;
            if (i + 1 < n_t) asm volatile("cp.async.wait_group %0;" ::"n"(DEPTH - 1) : "memory");
            else asm volatile("cp.async.wait_group 0;" ::: "memory");
            uint8_t* kt = my_ring + (i % DEPTH) * 2 * TILE_BYTES;
            if (k0 + TILE_KEYS > old_len) {                            // this pass's keys and values, and zeros behind them (finite: their weight is zero)
                for (int c = lane; c < TILE_KEYS * 8; c += 32) {
                    const int key = c >> 3, ch = c & 7, pk = k0 + key;
                    if (pk < old_len) continue;
                    const int off = key * (HD * 2) + ((ch ^ (key & 7)) << 4);
                    uint4 kv = make_uint4(0, 0, 0, 0), vv = kv;
                    for (int j = r0; j <= last; ++j)
                        if (sh.plan.pos[j] == pk) { kv = reinterpret_cast<const uint4*>(sh.qkv[1][j])[ch]; vv = reinterpret_cast<const uint4*>(sh.qkv[2][j])[ch]; }
                    *reinterpret_cast<uint4*>(kt + off) = kv;
                    *reinterpret_cast<uint4*>(kt + TILE_BYTES + off) = vv;
                }
            }
            __syncwarp();
            const uint32_t kb = smem_u32(kt), vb = kb + TILE_BYTES;
            float S[2][4];
#pragma unroll
            for (int n = 0; n < 2; ++n) S[n][0] = S[n][1] = S[n][2] = S[n][3] = 0.f;
            {
                const int key = 8 * (mi >> 1) + lr;
#pragma unroll
                for (int ks = 0; ks < HD / 16; ++ks) {
                    uint32_t b[4];
                    ldmatrix_x4(kb + (uint32_t)key * (HD * 2) + (uint32_t)(((2 * ks + (mi & 1)) ^ (key & 7)) << 4), b);
                    mma_bf16(S[0], a[ks][0], 0u, a[ks][1], 0u, b[0], b[1]);
                    mma_bf16(S[1], a[ks][0], 0u, a[ks][1], 0u, b[2], b[3]);
                }
            }
            float mx = -INFINITY;
#pragma unroll
            for (int n = 0; n < 2; ++n)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int pk = k0 + 8 * n + 2 * tig + e;
                    S[n][e] = pk <= pos ? S[n][e] * sl2 : -INFINITY;
                    mx = fmaxf(mx, S[n][e]);
                }
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1)); mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            const float mn = fmaxf(m_run, mx), corr = mn == -INFINITY ? 1.f : exp2f(m_run - mn);
            m_run = mn;
            float sum = 0.f;
#pragma unroll
            for (int n = 0; n < 2; ++n)
#pragma unroll
                for (int e = 0; e < 2; ++e) { S[n][e] = mn == -INFINITY ? 0.f : exp2f(S[n][e] - mn); sum += S[n][e]; }
            l_run = l_run * corr + sum;
            const uint32_t pa0 = pack_bf16(S[0][0], S[0][1]), pa2 = pack_bf16(S[1][0], S[1][1]);
            {
                const int key = 8 * (mi & 1) + lr;
#pragma unroll
                for (int nv = 0; nv < HD / 8; nv += 2) {
                    O[nv][0] *= corr; O[nv][1] *= corr; O[nv + 1][0] *= corr; O[nv + 1][1] *= corr;
                    uint32_t v[4];
                    ldmatrix_x4_trans(vb + (uint32_t)key * (HD * 2) + (uint32_t)(((nv + (mi >> 1)) ^ (key & 7)) << 4), v);
                    mma_bf16(O[nv], pa0, 0u, pa2, 0u, v[0], v[1]);
                    mma_bf16(O[nv + 1], pa0, 0u, pa2, 0u, v[2], v[3]);
                }
            }
            __syncwarp();                                              // the tile's place may be filled again
            if (i + DEPTH < n_t) request(i + DEPTH);
        }
        l_run += __shfl_xor_sync(0xffffffffu, l_run, 1); l_run += __shfl_xor_sync(0xffffffffu, l_run, 2);
        if (gid < 2) {
#pragma unroll
            for (int nv = 0; nv < HD / 8; ++nv) *reinterpret_cast<float2*>(&sh.o[warp][gid][8 * nv + 2 * tig]) = make_float2(O[nv][0], O[nv][1]);
            if (tig == 0) { sh.ml[warp][gid][0] = m_run; sh.ml[warp][gid][1] = l_run; }
        }
    }
    __syncthreads();
    {   // the CTA's warps, then the cluster's CTAs: weights relative to the largest score seen
        const int m = t >> 6, e = t & 63;
        if (m < rows) {
            const int sq = m / p.rows_per_seq, j = m % p.rows_per_seq;
            float M = -INFINITY, L = 0.f, acc = 0.f, mw[WARPS], lw[WARPS], ow[WARPS];
#pragma unroll
            for (int k = 0; k < WARPS; ++k) {                          // (all reads on their way at once)
                const int w = sq + k * p.n_seq;
                const bool on = w < WARPS;
                mw[k] = on ? sh.ml[w][j][0] : -INFINITY; lw[k] = on ? sh.ml[w][j][1] : 0.f; ow[k] = on ? sh.o[w][j][e] : 0.f;
            }
#pragma unroll
            for (int k = 0; k < WARPS; ++k) M = fmaxf(M, mw[k]);
#pragma unroll
            for (int k = 0; k < WARPS; ++k) {
                const float f = mw[k] == -INFINITY ? 0.f : exp2f(mw[k] - M);
                L = fmaf(f, lw[k], L);
                acc = fmaf(f, ow[k], acc);
            }
#pragma unroll
            for (int r = 0; r < RANKS; ++r) cluster.map_shared_rank(&sh.ro[rank][m][0], r)[e] = acc;
            if (e < RANKS) { float* dst = cluster.map_shared_rank(&sh.rml[rank][m][0], e); dst[0] = M; dst[1] = L; }
        }
    }
    cluster_arrive(); cluster_wait();                                  // (the last access to another CTA's shared memory)
    {
        const int m = t >> 6, e = t & 63;
        if (m < rows) {
            float M = -INFINITY, L = 0.f, acc = 0.f;
#pragma unroll
            for (int r = 0; r < RANKS; ++r) M = fmaxf(M, sh.rml[r][m][0]);
#pragma unroll
            for (int r = 0; r < RANKS; ++r) {
                const float mr = sh.rml[r][m][0], f = mr == -INFINITY ? 0.f : exp2f(mr - M);
                L = fmaf(f, sh.rml[r][m][1], L);
                acc = fmaf(f, sh.ro[r][m][e], acc);
            }
            const float x = L > 0.f ? acc * (1.f / L) : 0.f;
            const bf16 hi = __float2bfloat16_rn(x);
            bf16* dst = reinterpret_cast<bf16*>(sh.xo + m * row_pitch(HD)) + e;
            dst[0] = hi;
            dst[ROWS * row_pitch(HD) / 2] = __float2bfloat16_rn(x - __bfloat162float(hi));
        }
    }
    __syncthreads();
    piece_out<2>(p, rank, head, [&](int k, uint4& a, uint4& b) { a = oa[k]; b = ob[k]; }, sh.xo, row_pitch(HD));
    if (t == 0) stamp_pair(p.stamp, ST_DONE_FIRST);
}

// NB: 32-wide k blocks of gate/up per group of two warps.  FC: features of a CTA (32 or 48).  The down matrix's part waits in shared memory: in
// registers beside gate/up's it would leave none for the work.
template <int NB, int FC>
__global__ void __cluster_dims__(RANKS, 1, 1) __launch_bounds__(THREADS, 1) k_draft_mlp(const __grid_constant__ DraftLayer p) {
    constexpr int TILES = 2 * FC / 16, MINE = TILES / 2, KG = WARPS / 2, FEATURES = RANKS * FC, NK = FEATURES / 32;      // tiles: eight features' gate and up rows; KG groups of k blocks
    static_assert(KG * TILES * 16 * ROWS <= RED_FLOATS, "exchange between the groups");
    extern __shared__ __align__(128) uint8_t dyn[];
    __shared__ float ssq[RANKS][ROWS][2];
    __shared__ __align__(16) uint8_t act[2 * ROWS * row_pitch(FEATURES)];         // the cluster's activations in two parts
    __shared__ Plan plan;                                              // (not used: the rows come from the kernel before; for rows_in, which is the same for both kernels)
    pdl_launch_dependents();
    cg::cluster_group cluster = cg::this_cluster();
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, gid = lane >> 2, tig = lane & 3;
    const int rank = blockIdx.x % RANKS, piece = blockIdx.x / RANKS, d = p.d, rows = p.n_seq * p.rows_per_seq;
    uint8_t* xs = dyn;
    float* red = reinterpret_cast<float*>(xs + 2 * ROWS * row_pitch(d));
    uint8_t* wd = reinterpret_cast<uint8_t*>(red + RED_FLOATS);        // [d / RANKS] rows of row_pitch(FEATURES) bytes
    cluster_arrive();
    const int half = warp & 1, kg = warp >> 1;
    uint4 wa[NB][MINE], wb[NB][MINE];
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int i = 0; i < MINE; ++i) {
            const int kb = kg + KG * b, f = piece * FEATURES + rank * FC + 8 * (MINE * half + i) + gid;      // gate rows of 64 features, then their up rows
            const bf16* w = p.w_in + (size_t)((f >> 6) * 128 + (f & 63)) * d + 32 * kb + 8 * tig;
            const bool on = 32 * kb < d;
            wa[b][i] = on ? ldg_stream(w) : make_uint4(0, 0, 0, 0);
            wb[b][i] = on ? ldg_stream(w + (size_t)64 * d) : make_uint4(0, 0, 0, 0);
        }
    for (int i = t; i < d / RANKS * (FEATURES / 8); i += THREADS) {
        const int n = i / (FEATURES / 8), c = i % (FEATURES / 8);
        cp_async16(smem_u32(wd) + (uint32_t)(n * row_pitch(FEATURES) + 16 * c), p.w_out + (size_t)(rank * (d / RANKS) + n) * p.F + piece * FEATURES + 8 * c);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    float4 gain = make_float4(0.f, 0.f, 0.f, 0.f);
    if ((t & 63) < d / RANKS / 4) gain = __ldg(reinterpret_cast<const float4*>(p.gain + rank * (d / RANKS)) + (t & 63));
    if (t == 0) stamp_first(p.stamp, ST_START);
    pdl_wait();
    if (t == 0) stamp_pair(p.stamp, ST_DEP_FIRST);
    cluster_wait();
    rows_in<2>(p, cluster, rank, piece == 0, plan, gain, red, xs, ssq);
    cluster_arrive(); cluster_wait();
    {
        float acc[MINE][2][4];
#pragma unroll
        for (int i = 0; i < MINE; ++i) clear(acc[i]);
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const int kb = kg + KG * b;
            if (32 * kb >= d) break;
            const uint8_t* x = xs + gid * row_pitch(d) + 64 * kb + 16 * tig;
            const uint4 hi = *reinterpret_cast<const uint4*>(x), lo = *reinterpret_cast<const uint4*>(x + ROWS * row_pitch(d));
#pragma unroll
            for (int i = 0; i < MINE; ++i) mma_block(acc[i], wa[b][i], wb[b][i], hi, lo);
        }
#pragma unroll
        for (int i = 0; i < MINE; ++i) {                               // [group][tile][feature][row]
            float* r = red + ((kg * TILES + MINE * half + i) * 16 + gid) * ROWS + 2 * tig;
            *reinterpret_cast<float2*>(r) = make_float2(acc[i][0][0] + acc[i][1][0], acc[i][0][1] + acc[i][1][1]);
            *reinterpret_cast<float2*>(r + 8 * ROWS) = make_float2(acc[i][0][2] + acc[i][1][2], acc[i][0][3] + acc[i][1][3]);
        }
    }
    __syncthreads();
    {
        const int m = t & 7, f = t >> 3;                               // row and feature this thread finishes
        if (f < FC && m < rows) {
            float g = 0.f, u = 0.f;
#pragma unroll
            for (int k = 0; k < KG; ++k) {
                const float* r = red + ((k * TILES + (f >> 3)) * 16 + (f & 7)) * ROWS + m;
                g += r[0]; u += r[8 * ROWS];
            }
            const float sc = row_scale(ssq, m, d, p.eps);
            g *= sc; u *= sc;
            const float x = g / (1.f + expf(-g)) * u;
            const bf16 hi = __float2bfloat16_rn(x), lo = __float2bfloat16_rn(x - __bfloat162float(hi));
#pragma unroll
            for (int r = 0; r < RANKS; ++r) {
                bf16* dst = reinterpret_cast<bf16*>(cluster.map_shared_rank(act, r) + m * row_pitch(FEATURES)) + rank * FC + f;
                dst[0] = hi;
                dst[ROWS * row_pitch(FEATURES) / 2] = lo;
            }
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");               // (this thread's part of the down matrix; the barrier covers the others')
    cluster_arrive(); cluster_wait();                                  // (the last access to another CTA's shared memory)
    const uint8_t* w0 = wd + (16 * warp + gid) * row_pitch(FEATURES) + 16 * tig;
    piece_out<NK>(p, rank, piece, [&](int k, uint4& a, uint4& b) {
        a = *reinterpret_cast<const uint4*>(w0 + 64 * k); b = *reinterpret_cast<const uint4*>(w0 + 8 * row_pitch(FEATURES) + 64 * k);
    }, act, row_pitch(FEATURES));
    if (t == 0) stamp_pair(p.stamp, ST_DONE_FIRST);
}

// A CTA of 64 threads per row and DL_TAIL columns.
__global__ void __launch_bounds__(64) k_draft_tail(const __grid_constant__ DraftLayer p, bf16* __restrict__ xn, int lo_off, float* __restrict__ ssq, int ssq_stride) {
    __shared__ float red[2];
    pdl_launch_dependents();
    const int row = blockIdx.x, k = blockIdx.y * DL_TAIL + 4 * threadIdx.x;
    const bool on = k < p.d;
    float4 gain = make_float4(0.f, 0.f, 0.f, 0.f), v = gain;
    if (on) gain = __ldg(reinterpret_cast<const float4*>(p.gain + k));
    pdl_wait();
    if (on) {
        v = __ldcg(reinterpret_cast<const float4*>(p.h_in + (size_t)row * p.d + k));
#pragma unroll 16
        for (int q = 0; q < p.n_in; ++q) {
            const float4 a = __ldcg(reinterpret_cast<const float4*>(p.part_in + ((size_t)q * ROWS + row) * p.d + k));
            v.x += a.x; v.y += a.y; v.z += a.z; v.w += a.w;
        }
        const float x[4] = {v.x * gain.x, v.y * gain.y, v.z * gain.z, v.w * gain.w};
        uint32_t hi[2], lo[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            hi[i] = pack_bf16(x[2 * i], x[2 * i + 1]);
            const float2 h = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&hi[i]));
            lo[i] = pack_bf16(x[2 * i] - h.x, x[2 * i + 1] - h.y);
        }
        *reinterpret_cast<uint2*>(xn + (size_t)row * p.d + k) = make_uint2(hi[0], hi[1]);
        *reinterpret_cast<uint2*>(xn + (size_t)(row + lo_off) * p.d + k) = make_uint2(lo[0], lo[1]);
    }
    const float ss = warp_sum((v.x * v.x + v.y * v.y) + (v.z * v.z + v.w * v.w));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    if (threadIdx.x == 0) ssq[(size_t)row * ssq_stride + blockIdx.y] = red[0] + red[1];
}

size_t attn_smem(int d) { return (size_t)WARPS * DEPTH * 2 * TILE_BYTES + 2 * ROWS * row_pitch(d) + RED_FLOATS * sizeof(float); }
size_t mlp_smem(int d, int features) { return (size_t)2 * ROWS * row_pitch(d) + RED_FLOATS * sizeof(float) + (size_t)(d / RANKS) * row_pitch(features); }

bool valid(const DraftLayer& p) {
    return p.n_seq >= 1 && (p.rows_per_seq == 1 || p.rows_per_seq == 2) && p.n_seq * p.rows_per_seq <= ROWS && p.d >= 64 && p.d <= MAX_D && p.d % 64 == 0;
}

template <typename K>
cudaError_t launch(K kern, int clusters, size_t smem, size_t most, int dependent, const DraftLayer& p, cudaStream_t st) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);      // (of any width: other threads launch the same kernel)
    if (e != cudaSuccess) return e;
    return launch_pdl(kern, dim3(clusters * RANKS), dim3(THREADS), smem, st, dependent, p);
}

}  // namespace

// Features of a cluster: the fewest with which both kernels' clusters are resident side by side; 0: none.
static int features_of(int n_heads, int F) {
    for (int f : {128, 192})
        if (F % f == 0 && n_heads + F / f <= MAX_CLUSTERS) return f;
    return 0;
}

bool draft_layer_fits(const sd_model_desc& m, int rows) {
    return m.dtype == SD_BF16 && rows >= 1 && rows <= ROWS && m.head_dim == HD && m.n_heads == m.n_kv_heads && m.d_model % 64 == 0 && m.d_model <= MAX_D &&
           features_of(m.n_heads, m.d_ffn) > 0;
}
int draft_layer_pieces(const sd_model_desc& m) { return m.d_ffn / features_of(m.n_heads, m.d_ffn); }

size_t draft_layer_scratch(const sd_model_desc& m) {
    return sizeof(float) * (size_t)ROWS * m.d_model * (2 + m.n_heads + draft_layer_pieces(m));
}

cudaError_t launch_draft_attention(const DraftLayer& p, int dependent, cudaStream_t st) {
    if (!valid(p)) return cudaErrorInvalidValue;
    return p.d <= 32 * WARPS ? launch(k_draft_attention<1>, p.n_heads, attn_smem(p.d), attn_smem(MAX_D), dependent, p, st)
                             : launch(k_draft_attention<2>, p.n_heads, attn_smem(p.d), attn_smem(MAX_D), dependent, p, st);
}

cudaError_t launch_draft_mlp(const DraftLayer& p, cudaStream_t st) {
    const int f = features_of(p.n_heads, p.F);
    if (!valid(p) || !f) return cudaErrorInvalidValue;
    const int n = p.F / f;
    const size_t smem = mlp_smem(p.d, f), most = mlp_smem(MAX_D, 192);
    if (f == 128) return p.d <= 512 ? launch(k_draft_mlp<2, 32>, n, smem, most, 1, p, st) : launch(k_draft_mlp<4, 32>, n, smem, most, 1, p, st);
    return p.d <= 512   ? launch(k_draft_mlp<2, 48>, n, smem, most, 1, p, st)
           : p.d <= 768 ? launch(k_draft_mlp<3, 48>, n, smem, most, 1, p, st)
                        : launch(k_draft_mlp<4, 48>, n, smem, most, 1, p, st);
}

cudaError_t launch_draft_tail(const DraftLayer& p, bf16* xn, int lo_off, float* ssq, int ssq_stride, cudaStream_t st) {
    if (!valid(p)) return cudaErrorInvalidValue;
    return launch_pdl(k_draft_tail, dim3(p.n_seq * p.rows_per_seq, (p.d + DL_TAIL - 1) / DL_TAIL), dim3(DL_TAIL / 4), 0, st, 1, p, xn, lo_off, ssq, ssq_stride);
}

}  // namespace sd
