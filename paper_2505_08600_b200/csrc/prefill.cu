// Prefill: the prompt rows of several sequences in one pass of a bf16 model (Section 2.1: the prompt goes through the
// target and the routed draft before the first iteration).  Hundreds of rows make the GEMMs a matter of tensor time
// instead of weight bandwidth, which asks for other tiles than the weight-streaming GEMM of the decoding passes:
//   k_pf_gemm       two CTAs of a cluster work on one tile of 256 output features x up to 256 token rows
//                   (tcgen05.mma.cta_group::2: each CTA loads 128 features and half of the token rows, so a byte that
//                   reaches shared memory is used twice as often as in a one-CTA tile); persistent, the accumulators of two
//                   tiles in TMEM so that a tile's epilogue runs under the next tile's MMAs.  QKV (rotary embedding, cache
//                   append) and gate/up (SwiGLU) finish in the epilogue; Wo and down leave fp32 sums for
//   k_pf_norm       residual add and the next RMSNorm, a CTA per row (folded around the GEMM as in the decoding passes: the
//                   rows are multiplied by the gain before it, its sums by the row's 1/rms in the epilogue).  (As an epilogue
//                   of Wo and down the step was slower: 1B layer at 1289 rows 210 us against 187 - a matrix of one wave of
//                   tiles has nothing to hide its epilogue under, and the next GEMM's CTAs cannot start loading weights while
//                   this one's hold the shared memory.)
//   k_pf_attention  causal attention, 64 query rows per CTA, online softmax
// A weight matrix is read from HBM once per pass whatever the number of rows (at most PF_MAX_ROWS).
// Measured (7B, 511 rows): 216 us per layer, of which QKV 45, gate/up 70, Wo 17, down 40 (tensor time at 1.65 PFLOP/s: 31, 56,
// 10, 28); sequence by sequence in 256-row passes of the weight-streaming GEMM it was 406.
#include <cuda.h>
#include <string.h>

#include <type_traits>

#include "prefill.h"
#include "tc_ptx.cuh"

namespace sd {
namespace {

constexpr int TILE_F = 128;                    // features per CTA
constexpr int TILE_K = 64;                     // one 128-byte swizzle row
constexpr int W_BYTES = TILE_F * TILE_K * 2;
constexpr int PF_GROUPS = 2;                   // groups of four epilogue warps; they take a tile's chunks in turn
constexpr int PF_THREADS = 64 + 128 * PF_GROUPS;
constexpr int PF_MAX_STAGES = 10;
constexpr int PF_RING = 192 * 1024;
constexpr int PF_CHUNK = 32;                   // accumulator columns (token rows) an epilogue thread takes at a time

struct PfShared {
    uint64_t full[PF_MAX_STAGES], empty[PF_MAX_STAGES], tfull[2], tempty[2];
    uint32_t tmem_base;
    int abort_flag, epi_abort[PF_GROUPS];
    float ex[PF_GROUPS][PF_CHUNK / 2][TILE_F]; // exchange between features half a head (or 64: gate and up) apart
};

__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}
// Tile into this CTA's shared memory; the bytes are counted on a barrier of the pair's first CTA.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.cta_group::2.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;"
        ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y), "l"(policy) : "memory");
}
__device__ __forceinline__ void umma_bf16_pair(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"(accumulate) : "memory");
}
// Arrives on the barrier at this offset in both CTAs once the MMAs issued so far have finished.
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr) : "memory");
}

// Which tile and which part of the reduction an item is: token tiles of the same weights next to each other.
struct Item { int ft, tt, piece, kb0, kb1; };
__device__ __forceinline__ Item item_of(const PrefillGemm& g, int it) {
    Item o;
    o.tt = it % g.n_tt;
    const int r = it / g.n_tt;
    o.ft = g.ft0 + r % g.n_ft;
    o.piece = r / g.n_ft;
    o.kb0 = (int)((long long)o.piece * g.kb / g.split);
    o.kb1 = (int)((long long)(o.piece + 1) * g.kb / g.split);
    return o;
}

// The low-rank update of feature n for 32 token rows (a row's adapter is the same in every lane).
__device__ __forceinline__ void add_lora(const PrefillGemm& g, int t0, int n, bool live, uint32_t (&v)[32]) {
    float b[32];
    int cur = -1;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        if (t0 + j >= g.rows) break;
        const int task = __ldcg(g.lora_task + t0 + j);
        if (task < 0 || task >= g.lora_n) continue;
        if (task != cur) {
            cur = task;
            const bf16* p = g.lora_b + ((size_t)task * g.n_out + (live ? n : 0)) * g.lora_r;
#pragma unroll
            for (int k = 0; k < 32; k += 8) {               // r is a multiple of 8, at most 32
                const uint4 raw = k < g.lora_r ? __ldg(reinterpret_cast<const uint4*>(p + k)) : make_uint4(0, 0, 0, 0);
                const __nv_bfloat162* h2 = reinterpret_cast<const __nv_bfloat162*>(&raw);
#pragma unroll
                for (int e = 0; e < 4; ++e) { const float2 f = __bfloat1622float2(h2[e]); b[k + 2 * e] = f.x; b[k + 2 * e + 1] = f.y; }
            }
        }
        const float* t = g.lora_t + (size_t)(t0 + j) * 128 + task * g.lora_r;
        float acc = 0.f;
#pragma unroll
        for (int k = 0; k < 32; k += 4)
            if (k < g.lora_r) {
                const float4 x = __ldcg(reinterpret_cast<const float4*>(t + k));
                acc = fmaf(x.x, b[k], acc); acc = fmaf(x.y, b[k + 1], acc); acc = fmaf(x.z, b[k + 2], acc); acc = fmaf(x.w, b[k + 3], acc);
            }
        v[j] = __float_as_uint(fmaf(g.lora_scale, acc, __uint_as_float(v[j])));
    }
}

// Bound: tensor cores (hundreds of rows), or HBM when the rows are few.  ST: with time stamps (as tests of the pointer they cost a prompt of
// 17 rows 4 %: every kernel of a chain reads its parameters once more before its first load and after its last store).
template <int MODE, bool LORA, bool ST>
__global__ void __launch_bounds__(PF_THREADS, 1) __cluster_dims__(2, 1, 1)
k_pf_gemm(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ PrefillGemm g, uint32_t* status) {
    extern __shared__ uint8_t dyn_smem[];
    __shared__ PfShared sh;
    pdl_launch_dependents();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t crank = blockIdx.x & 1u;
    const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
    const uint32_t tiles0 = (smem_u32(dyn_smem) + 1023u) & ~1023u;
    const uint32_t x_bytes = (uint32_t)g.bn * 64u, stage_bytes = W_BYTES + x_bytes;      // half of the token rows x 128 bytes
    volatile int* abort_flag = &sh.abort_flag;
    if (ST && threadIdx.x == 0) stamp_first(g.stamp, ST_START);
    uint32_t tmem_cols = 32;
    while (tmem_cols < 2u * (uint32_t)g.bn) tmem_cols <<= 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < g.stages; ++s) { mbar_init(smem_u32(&sh.full[s]), 1); mbar_init(smem_u32(&sh.empty[s]), 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(smem_u32(&sh.tfull[b]), 1); mbar_init(smem_u32(&sh.tempty[b]), 2 * 4 * PF_GROUPS); }
        sh.abort_flag = 0;
        for (int i = 0; i < PF_GROUPS; ++i) sh.epi_abort[i] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh.tmem_base)), "r"(tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync_all();                                    // both CTAs' barriers exist before either is signalled
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = sh.tmem_base;

    if (warp == 0) {
        // ------------------------------------------------------------------ producer: this CTA's features and its half of the token rows
        const bool leader = elect_one();
        uint64_t pol_w, pol_x;
        if (g.keep_w) asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol_w));
        else asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol_w));
        asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol_x));
        const uint32_t full0 = map_to_rank(smem_u32(&sh.full[0]), 0u);
        int s = 0; uint32_t use = 0;
        bool ok = true, waited = false;
        uint32_t done = 0;
        // The ring is filled with weights before the wait for the kernel before; the token rows of those stages follow.
        auto weights = [&](const Item& o, int kb, int st) {
            if (leader) {
                if (crank == 0) mbar_expect_tx(smem_u32(&sh.full[st]), 2u * stage_bytes);
                tma_load_2d_pair(tiles0 + st * stage_bytes, &tm_w, kb * TILE_K, o.ft * 2 * TILE_F + (int)crank * TILE_F, full0 + 8u * st, pol_w);
            }
        };
        auto rows = [&](const Item& o, int kb, int st) {
            if (leader) tma_load_2d_pair(tiles0 + st * stage_bytes + W_BYTES, &tm_x, kb * TILE_K, o.tt * g.bn + (int)crank * (g.bn / 2), full0 + 8u * st, pol_x);
        };
        for (int it = pair; it < g.n_items && ok; it += n_pairs) {
            const Item o = item_of(g, it);
            int kb = o.kb0;
            if (!waited) {
                const int ahead = min(g.stages, o.kb1 - o.kb0);
                for (int j = 0; j < ahead; ++j) weights(o, kb + j, j);
                pdl_wait();
                if (ST && leader) stamp_pair(g.stamp, ST_DEP_FIRST);
                waited = true;
                for (int j = 0; j < ahead; ++j) rows(o, kb + j, j);
                kb += ahead; s = ahead; done = ahead;
                if (s == g.stages) { s = 0; use = 1; }
            }
            for (; kb < o.kb1; ++kb) {
                if (use > 0u && !mbar_wait_warp(smem_u32(&sh.empty[s]), (use & 1u) ^ 1u, abort_flag)) { ok = false; break; }
                weights(o, kb, s);
                rows(o, kb, s);
                ++done;
                if (++s == g.stages) { s = 0; ++use; }
            }
        }
        // nobody leaves while its shared memory may still be read or its barriers signalled: wait for the last use of every stage
        const uint32_t n = min(done, (uint32_t)g.stages);
        for (uint32_t j = 0; j < n && ok; ++j) {
            if (s == 0) { s = g.stages; --use; }
            --s;
            ok = mbar_wait_warp(smem_u32(&sh.empty[s]), use & 1u, abort_flag);
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (one lane of the pair's first CTA)
        if (crank == 0) {
            const bool leader = elect_one();
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(g.bn >> 3) << 17) | ((uint32_t)(2 * TILE_F >> 4) << 24);
            const uint64_t desc0 = umma_desc(tiles0);
            int s = 0; uint32_t use = 0, seg = 0;
            bool ok = true;
            for (int it = pair; it < g.n_items && ok; it += n_pairs, ++seg) {
                const Item o = item_of(g, it);
                const uint32_t buf = seg & 1u;
                if (!mbar_wait_warp(smem_u32(&sh.tempty[buf]), ((seg >> 1) & 1u) ^ 1u, abort_flag)) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t d_tmem = tmem_base + buf * (uint32_t)g.bn;
                for (int kb = o.kb0; kb < o.kb1; ++kb) {
                    if (!mbar_wait_warp(smem_u32(&sh.full[s]), use & 1u, abort_flag)) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint64_t da = desc0 + (uint64_t)((uint32_t)s * (stage_bytes >> 4)), db = da + (W_BYTES >> 4);
                    if (leader) {
                        if (ST && it == pair && kb == o.kb0) stamp_pair(g.stamp, ST_DATA_FIRST);
#pragma unroll
                        for (uint32_t k = 0; k < TILE_K / 16; ++k)
                            umma_bf16_pair(d_tmem, da + 2 * k, db + 2 * k, idesc, (uint32_t)(kb != o.kb0) | k);
                        umma_commit_pair(smem_u32(&sh.empty[s]));
                    }
                    if (++s == g.stages) { s = 0; ++use; }
                }
                if (ok && leader) umma_commit_pair(smem_u32(&sh.tfull[buf]));
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue: thread = feature, columns = token rows
        const uint32_t quarter = (uint32_t)(warp & 3);
        const int et = (int)quarter * 32 + lane, grp = (warp - 2) >> 2;
        const uint32_t tempty0 = map_to_rank(smem_u32(&sh.tempty[0]), 0u);
        auto group_bar = [&]() { asm volatile("bar.sync %0, 128;" ::"r"(1 + grp) : "memory"); };
        float (*ex)[TILE_F] = sh.ex[grp];
        // Features `half` apart (a head's rotary pairs; gate and up) meet through shared memory: the lower one finishes a chunk's
        // first 16 token rows, the upper one the last 16.
        const int half = MODE == PF_QKV ? g.hd >> 1 : 64;
        const bool lower = (et & half) == 0;              // uniform in a warp
        uint32_t seg = 0;
        pdl_wait();                                       // outputs may still be read, and the row plan written, by kernels before
        for (int it = pair; it < g.n_items; it += n_pairs, ++seg) {
            const Item o = item_of(g, it);
            const uint32_t buf = seg & 1u;
            const int f0 = o.ft * 2 * TILE_F + (int)crank * TILE_F, n = f0 + et;
            const bool live = n < g.n_out;
            // what the rows bring along (1/rms; QKV: positions, cache rows, rotary factors) arrives under the MMAs, and for the
            // later chunks under the chunk before
            const int hd = MODE == PF_QKV ? g.hd : 128, head = n / hd, e = (et % hd) & (half - 1);
            const bool rot = MODE == PF_QKV && head < g.H + g.Hkv;
            constexpr int MY_CHUNKS = 256 / PF_CHUNK / PF_GROUPS;
            int my_pos[MY_CHUNKS], my_row[MY_CHUNKS];     // (row of the cache: kv head 0 of the row's slot)
            float cs[16], sn[16], sc[16];
            auto fetch_scale = [&](int c) {               // of the 16 rows this thread finishes in its group's chunk c
                const float4* p = reinterpret_cast<const float4*>(g.scale + o.tt * g.bn + min((c * PF_GROUPS + grp) * PF_CHUNK, g.bn - PF_CHUNK) + (lower ? 0 : 16));
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 v = __ldcg(p + i);
                    sc[4 * i] = v.x; sc[4 * i + 1] = v.y; sc[4 * i + 2] = v.z; sc[4 * i + 3] = v.w;
                }
            };
            auto fetch = [&](int p) {
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const int pos = max(__shfl_sync(0xffffffffu, p, i), 0);
                    cs[i] = rot ? __ldg(g.rcos + (size_t)pos * half + e) : 1.f;
                    sn[i] = rot ? __ldg(g.rsin + (size_t)pos * half + e) : 0.f;
                }
            };
            if (MODE != PF_PARTIAL) fetch_scale(0);
            if (MODE == PF_QKV) {
#pragma unroll
                for (int c = 0; c < MY_CHUNKS; ++c) {
                    const int c0 = (c * PF_GROUPS + grp) * PF_CHUNK, row = o.tt * g.bn + c0 + (lower ? 0 : 16) + (lane & 15);
                    const bool on = c0 < g.bn && row < g.rows;
                    my_pos[c] = on ? __ldcg(g.row_pos + row) : -1;
                    my_row[c] = on ? __ldcg(g.row_slot + row) * g.Hkv * g.max_ctx + my_pos[c] : -1;
                }
                fetch(my_pos[0]);
            }
            if (!mbar_wait(smem_u32(&sh.tfull[buf]), (seg >> 1) & 1u, abort_flag)) sh.epi_abort[grp] = 1;
            group_bar();
            if (sh.epi_abort[grp]) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t t_addr = tmem_base + ((quarter * 32u) << 16) + buf * (uint32_t)g.bn;
#pragma unroll
            for (int c = 0; c < MY_CHUNKS; ++c) {
                const int c0 = (c * PF_GROUPS + grp) * PF_CHUNK, t0 = o.tt * g.bn + c0;
                if (c0 >= g.bn || t0 >= g.rows) break;    // uniform
                uint32_t r[32];
                tmem_ld32(t_addr + (uint32_t)c0, r);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (LORA && o.piece == 0) add_lora(g, t0, n, live, r);
                if (MODE == PF_PARTIAL) {
                    float* dst = g.part + ((size_t)o.piece * g.rows + t0) * g.part_ld + (n - g.f_lo);
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (live && n >= g.f_lo && t0 + j < g.rows) __stcg(dst + (size_t)j * g.part_ld, __uint_as_float(r[j]));
                    continue;
                }
#pragma unroll
                for (int i = 0; i < 16; ++i) ex[i][et] = __uint_as_float(lower ? r[16 + i] : r[i]);
                group_bar();
                float mine[16], other[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) { mine[i] = __uint_as_float(lower ? r[i] : r[16 + i]) * sc[i]; other[i] = ex[i][et ^ half] * sc[i]; }
                if (c + 1 < MY_CHUNKS) fetch_scale(c + 1);
                group_bar();                              // the buffer may be written again
                const int tb = t0 + (lower ? 0 : 16);
                if (MODE == PF_SWIGLU) {
                    const int f = (f0 >> 1) + (et & 63);
                    __nv_bfloat162 w[8];                  // (shuffles and stores in loops of their own: interleaved they run one by one)
#pragma unroll
                    for (int i = 0; i < 16; i += 2) {     // two neighbouring lanes exchange token rows: each stores two adjacent features
                        float x[2];
#pragma unroll
                        for (int k = 0; k < 2; ++k) {
                            const float gt = lower ? mine[i + k] : other[i + k], up = lower ? other[i + k] : mine[i + k];
                            x[k] = gt / (1.f + expf(-gt)) * up;
                        }
                        const float got = __shfl_xor_sync(0xffffffffu, (lane & 1) ? x[0] : x[1], 1);
                        w[i / 2] = (lane & 1) ? __floats2bfloat162_rn(got, x[1]) : __floats2bfloat162_rn(x[0], got);
                    }
                    const int row = tb + (lane & 1);
                    bf16* dst = g.act + (size_t)row * g.F + (f & ~1);
#pragma unroll
                    for (int i = 0; i < 16; i += 2)
                        if (live && row + i < g.rows) *reinterpret_cast<__nv_bfloat162*>(dst + (size_t)i * g.F) = w[i / 2];
                } else {
                    // two neighbouring lanes exchange halves so that each stores two adjacent elements: the even lane of the
                    // rotated pair's first element, the odd lane of its second
                    __nv_bfloat162 w[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const float a = lower ? mine[i] : other[i], b = lower ? other[i] : mine[i];
                        const float ra = a * cs[i] - b * sn[i], rb = a * sn[i] + b * cs[i];
                        const float got = __shfl_xor_sync(0xffffffffu, (lane & 1) ? ra : rb, 1);
                        w[i] = (lane & 1) ? __floats2bfloat162_rn(got, rb) : __floats2bfloat162_rn(ra, got);
                    }
                    const int e2 = (e & ~1) + ((lane & 1) ? half : 0);
                    if (head < g.H) {
                        bf16* dst = g.q_out + ((size_t)tb * g.H + head) * hd + e2;
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (live && tb + i < g.rows) *reinterpret_cast<__nv_bfloat162*>(dst + (size_t)i * g.H * hd) = w[i];
                    } else {
                        bf16* dst = (rot ? g.kc : g.vc) + (size_t)((head - g.H) % g.Hkv) * g.max_ctx * hd + e2;
                        int at[16];
#pragma unroll
                        for (int i = 0; i < 16; ++i) at[i] = __shfl_sync(0xffffffffu, my_row[c], i);
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (live && at[i] >= 0) *reinterpret_cast<__nv_bfloat162*>(dst + (size_t)at[i] * hd) = w[i];
                    }
                    if (c + 1 < MY_CHUNKS) fetch(my_pos[c + 1]);
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(tempty0 + 8u * buf) : "memory");
        }
    }

    // ---------------------------------------------------------------------- wind-down
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (ST && threadIdx.x == 0) stamp_pair(g.stamp, ST_DONE_FIRST);
    if (sh.abort_flag) {
        if (threadIdx.x == 0 && status) atomicOr(status, SD_DEV_WAIT_EXPIRED);
        const uint64_t t0 = global_ns();                   // let copies in flight land before the CTA goes away
        while (global_ns() - t0 < 200000ull) __nanosleep(1000);
        __syncthreads();
    }
    cluster_sync_all();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
    }
}

// A row is spread over whole warps of one CTA, four float4 per thread: the last warp may hold as few as eight columns.
constexpr int NORM_VECS = 4;
int norm_threads(int d) { return (d + 4 * NORM_VECS * 32 - 1) / (4 * NORM_VECS * 32) * 32; }

// xn = bf16(v * gain) and 1/rms(v) for a row held in registers.
__device__ __forceinline__ void norm_row(const float4 (&v)[NORM_VECS], int d, const float* __restrict__ gain, float eps, bf16* __restrict__ xn,
                                         float* __restrict__ scale, float* red) {
    float ss = 0.f;
#pragma unroll
    for (int i = 0; i < NORM_VECS; ++i) {
        ss += v[i].x * v[i].x + v[i].y * v[i].y + v[i].z * v[i].z + v[i].w * v[i].w;
        const int k = 4 * (i * (int)blockDim.x + (int)threadIdx.x);
        if (k >= d) continue;
        const float4 w = __ldg(reinterpret_cast<const float4*>(gain + k));
        __nv_bfloat162 lo = __floats2bfloat162_rn(v[i].x * w.x, v[i].y * w.y), hi = __floats2bfloat162_rn(v[i].z * w.z, v[i].w * w.w);
        *reinterpret_cast<uint2*>(xn + k) = make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
    }
    ss = block_sum(ss, red);
    if (threadIdx.x == 0) *scale = rsqrtf(ss * (1.f / d) + eps);
}

__global__ void __launch_bounds__(512) k_pf_embed(SeqState S, const __grid_constant__ PrefillSegs segs, const bf16* __restrict__ embed, int d, int vocab,
                                                  const float* __restrict__ gain, float eps, float* __restrict__ h, bf16* __restrict__ xn,
                                                  float* __restrict__ scale, int32_t* __restrict__ row_slot, int32_t* __restrict__ row_pos,
                                                  int32_t* __restrict__ row_task) {
    __shared__ float red[32];
    const int r = blockIdx.x;
    int s = 0;
    while (s + 1 < segs.n && r >= segs.row0[s + 1]) ++s;
    const int slot = segs.slot[s], pos = segs.pos0[s] + (r - segs.row0[s]);
    int tok = S.tokens[(size_t)slot * S.tok_stride + pos];
    if (tok < 0 || tok >= vocab) { if (threadIdx.x == 0) atomicOr(S.status, SD_DEV_BAD_TOKEN); tok = 0; }
    if (threadIdx.x == 0) { row_slot[r] = slot; row_pos[r] = pos; row_task[r] = S.draft_id[slot]; }
    const bf16* e = embed + (size_t)tok * d;
    float4 v[NORM_VECS];
#pragma unroll
    for (int i = 0; i < NORM_VECS; ++i) {
        const int k = 4 * (i * (int)blockDim.x + (int)threadIdx.x);
        v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (k < d) {
            const uint2 raw = __ldg(reinterpret_cast<const uint2*>(e + k));
            const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.x)), b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.y));
            v[i] = make_float4(a.x, a.y, b.x, b.y);
            *reinterpret_cast<float4*>(h + (size_t)r * d + k) = v[i];
        }
    }
    norm_row(v, d, gain, eps, xn + (size_t)r * d, scale + r, red);
}

// Bound: L2 (reads h and the pieces, writes h and half of that again).
template <bool ST>
__global__ void __launch_bounds__(512) k_pf_norm(float* __restrict__ h, const float* __restrict__ part, int split, int rows, int d,
                                                 const float* __restrict__ gain, float eps, bf16* __restrict__ xn, float* __restrict__ scale,
                                                 unsigned long long* stamp) {
    __shared__ float red[32];
    pdl_launch_dependents();
    const int r = blockIdx.x;
    if (ST && threadIdx.x == 0) stamp_first(stamp, ST_START);
    pdl_wait();
    if (ST && threadIdx.x == 0) stamp_pair(stamp, ST_DEP_FIRST);
    float4 v[NORM_VECS];
#pragma unroll
    for (int i = 0; i < NORM_VECS; ++i) {
        const int k = 4 * (i * (int)blockDim.x + (int)threadIdx.x);
        v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (k < d) {
            v[i] = __ldcg(reinterpret_cast<const float4*>(h + (size_t)r * d + k));
            float4 a = __ldcg(reinterpret_cast<const float4*>(part + (size_t)r * d + k));
            for (int p = 1; p < split; ++p) {
                const float4 b = __ldcg(reinterpret_cast<const float4*>(part + ((size_t)p * rows + r) * d + k));
                a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
            }
            v[i].x += a.x; v[i].y += a.y; v[i].z += a.z; v[i].w += a.w;
            __stcg(reinterpret_cast<float4*>(h + (size_t)r * d + k), v[i]);
        }
    }
    norm_row(v, d, gain, eps, xn + (size_t)r * d, scale + r, red);
    if (ST && threadIdx.x == 0) stamp_pair(stamp, ST_DONE_FIRST);
}


// One CTA: 64 consecutive query rows of one run x one query head; a warp owns 16 rows.  The cache is walked in chunks of 64
// positions up to the block's last row, double-buffered by 16-byte asynchronous copies into an XOR-swizzled layout.
// Bound: latency of a block's chain of chunks; so only the chunks at a warp's diagonal are masked, and the output is scaled only when the
// largest score has grown (time a launch adds to a pass: 7B, 511 rows 27.1 -> 24.8 us; 1B, 1,289 rows of five sequences 24.2 -> 19.0).
template <int HD, bool ST>
__global__ void __launch_bounds__(128) k_pf_attention(const bf16* __restrict__ q, const bf16* __restrict__ kc, const bf16* __restrict__ vc, bf16* __restrict__ out,
                                                      const __grid_constant__ PrefillSegs segs, int H, int Hkv, int max_ctx, unsigned long long* stamp) {
    constexpr int CK = 64, ROWB = HD * 2, CPR = HD / 8, KS = HD / 16, NV = HD / 8, BUF = CK * ROWB;
    extern __shared__ __align__(128) uint8_t sm_raw[];
    pdl_launch_dependents();
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, gid = lane >> 2, tig = lane & 3;
    if (ST && t == 0) stamp_first(stamp, ST_START);
    const uint32_t smem0 = smem_u32(sm_raw);
    const int blk = (int)gridDim.x - 1 - (int)blockIdx.x, head = blockIdx.y;      // a run's last rows see the most positions: they start first
    int s = 0;
    while (s + 1 < segs.n && blk >= segs.blk0[s + 1]) ++s;
    const int j0 = (blk - segs.blk0[s]) * PF_QBLOCK;                              // rows of the run in front of this block
    const int n_run = segs.row0[s + 1] - segs.row0[s];
    const int r0 = segs.row0[s] + j0, nr = min(PF_QBLOCK, n_run - j0), p0 = segs.pos0[s] + j0;
    const int np = p0 + nr;                                                       // positions the block's last row sees
    const size_t head_off = ((size_t)segs.slot[s] * Hkv + head / (H / Hkv)) * max_ctx * HD;
    const bf16* K = kc + head_off;
    const bf16* V = vc + head_off;
    auto issue = [&](int c) {
        const int nk = min(CK, np - c * CK);
        const uint32_t kb = smem0 + (uint32_t)(c & 1) * 2u * BUF, vb = kb + BUF;
        for (int i = t; i < nk * CPR; i += 128) {
            const int key = i / CPR, ch = i % CPR;
            const uint32_t off = (uint32_t)key * ROWB + (uint32_t)((ch ^ (key & 7)) << 4);
            cp_async16(kb + off, K + (size_t)c * CK * HD + (size_t)i * 8);
            cp_async16(vb + off, V + (size_t)c * CK * HD + (size_t)i * 8);
        }
        for (int i = nk * CPR + t; i < CK * CPR; i += 128) {                      // value rows past the end must be finite (their weight is zero)
            const int key = i / CPR, ch = i % CPR;
            *reinterpret_cast<uint4*>(sm_raw + (size_t)(c & 1) * 2 * BUF + BUF + (size_t)key * ROWB + ((ch ^ (key & 7)) << 4)) = make_uint4(0, 0, 0, 0);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    pdl_wait();
    if (ST && t == 0) stamp_pair(stamp, ST_DEP_FIRST);
    issue(0);
    const int w0 = 16 * warp, i_lo = w0 + gid, i_hi = i_lo + 8;                   // this thread's two rows of the block
    const bool on_lo = i_lo < nr, on_hi = i_hi < nr;
    uint32_t a[KS][4];
    {
        const bf16* q_lo = q + ((size_t)(r0 + i_lo) * H + head) * HD;
        const bf16* q_hi = q + ((size_t)(r0 + i_hi) * H + head) * HD;
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
            a[ks][0] = on_lo ? __ldcg(reinterpret_cast<const uint32_t*>(q_lo + 16 * ks + 2 * tig)) : 0u;
            a[ks][1] = on_hi ? __ldcg(reinterpret_cast<const uint32_t*>(q_hi + 16 * ks + 2 * tig)) : 0u;
            a[ks][2] = on_lo ? __ldcg(reinterpret_cast<const uint32_t*>(q_lo + 16 * ks + 8 + 2 * tig)) : 0u;
            a[ks][3] = on_hi ? __ldcg(reinterpret_cast<const uint32_t*>(q_hi + 16 * ks + 8 + 2 * tig)) : 0u;
        }
    }
    const int pos_lo = on_lo ? p0 + i_lo : -1, pos_hi = on_hi ? p0 + i_hi : -1;
    const int last = w0 < nr ? p0 + min(w0 + 15, nr - 1) : -1;                    // last position the warp's rows see
    const float sl2 = rsqrtf((float)HD) * 1.4426950408889634f;                    // softmax scale in the exp2 domain
    float m_lo = -INFINITY, m_hi = -INFINITY, l_lo = 0.f, l_hi = 0.f;
    float O[NV][4];
#pragma unroll
    for (int i = 0; i < NV; ++i) { O[i][0] = O[i][1] = O[i][2] = O[i][3] = 0.f; }
    const int mi = lane >> 3, lr = lane & 7;
    const int n_chunks = (np + CK - 1) / CK;
    for (int c = 0; c < n_chunks; ++c) {
        if (c + 1 < n_chunks) { issue(c + 1); asm volatile("cp.async.wait_group 1;" ::: "memory"); }
        else asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        if (c * CK <= last) {
            const uint32_t kb = smem0 + (uint32_t)(c & 1) * 2u * BUF, vb = kb + BUF;
            float Sc[8][4];
#pragma unroll
            for (int i = 0; i < 8; ++i) { Sc[i][0] = Sc[i][1] = Sc[i][2] = Sc[i][3] = 0.f; }
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) {                                      // 16 keys
                const int key = 16 * nt + 8 * (mi >> 1) + lr;
                const uint32_t rowaddr = kb + (uint32_t)key * ROWB;
#pragma unroll
                for (int ks = 0; ks < KS; ++ks) {
                    uint32_t b[4];
                    ldmatrix_x4(rowaddr + (uint32_t)(((2 * ks + (mi & 1)) ^ (key & 7)) << 4), b);
                    mma_bf16(Sc[2 * nt], a[ks], b[0], b[1]);
                    mma_bf16(Sc[2 * nt + 1], a[ks], b[2], b[3]);
                }
            }
            float mx_lo = -INFINITY, mx_hi = -INFINITY;
            const int pb = c * CK + 2 * tig;
            auto scale = [&](auto masked) {                                       // (only the chunks that reach past the warp's first row need the mask)
#pragma unroll
                for (int nt = 0; nt < 8; ++nt)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int p = pb + 8 * nt + (e & 1);
                        const float v = !decltype(masked)::value || p <= ((e < 2) ? pos_lo : pos_hi) ? Sc[nt][e] * sl2 : -INFINITY;
                        Sc[nt][e] = v;
                        if (e < 2) mx_lo = fmaxf(mx_lo, v); else mx_hi = fmaxf(mx_hi, v);
                    }
            };
            if (c * CK + CK <= p0 + w0 + 1 && w0 + 16 <= nr) scale(std::false_type()); else scale(std::true_type());
            mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 1)); mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 2));
            mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 1)); mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 2));
            const float mn_lo = fmaxf(m_lo, mx_lo), mn_hi = fmaxf(m_hi, mx_hi);
            const bool grown = mn_lo > m_lo || mn_hi > m_hi;
            const float ref_lo = mn_lo == -INFINITY ? 0.f : mn_lo, ref_hi = mn_hi == -INFINITY ? 0.f : mn_hi;      // (nothing seen yet: any finite reference gives weights of zero)
            float s_lo = 0.f, s_hi = 0.f;
#pragma unroll
            for (int nt = 0; nt < 8; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float pr = exp2_ftz(Sc[nt][e] - (e < 2 ? ref_lo : ref_hi));
                    Sc[nt][e] = pr;
                    if (e < 2) s_lo += pr; else s_hi += pr;
                }
            if (__any_sync(0xffffffffu, grown)) {                                 // (once the largest score has been seen, nothing is scaled any more)
                const float c_lo = exp2_ftz(m_lo - ref_lo), c_hi = exp2_ftz(m_hi - ref_hi);
                l_lo *= c_lo; l_hi *= c_hi;
#pragma unroll
                for (int nv = 0; nv < NV; ++nv) { O[nv][0] *= c_lo; O[nv][1] *= c_lo; O[nv][2] *= c_hi; O[nv][3] *= c_hi; }
            }
            m_lo = mn_lo; m_hi = mn_hi;
            l_lo += s_lo; l_hi += s_hi;
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {                                      // 16 keys
                uint32_t pa[4];
                pa[0] = pack_bf16(Sc[2 * ks][0], Sc[2 * ks][1]); pa[1] = pack_bf16(Sc[2 * ks][2], Sc[2 * ks][3]);
                pa[2] = pack_bf16(Sc[2 * ks + 1][0], Sc[2 * ks + 1][1]); pa[3] = pack_bf16(Sc[2 * ks + 1][2], Sc[2 * ks + 1][3]);
                const int key = 16 * ks + 8 * (mi & 1) + lr;
                const uint32_t rowaddr = vb + (uint32_t)key * ROWB;
#pragma unroll
                for (int nv = 0; nv < NV; nv += 2) {
                    uint32_t v[4];
                    ldmatrix_x4_trans(rowaddr + (uint32_t)(((nv + (mi >> 1)) ^ (key & 7)) << 4), v);
                    mma_bf16(O[nv], pa, v[0], v[1]);
                    mma_bf16(O[nv + 1], pa, v[2], v[3]);
                }
            }
        }
        __syncthreads();                                                          // the buffer may be refilled from here on
    }
    l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 1); l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 2);
    l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 1); l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 2);
    const float inv_lo = l_lo > 0.f ? 1.f / l_lo : 0.f, inv_hi = l_hi > 0.f ? 1.f / l_hi : 0.f;
    uint32_t* o_lo = reinterpret_cast<uint32_t*>(out + ((size_t)(r0 + i_lo) * H + head) * HD + 2 * tig);
    uint32_t* o_hi = reinterpret_cast<uint32_t*>(out + ((size_t)(r0 + i_hi) * H + head) * HD + 2 * tig);
#pragma unroll
    for (int nv = 0; nv < NV; ++nv) {
        if (on_lo) o_lo[4 * nv] = pack_bf16(O[nv][0] * inv_lo, O[nv][1] * inv_lo);
        if (on_hi) o_hi[4 * nv] = pack_bf16(O[nv][2] * inv_hi, O[nv][3] * inv_hi);
    }
    if (ST && t == 0) stamp_pair(stamp, ST_DONE_FIRST);
}

}  // namespace

// The tile is the one whose waves of CTA pairs take the least time: measured per k block 0.2 us up to 64 columns, 0.25 at 128,
// 0.4 at 256 with all SMs at work, which the model below follows within a few per cent (7B and 1B shapes, 127...1289 rows: the
// pick is the fastest of all tiles or within 5 % of it).
PrefillGemm prefill_geometry(int mode, int rows, int n_out, int K, int n_sm, int max_part_rows, int ft0) {
    PrefillGemm g;
    memset(&g, 0, sizeof(g));
    g.mode = mode; g.rows = rows; g.n_out = n_out; g.K = K; g.ft0 = ft0; g.part_ld = n_out;
    g.n_ft = (n_out + 2 * TILE_F - 1) / (2 * TILE_F) - ft0;
    g.kb = (K + TILE_K - 1) / TILE_K;
    const int pairs = std::max(1, n_sm / 2);
    double best = 1e300;
    for (int bn = 32; bn <= 256; bn += 32) {
        const int tt = (rows + bn - 1) / bn;
        for (int split = 1; split <= (mode == PF_PARTIAL ? 4 : 1); ++split) {
            if (split > 1 && ((long long)split * rows > max_part_rows || g.kb / split < 8)) continue;
            const long long items = (long long)g.n_ft * tt * split;
            const long long waves = (items + pairs - 1) / pairs;
            // cycles of a k block: the MMAs (2 per column), the operands coming in at the rate a loaded L2 gives an SM, or the
            // waits, issue and commit
            const double t_kb = std::max(360.0, std::max(2.0 * bn, (W_BYTES + 64.0 * bn) / 64.0));
            const double t = (double)waves * ((g.kb + split - 1) / split) * t_kb + 12.0 * bn + 600.0 * (split - 1);      // epilogue; the norm kernel reads every piece
            if (t < best) { best = t; g.bn = bn; g.n_tt = tt; g.split = split; g.n_items = (int)items; }
        }
    }
    g.keep_w = g.n_tt > 1;
    g.stages = std::min(PF_MAX_STAGES, PF_RING / (W_BYTES + g.bn * 64));
    return g;
}

cudaError_t launch_prefill_gemm(const TensorMap& tm_w, const TensorMap& tm_x, const PrefillGemm& g, int n_sm, uint32_t* status, cudaStream_t st) {
    if (g.rows < 1 || g.n_ft < 1 || g.bn < 32 || g.bn > 256 || (g.bn & 31) || g.stages < 2 || g.split < 1 || (g.split > 1 && g.mode != PF_PARTIAL)) return cudaErrorInvalidValue;
    if (g.mode == PF_QKV && (g.hd != 64 && g.hd != 128)) return cudaErrorInvalidValue;
    if (g.mode == PF_SWIGLU && (g.F % 64)) return cudaErrorInvalidValue;
    if (g.lora_b && (g.lora_r < 8 || g.lora_r > 32 || (g.lora_r & 7) || g.lora_n * g.lora_r > 128)) return cudaErrorInvalidValue;
    typedef void (*Kernel)(const CUtensorMap, const CUtensorMap, const PrefillGemm, uint32_t*);
    static const Kernel kernels[2][2][3] = {{{k_pf_gemm<PF_QKV, false, false>, k_pf_gemm<PF_SWIGLU, false, false>, k_pf_gemm<PF_PARTIAL, false, false>},
                                             {k_pf_gemm<PF_QKV, true, false>, k_pf_gemm<PF_SWIGLU, true, false>, k_pf_gemm<PF_PARTIAL, true, false>}},
                                            {{k_pf_gemm<PF_QKV, false, true>, k_pf_gemm<PF_SWIGLU, false, true>, k_pf_gemm<PF_PARTIAL, false, true>},
                                             {k_pf_gemm<PF_QKV, true, true>, k_pf_gemm<PF_SWIGLU, true, true>, k_pf_gemm<PF_PARTIAL, true, true>}}};
    if (g.mode < 0 || g.mode > PF_PARTIAL) return cudaErrorInvalidValue;
    const Kernel kern = kernels[g.stamp ? 1 : 0][g.lora_b ? 1 : 0][g.mode];
    const size_t smem = (size_t)g.stages * (W_BYTES + g.bn * 64) + 1024;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, PF_RING + 1024);
    if (e != cudaSuccess) return e;
    const int pairs = std::min(std::max(1, n_sm / 2), g.n_items);
    return launch_pdl(kern, dim3(2 * pairs), dim3(PF_THREADS), smem, st, 1, *(const CUtensorMap*)&tm_w, *(const CUtensorMap*)&tm_x, g, status);
}

cudaError_t launch_prefill_embed(const SeqState& S, const PrefillSegs& segs, const bf16* embed, int d, int vocab, const float* gain, float eps,
                                 float* h, bf16* xn, float* scale, int32_t* row_slot, int32_t* row_pos, int32_t* row_task, cudaStream_t st) {
    if (norm_threads(d) > 512 || (d & 3)) return cudaErrorInvalidValue;
    k_pf_embed<<<segs.rows, norm_threads(d), 0, st>>>(S, segs, embed, d, vocab, gain, eps, h, xn, scale, row_slot, row_pos, row_task);
    return cudaGetLastError();
}

cudaError_t launch_prefill_norm(float* h, const float* part, int split, int rows, int d, const float* gain, float eps, bf16* xn, float* scale,
                                unsigned long long* stamp, cudaStream_t st) {
    if (norm_threads(d) > 512 || (d & 3)) return cudaErrorInvalidValue;
    return launch_pdl(stamp ? k_pf_norm<true> : k_pf_norm<false>, dim3(rows), dim3(norm_threads(d)), 0, st, 1, h, part, split, rows, d, gain, eps, xn, scale, stamp);
}

cudaError_t launch_prefill_attention(const bf16* q, const bf16* kc, const bf16* vc, bf16* out, const PrefillSegs& segs, int H, int Hkv, int hd,
                                     int max_ctx, unsigned long long* stamp, cudaStream_t st) {
    if (hd != 64 && hd != 128) return cudaErrorInvalidValue;
    void (*kern)(const bf16*, const bf16*, const bf16*, bf16*, const PrefillSegs, int, int, int, unsigned long long*) = hd == 128 ? (stamp ? k_pf_attention<128, true> : k_pf_attention<128, false>)
                                                                              : (stamp ? k_pf_attention<64, true> : k_pf_attention<64, false>);
    const int smem = 4 * 64 * hd * 2;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(kern, dim3(segs.blk0[segs.n], H), dim3(128), smem, st, 1, q, kc, vc, out, segs, H, Hkv, max_ctx, stamp);
}

}  // namespace sd
