// Interface of the prefill path (prefill.cu): many prompt rows of several sequences in one pass of a bf16 model.
#pragma once
#include "gemm_tc.h"
#include "kernels.h"

namespace sd {

constexpr int PF_MAX_ROWS = 2048;       // prompt rows of one pass
constexpr int PF_QBLOCK = 64;           // query rows per attention CTA

// The rows of a pass: runs of consecutive prompt positions of one sequence each, packed one after the other.
struct PrefillSegs {
    int n, rows;
    int row0[SD_MAX_BATCH + 1];         // first row of each run; row0[n] = rows
    int slot[SD_MAX_BATCH], pos0[SD_MAX_BATCH];
    int blk0[SD_MAX_BATCH + 1];         // first attention block of each run; blk0[n] = number of blocks
};

enum { PF_QKV = 0, PF_SWIGLU = 1, PF_PARTIAL = 2 };
struct PrefillGemm {
    int mode;
    int rows, n_out, K;                 // Y[rows][n_out] = X[rows][K] W[n_out][K]^T
    int bn;                             // token rows per tile
    int n_ft, ft0, n_tt;                // 256-feature tiles (the first one worked on is ft0), token tiles
    int kb, split;                      // 64-wide k blocks; pieces the reduction is cut into (PF_PARTIAL only)
    int n_items, stages;
    int keep_w;                         // several token tiles read a weight tile: leave it in L2
    const float* scale;                 // PF_QKV, PF_SWIGLU: 1/rms factor of each row (readable up to a multiple of 256 rows)
    // PF_QKV
    bf16* q_out; bf16* kc; bf16* vc; const int32_t* row_slot; const int32_t* row_pos;
    int H, Hkv, hd, max_ctx; const float* rcos; const float* rsin;      // [position][hd/2]
    // PF_SWIGLU
    bf16* act; int F;
    // PF_PARTIAL: part[piece][row][part_ld], features from f_lo on
    float* part; int part_ld, f_lo;
    unsigned long long* stamp;          // optional time stamps of the launch (see LaunchStamp)
    // Low-rank adapters (lora_b nullptr: none): lora_scale * sum_j t[row][task r + j] B[task][n][j] is added to output n (of the
    // first piece); t = X A^T comes from a launch of its own over the matrix's last 128 rows.
    const bf16* lora_b; const float* lora_t; const int32_t* lora_task; int lora_r, lora_n; float lora_scale;
};

// Picks tile and split; max_part_rows bounds split * rows (PF_PARTIAL).  ft0: features below 256 * ft0 are not computed.
PrefillGemm prefill_geometry(int mode, int rows, int n_out, int K, int n_sm, int max_part_rows, int ft0 = 0);
cudaError_t launch_prefill_gemm(const TensorMap& tm_w, const TensorMap& tm_x, const PrefillGemm& g, int n_sm, uint32_t* status, cudaStream_t st);
// Tokens of the rows -> h (fp32), xn = bf16(h * gain), scale = 1/rms(h), row_slot, row_pos, row_task.
cudaError_t launch_prefill_embed(const SeqState& S, const PrefillSegs& segs, const bf16* embed, int d, int vocab, const float* gain, float eps,
                                 float* h, bf16* xn, float* scale, int32_t* row_slot, int32_t* row_pos, int32_t* row_task, cudaStream_t st);
// h += sum of the pieces (in their order); xn = bf16(h * gain), scale = 1/rms(h).
cudaError_t launch_prefill_norm(float* h, const float* part, int split, int rows, int d, const float* gain, float eps, bf16* xn, float* scale,
                                unsigned long long* stamp, cudaStream_t st);
// Causal attention of the rows over their sequences' caches (the rows' own keys and values included).
cudaError_t launch_prefill_attention(const bf16* q, const bf16* kc, const bf16* vc, bf16* out, const PrefillSegs& segs, int H, int Hkv, int hd,
                                     int max_ctx, unsigned long long* stamp, cudaStream_t st);

}  // namespace sd
