// Interface of the draft layers in two kernels (draft_layer.cu).
#pragma once
#include "gemm_tc.h"

namespace sd {

constexpr int DL_MAX_ROWS = 8;          // token rows of a pass

struct DraftLayer {
    // row plan: what the embedding kernel would work out, worked out by every kernel for itself
    SeqState S;
    int n_seq, rows_per_seq;            // rows_per_seq 2: PLAN_DRAFT_FIRST, 1: PLAN_DRAFT_NEXT
    int ids[DL_MAX_ROWS], out[DL_MAX_ROWS];
    int step, gamma; const int32_t* x;  // PLAN_DRAFT_NEXT: token of row i is x[out[i]][step - 1]
    const bf16* embed; int vocab;       // non-null: the residual stream begins here (first layer)
    int d, n_heads, F, max_ctx;
    float eps;
    const bf16* w_in; const bf16* w_out;        // QKV and Wo, or gate/up and down
    const float* gain;                          // of the norm in front of w_in
    // Residual stream [DL_MAX_ROWS][d]: h_in plus the n_in pieces [piece][DL_MAX_ROWS][d] that the kernel before left; the sum goes to h_out.
    const float* h_in; const float* part_in; int n_in; float* h_out;
    float* part_out;                            // this kernel's pieces: one per head, or draft_layer_pieces()
    bf16* kc; bf16* vc; const float* rcos; const float* rsin;      // attention: the layer's cache, rotary factors [position][32]
    unsigned long long* stamp;
};

// Whether the layers of a bf16 model run on these kernels for `rows` rows.
bool draft_layer_fits(const sd_model_desc& m, int rows);
int draft_layer_pieces(const sd_model_desc& m);                 // that the feed-forward kernel leaves
size_t draft_layer_scratch(const sd_model_desc& m);             // bytes: two residual streams and the pieces of both kernels
// dependent = 0 for the first kernel of a pass: it begins when everything before it has finished, and later ones after it did.
cudaError_t launch_draft_attention(const DraftLayer& p, int dependent, cudaStream_t st);
cudaError_t launch_draft_mlp(const DraftLayer& p, cudaStream_t st);
// h_in + pieces -> xn = h * gain in two bf16 parts (the second lo_off rows further down) and the rows' sums of squares, a piece per 256 columns.
constexpr int DL_TAIL = 256;
cudaError_t launch_draft_tail(const DraftLayer& p, bf16* xn, int lo_off, float* ssq, int ssq_stride, cudaStream_t st);

}  // namespace sd
