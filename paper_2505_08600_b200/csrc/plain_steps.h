// Interface of the fp32 few-rows layer kernels (plain_steps.cu).
#pragma once
#include "kernels.h"

namespace sd {

constexpr int PS_MAX_ROWS = 8;
enum { PS_QKV = 0, PS_RESIDUAL = 1, PS_GU = 2, PS_LM = 3 };
struct PlainStep {
    int mode, rows, n_out, K;
    const float* w;                     // [n_out][K]
    const float* x;                     // [rows][K]: residual stream (PS_QKV, PS_GU, PS_LM: normed on the way in) or the step's input
    const float* gain; float eps;       // of the norm
    int row_stride, row_offset;         // PS_LM: output row i is token row i * row_stride + row_offset
    float* y;                           // PS_RESIDUAL: [rows][n_out], added to; PS_GU: [rows][F]; PS_LM: [rows][n_out]
    int F;                              // PS_GU: gate rows, then up rows
    // PS_QKV: rotary embedding, query buffer, cache append
    float* q; float* kc; float* vc; const int32_t* row_slot; const int32_t* row_pos;
    int H, Hkv, hd, max_ctx; const float* rcos; const float* rsin;      // [position][hd/2]
};
// Whether a model's passes of `rows` rows run on these kernels.
bool plain_steps_fit(const sd_model_desc& m, int rows, int max_ctx);
cudaError_t launch_plain_step(const PlainStep& p, cudaStream_t st);
cudaError_t launch_plain_attention(const float* q, const float* kc, const float* vc, float* out, const int32_t* row_slot, const int32_t* row_pos, int n_rows,
                                   int H, int Hkv, int hd, int max_ctx, cudaStream_t st);

}  // namespace sd
