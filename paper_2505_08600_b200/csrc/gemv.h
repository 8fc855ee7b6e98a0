// Interface of the few-rows matrix kernel with the following step fused in (gemv.cu).
#pragma once
#include "gemm_tc.h"

namespace sd {

constexpr int GEMV_MAX_ROWS = 16;
constexpr int GEMV_SSQ_STRIDE = 512;    // floats per token row of the sums of squares that EPI_RESIDUAL leaves, one per 16-feature tile

struct Gemv {
    const bf16* w;                      // [n_out][K]
    const bf16* x;                      // [rows][K], second parts ep.lo_off rows further down
    int rows, n_out, K;
    const float* lora_t;                // [row][128]: x A^T of all adapters (with ep.lora_b)
    Epilogue ep;                        // as for launch_fused_step; rs.n_parts counts this kernel's 16-feature tiles where it wrote them
};
bool gemv_supported(const Gemv& g);
// dependent = 0 for the kernel that follows the one that wrote the row plan (which is read ahead of the wait).
cudaError_t launch_gemv(const Gemv& g, int dependent, cudaStream_t st);

}  // namespace sd
