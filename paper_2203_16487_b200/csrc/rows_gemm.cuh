// GEMM for passes of few activation rows:  C[r, n] = sum_k A[r, k] W[n, k]  (bf16 operands, fp32 accumulation), see rows_gemm.cu.
#pragma once
#include "kernels.cuh"

namespace sd {

struct RowsArgs {
    GemmArgs<bf16> g;            // A (bf16 rows) unless ln_x is set; W, bias, N, K, n_rows and the epilogue fields
    const float* ln_x;           // LayerNorm prologue: fp32 rows [rows, K] ...
    const float* ln_g; const float* ln_b; float ln_eps;
    long long* trace;            // optional: CTA 0 records %globaltimer at a few points (debugging aid)
    int* err_word;               // raised when a bounded wait gives up
};

// Up to here this kernel beats the 128-row tensor-core tiles (verify step, us, before / after: 26 rows 220 / 178, 52 rows 310 / 186, 104 rows
// 346 / 211, 208 rows 363 / 278, 312 rows 373 / 339, 364 rows 378 / 354; 416 rows 381 / 389).  Every CTA reads all of its
// operands from L2 once, so the traffic grows with rows x columns while a tile of 128 rows shares its weights.
constexpr int RG_MAX_ROWS = 384;
// The two encoders run side by side on two streams and fill the SMs sooner (time to the first tokens: 160 rows 757 / 683, 320 rows 828 / 856).
constexpr int RG_MAX_ROWS_ENC = 208;
// Up to here the LayerNorm in front runs inside the GEMM (16-row tiles; 130 rows 260 / 232), beyond it is a launch of its own (156 rows 264 / 274).
constexpr int RG_LN_ROWS = 144;

bool rg_supported(int epi, int N, int K, int lda, int rows_ub, bool cluster);
inline bool rg_ln_width(int K) { return K == 256 || K == 512 || K == 768; }    // widths that the LayerNorm prologue exists for
cudaError_t rg_launch(int epi, const RowsArgs& a, int rows_ub, bool cluster, bool pdl, cudaStream_t st);

}  // namespace sd
