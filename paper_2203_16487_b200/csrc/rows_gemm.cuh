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

// Row limits, by the width of the model (the smaller side of a weight matrix).  Every CTA reads all of its operands from L2 once, so the
// traffic grows with rows x columns, while a tensor-core tile of 128 rows shares its weights among them.
constexpr int RG_MAX_ROWS = 384;                             // in general; shapes that the tensor-core tiles serve too go over to them at
// (verify step, us, this kernel / tiles: width 512: 104 rows 191 / 241, 208 rows 238 / 253, 260 rows 295 / 294, 364 rows 343 / 298;
// width 768: 78 rows 272 / 298, 104 rows 304 / 306, 156 rows 363 / 342)
__host__ __device__ constexpr int rg_tile_rows(int width) { return width <= 512 ? 256 : 112; }
// ... and in the encoders, two of which run side by side on two streams and fill the SMs sooner (first tokens: width 512: 60 rows
// 497 / 560, 180 rows 650 / 656, 240 rows 684 / 684; width 768: 60 rows 577 / 543).
__host__ __device__ constexpr int rg_tile_rows_enc(int width) { return width <= 512 ? 208 : 48; }
// Up to here the LayerNorm in front runs inside the GEMM, on 16-row tiles; beyond it is a launch of its own (inside / in front: width 512,
// 130 rows 202 / 218; width 768, 104 rows 330 / 304).
__host__ __device__ constexpr int rg_ln_rows(int width) { return width <= 512 ? 144 : 80; }

bool rg_supported(int epi, int N, int K, int lda, int rows_ub, bool cluster);
inline bool rg_ln_width(int K) { return K == 256 || K == 512 || K == 768; }    // widths that the LayerNorm prologue exists for
cudaError_t rg_launch(int epi, const RowsArgs& a, int rows_ub, bool cluster, bool pdl, cudaStream_t st);

}  // namespace sd
