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
// (verify step, us, this kernel / tiles: width 512: 130 rows 200 / 221, 160 rows 217 / 224, 182 rows 229 / 227, 208 rows 237 / 228;
// width 768: 78 rows 262 / 294, 96 rows 285 / 294, 104 rows 309 / 291)
__host__ __device__ constexpr int rg_tile_rows(int width) { return width <= 512 ? 176 : 96; }
// ... reductions of 2048 and more sooner, to the split-K tiles, where these exist (512 wide 121 rows 174.3 / 174.7, 130 rows 181.3 / 178.4, 156 rows 191.5 / 190; 768 wide 78 rows
// 254 / 254, 88 rows 262 / 227; a reduction of 2112, which has none, two layers: 130 rows 180.3 / 195.3 on whole tiles, 144 rows 193.6 / 209.3) ...
__host__ __device__ constexpr int rg_tile_rows_long(int width) { return width <= 512 ? 128 : 80; }
// ... and in the encoders, two of which run side by side on two streams and fill the SMs sooner (first tokens: width 512: 60 rows
// 497 / 560, 80 rows 531 / 526, 120 rows 651 / 582; width 768: 40 rows 527 / 527, 60 rows 561 / 524).
__host__ __device__ constexpr int rg_tile_rows_enc(int width) { return width <= 512 ? 72 : 40; }
// Up to here the LayerNorm in front runs inside the GEMM, on 16-row tiles; beyond it is a launch of its own (inside / in front: width 512,
// 130 rows 202 / 218; width 768, 104 rows 330 / 304).
__host__ __device__ constexpr int rg_ln_rows(int width) { return width <= 512 ? 144 : 80; }

// Rows of a tile (16 or 32) where a GEMM of the usual widths goes on here beyond those rows, with the weights as register fragments; 0: it does not.
// (LayerNorm in front, or none.)
int rg_frag_rows(int epi, int N, int K, int rows_ub, int n_sm, bool enc);
bool rg_supported(int epi, int N, int K, int lda, int rows_ub, bool cluster);
inline bool rg_ln_width(int K) { return K == 256 || K == 512 || K == 768; }    // widths that the LayerNorm prologue exists for
cudaError_t rg_init();           // once per handle, before the first launch
cudaError_t rg_launch(int epi, const RowsArgs& a, int rows_ub, int frag, bool cluster, bool pdl, cudaStream_t st);

}  // namespace sd
