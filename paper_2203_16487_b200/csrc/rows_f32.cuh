// fp32 path: GEMM and attention for passes of few rows, see rows_f32.cu.
#pragma once
#include "kernels.cuh"

namespace sd {

struct RowsF32Args {
    GemmArgs<float> g;           // A unless ln_x is set; W, bias, N, K, n_rows and the epilogue fields
    const float* ln_x;           // LayerNorm prologue: rows [rows, K] ...
    const float* ln_g; const float* ln_b; float ln_eps;
};
inline bool rf_ln_width(int K) { return K <= 512; }          // widths that the LayerNorm prologue exists for
bool rf_supported(int epi, int N, int K, int lda, int rows_ub);
cudaError_t rf_init();           // once per handle, before the first launch of either kernel
cudaError_t rf_launch(int epi, const RowsF32Args& a, int rows_ub, bool pdl, cudaStream_t st);

struct AttnF32Args {
    const float* q; int q_stride; const int* q_index;    // query row r reads q + (q_index ? q_index[r] : r) * q_stride
    const float* k; const float* v; int kv_stride;       // contiguous: key t of sequence b at row kv_off[b] + t
    const int* kv_off;
    Paged pg;                                             // paged: row pg.row(b, t)
    const int* q_off; const int* q_cnt;                   // per sequence: first query row, number of query rows
    const int* seq_of;                                    // the sequence of grid slice z (-1: none), or null: slice z is sequence z
    const int* nkeys;                                     // per query row: visible keys (0..nkeys-1)
    const int* pre_keys;                                  // per sequence (or null): keys 0..pre-1 were written before this
                                                          // step began, so they may be fetched before the dependency wait
    float* out; int out_stride;
    int max_keys, d_head;                                 // upper bound on nkeys; head size
    float scale;
};
bool af_supported(int d_head, int max_keys);
cudaError_t af_launch(bool paged, const AttnF32Args& a, int q_ub, int n_heads, int slots, bool pdl, cudaStream_t st);

}  // namespace sd
