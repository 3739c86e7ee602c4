// fp32 path (SPECDEC_DTYPE_F32): GEMM and attention for passes of few rows.  Both are bounded by latency -- an iteration of a small
// pair is a chain of some forty launches over kilobytes -- so, as in the bf16 path, everything that predates the
// predecessor (weights, page rows, cached keys) is requested before the dependency wait, the LayerNorm in front runs inside, K and V
// leave the QKV epilogue for the cache, and the work of a launch is spread over enough warps for one short round trip.
#include "barriers.cuh"
#include "rows_f32.cuh"
#include "attention.cuh"

namespace sd {

// ------------------------------------------------------------------ GEMM
// One CTA = 16 rows x BN columns, 256 threads = 4 slices of every K chunk x (8 row pairs x 8 column lanes); a thread owns rows
// rg, rg + 8 and columns c, c + 8, ...  The rows are resident, the weights pass through a ring of three 128-wide K chunks (small
// K: all of it requested before the wait).  FFMA from 16-byte shared loads; slices added in a fixed order.
constexpr int RF_BM = 16, RF_KC = 128, RF_NS = 3, RF_THREADS = 256;
static size_t rf_smem(int BN, int K) {
    const size_t ring = (size_t)RF_NS * BN * (RF_KC + 4) * 4, red = (size_t)4 * RF_BM * (BN + 4) * 4;
    return (size_t)RF_BM * (K + 4) * 4 + (ring > red ? ring : red);          // rows, weights
}

// LN > 0: the rows are LayerNorm(ln_x) of at most 32 LN elements, normalised in registers (two rows per warp).
template <int EPI, int BN, int LN>
__global__ void __launch_bounds__(RF_THREADS) k_rows_f32(RowsF32Args a) {
    constexpr int TN = BN / 8, RP = BN + 4, WP = RF_KC + 4;
    extern __shared__ __align__(16) float rf_sm[];
    __shared__ int s_kv[RF_BM];
    const GemmArgs<float>& g = a.g;
    const int K = g.K, N = g.N, AP = K + 4;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n0 = blockIdx.x * BN, m0 = blockIdx.y * RF_BM;
    const int R = min((g.rows_static >= 0 ? g.rows_static : *g.n_rows) - m0, RF_BM);
    if (R <= 0 && blockIdx.y > 0) return;
    float* As = rf_sm;
    float* Ws = As + RF_BM * AP;
    const int nch = (K + RF_KC - 1) / RF_KC;
    auto load_w = [&](int ch) {
        const int k0 = ch * RF_KC, kv4 = min(RF_KC, K - k0) >> 2;
        float* dst = Ws + (ch % RF_NS) * BN * WP;
        for (int i = tid; i < BN * (RF_KC / 4); i += RF_THREADS) {
            const int r = i / (RF_KC / 4), c = i % (RF_KC / 4);
            if (c >= kv4) continue;
            if (n0 + r < N) cp_async16(smem_u32(dst + r * WP + c * 4), g.W + (size_t)(n0 + r) * K + k0 + c * 4);
            else *reinterpret_cast<float4*>(dst + r * WP + c * 4) = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    pdl_launch_dependents();
    int issued = 0;
    for (; issued < min(nch, RF_NS); ++issued) load_w(issued);
    float gm[LN ? LN : 1], bt[LN ? LN : 1];
#pragma unroll
    for (int i = 0; i < LN; ++i) {
        gm[i] = lane + 32 * i < K ? ldg_pinned(a.ln_g + lane + 32 * i) : 0.f;
        bt[i] = lane + 32 * i < K ? ldg_pinned(a.ln_b + lane + 32 * i) : 0.f;
    }
    if (EPI == EPI_QKV && tid < RF_BM) s_kv[tid] = tid < R ? (int)g.pg.row(g.seq[m0 + tid], g.pos[m0 + tid]) : 0;
    // this thread's outputs: columns co + 16 i of row ro.  Their bias is a weight; fetched where it is added, it was a round trip at the end of every launch
    constexpr int PO = BN / 16;
    const int ro = tid >> 4, co = tid & 15;
    float bz[PO];
#pragma unroll
    for (int i = 0; i < PO; ++i) bz[i] = EPI != EPI_STATS && g.bias && n0 + co + 16 * i < N ? ldg_pinned(g.bias + n0 + co + 16 * i) : 0.f;
    pdl_wait();
    float ld = CUDART_INF_F;                           // EPI_STATS: the row's draft and its logit, requested with the rows
    int id = -1;
    if (EPI == EPI_STATS && ro < R) { if (g.ld) ld = g.ld[m0 + ro]; if (g.ld_id) id = g.ld_id[m0 + ro]; }
    if constexpr (LN > 0) {
        float x[2][LN], sum[2] = {0.f, 0.f}, mu[2], rs[2];
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int i = 0; i < LN; ++i) {
                const int m = warp + 8 * s, e = lane + 32 * i;
                x[s][i] = (m < R && e < K) ? a.ln_x[(size_t)(m0 + m) * K + e] : 0.f;
            }
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int i = 0; i < LN; ++i) sum[s] += x[s][i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { sum[0] += __shfl_xor_sync(0xffffffffu, sum[0], o); sum[1] += __shfl_xor_sync(0xffffffffu, sum[1], o); }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            mu[s] = sum[s] / K; sum[s] = 0.f;
#pragma unroll
            for (int i = 0; i < LN; ++i) if (lane + 32 * i < K) { const float c = x[s][i] - mu[s]; sum[s] += c * c; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { sum[0] += __shfl_xor_sync(0xffffffffu, sum[0], o); sum[1] += __shfl_xor_sync(0xffffffffu, sum[1], o); }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            rs[s] = 1.0f / sqrtf(sum[s] / K + a.ln_eps);
            const int m = warp + 8 * s;
#pragma unroll
            for (int i = 0; i < LN; ++i) {
                const int e = lane + 32 * i;
                if (e < K) {
                    const float y = (x[s][i] - mu[s]) * rs[s] * gm[i] + bt[i];
                    As[m * AP + e] = m < R ? y : 0.f;
                    if (g.ln_out && blockIdx.x == 0 && m < R) g.ln_out[(size_t)(m0 + m) * K + e] = y;
                }
            }
        }
    } else {
        const float* A = g.A + (size_t)m0 * g.lda;
        const int q = K >> 2;
        for (int r = warp; r < RF_BM; r += RF_THREADS / 32)
            for (int c = lane; c < q; c += 32) {
                if (r < R) cp_async16(smem_u32(As + r * AP + c * 4), A + (size_t)r * g.lda + c * 4);
                else *reinterpret_cast<float4*>(As + r * AP + c * 4) = make_float4(0.f, 0.f, 0.f, 0.f);
            }
    }
    float xo[PO];                                      // residual values
    if (EPI == EPI_RESID) {
#pragma unroll
        for (int i = 0; i < PO; ++i) xo[i] = (ro < R && n0 + co + 16 * i < N) ? g.resid[(size_t)(m0 + ro) * N + n0 + co + 16 * i] : 0.f;
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    const int sl = tid >> 6, c = tid & 7, rg = (tid >> 3) & 7;
    float acc[2][TN];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;
    for (int ch = 0; ch < nch; ++ch) {
        const int k0 = ch * RF_KC, ks = min(RF_KC, K - k0) >> 2;              // floats per slice (a multiple of 4)
        const float* w = Ws + (ch % RF_NS) * BN * WP + c * WP + sl * ks;
        const float* a0 = As + rg * AP + k0 + sl * ks;
        const float* a1 = a0 + 8 * AP;
#pragma unroll 2
        for (int k = 0; k < ks; k += 4) {
            const float4 x0 = *reinterpret_cast<const float4*>(a0 + k), x1 = *reinterpret_cast<const float4*>(a1 + k);
#pragma unroll
            for (int j = 0; j < TN; ++j) {
                const float4 y = *reinterpret_cast<const float4*>(w + j * 8 * WP + k);
                acc[0][j] = fmaf(x0.x, y.x, acc[0][j]); acc[0][j] = fmaf(x0.y, y.y, acc[0][j]);
                acc[0][j] = fmaf(x0.z, y.z, acc[0][j]); acc[0][j] = fmaf(x0.w, y.w, acc[0][j]);
                acc[1][j] = fmaf(x1.x, y.x, acc[1][j]); acc[1][j] = fmaf(x1.y, y.y, acc[1][j]);
                acc[1][j] = fmaf(x1.z, y.z, acc[1][j]); acc[1][j] = fmaf(x1.w, y.w, acc[1][j]);
            }
        }
        if (issued < nch) {                            // long K: the next chunk replaces the one just used
            __syncthreads();
            load_w(issued++);
            asm volatile("cp.async.commit_group;" ::: "memory");
            cp_wait_pending(issued - ch - 2 < 1 ? 0 : 1);
            __syncthreads();
        } else if (nch > RF_NS) {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();
        }
    }
    __syncthreads();                                   // the ring is dead: partial sums take its place
    float* red = Ws;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
        red[(sl * RF_BM + rg) * RP + c + 8 * j] = acc[0][j];
        red[(sl * RF_BM + rg + 8) * RP + c + 8 * j] = acc[1][j];
    }
    __syncthreads();
    float v[PO];
#pragma unroll
    for (int i = 0; i < PO; ++i) {
        const float* p = red + ro * RP + co + 16 * i;
        v[i] = (p[0] + p[RF_BM * RP]) + (p[2 * RF_BM * RP] + p[3 * RF_BM * RP]);
    }
    const int r = m0 + ro;
    if constexpr (EPI == EPI_STATS) {                  // the 16 threads of a row are half a warp
        const bool live = ro < R;
        RowPart p; p.mx = -CUDART_INF_F; p.arg = 0x7fffffff; p.sum = 0.f; p.cnt = 0;
#pragma unroll
        for (int i = 0; i < PO; ++i) {
            const int n = n0 + co + 16 * i;
            if (n >= N) { v[i] = -CUDART_INF_F; continue; }
            if (n == id) v[i] = ld;                    // the draft's column takes the pre-pass value
            if (v[i] > p.mx) { p.mx = v[i]; p.arg = n; }
            p.cnt += v[i] > ld ? 1 : 0;
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            RowPart q;
            q.mx = __shfl_xor_sync(0xffffffffu, p.mx, o);
            q.arg = __shfl_xor_sync(0xffffffffu, p.arg, o);
            q.cnt = __shfl_xor_sync(0xffffffffu, p.cnt, o);
            part_merge_nosum(p, q);
        }
        if (g.want_sum) {
            float s = 0.f;
#pragma unroll
            for (int i = 0; i < PO; ++i) if (n0 + co + 16 * i < N) s += expf(v[i] - p.mx);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            p.sum = s;
        }
        if (live && co == 0) g.part[(size_t)r * g.n_tiles + blockIdx.x] = p;
    } else {
        if (ro >= R) return;
#pragma unroll
        for (int i = 0; i < PO; ++i) {
            const int n = n0 + co + 16 * i;
            if (n >= N) continue;
            float y = v[i] + bz[i];
            if (EPI == EPI_RESID) { g.resid[(size_t)r * N + n] = xo[i] + y; continue; }
            if (EPI == EPI_RELU) y = ffn_act(y, g.act);
            float* o = g.out + (size_t)r * g.ldo + n;
            if (EPI == EPI_QKV && n >= g.kv_d) {
                const size_t row = (size_t)s_kv[ro] * g.kv_d;
                o = n < 2 * g.kv_d ? g.kc + row + (n - g.kv_d) : g.vc + row + (n - 2 * g.kv_d);
            }
            *o = y;
        }
    }
}

constexpr size_t RF_MAX_SMEM = 227 * 1024 - 1024;
// Beyond, the 64 x 64 tiles of k_gemm_simt share more per load (verify step of the Transformer-base shapes in fp32, both kernels here against
// k_gemm_simt and the warp-per-row attention: 26 rows 0.62 / 2.58 ms, 104 rows 0.94 / 2.73, 416 rows 2.55 / 3.58, 1664 rows 9.3 / 8.2).
constexpr int RF_MAX_ROWS = 768;
bool rf_supported(int epi, int N, int K, int lda, int rows_ub) {
    if (epi == EPI_F32 || K % 16 || lda % 4 || rows_ub > RF_MAX_ROWS) return false;
    return rf_smem(epi == EPI_STATS ? 64 : 32, K) <= RF_MAX_SMEM;
}
template <int EPI, int BN, int LN>
static cudaError_t rf_go(const RowsF32Args& a, int rows_ub, bool pdl, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((a.g.N + BN - 1) / BN, (rows_ub + RF_BM - 1) / RF_BM); cfg.blockDim = dim3(RF_THREADS);
    cfg.dynamicSmemBytes = rf_smem(BN, a.g.K); cfg.stream = st;        // (allowed by rf_init)
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k_rows_f32<EPI, BN, LN>, a);
}
template <int EPI, int BN>
static cudaError_t rf_ln(const RowsF32Args& a, int rows_ub, bool pdl, cudaStream_t st) {
    if (!a.ln_x) return rf_go<EPI, BN, 0>(a, rows_ub, pdl, st);
    return a.g.K <= 128 ? rf_go<EPI, BN, 4>(a, rows_ub, pdl, st) : rf_go<EPI, BN, 16>(a, rows_ub, pdl, st);
}
cudaError_t rf_launch(int epi, const RowsF32Args& a, int rows_ub, bool pdl, cudaStream_t st) {
    switch (epi) {
        case EPI_STORE: return rf_ln<EPI_STORE, 32>(a, rows_ub, pdl, st);
        case EPI_RELU: case EPI_GELU: return rf_ln<EPI_RELU, 32>(a, rows_ub, pdl, st);      // (activation chosen by g.act)
        case EPI_QKV: return rf_ln<EPI_QKV, 32>(a, rows_ub, pdl, st);
        case EPI_STATS: return rf_ln<EPI_STATS, 64>(a, rows_ub, pdl, st);
        default: return rf_go<EPI_RESID, 32, 0>(a, rows_ub, pdl, st);
    }
}

// ------------------------------------------------------------------ attention
// One CTA per (16 queries, head, sequence), 8 warps of two queries each.  K and V of every visible key sit in shared memory; a lane takes
// keys lane, lane + 32, ... for the scores and, for the output, four head columns of every 32 / (d_head / 4)-th key.
// Softmax with the true row maximum; the same terms as the warp-per-row kernel that serves the other head sizes.
constexpr int AF_Q = 16, AF_WARPS = 8;
static size_t af_smem(int dh, int max_keys) {
    const size_t mk = (size_t)((max_keys + 3) & ~3);
    return (mk * (dh + 4) * 2 + (size_t)AF_Q * dh + AF_Q * mk) * 4;
}

template <bool PAGED>
__global__ void __launch_bounds__(AF_WARPS * 32) k_attn_f32(AttnF32Args a) {
    extern __shared__ __align__(16) float af_sm[];
    const int b = a.seq_of ? a.seq_of[blockIdx.z] : (int)blockIdx.z, h = blockIdx.y, qt = blockIdx.x;
    if (b < 0) return;
    // (row metadata, page table and sequence lengths predate the step's kernel chain: readable before the wait)
    const int cnt = a.q_cnt[b], q_first = a.q_off[b];
    const int pre = a.pre_keys ? min(a.pre_keys[b], a.max_keys) : 0, kv0 = PAGED ? 0 : a.kv_off[b];
    pdl_launch_dependents();
    if (qt * AF_Q >= cnt) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, dh = a.d_head, KP = dh + 4, mk = (a.max_keys + 3) & ~3;
    const int r0 = q_first + qt * AF_Q, nq = min(AF_Q, cnt - qt * AF_Q);
    float* Ks = af_sm;
    float* Vs = Ks + mk * KP;
    float* Qs = Vs + mk * KP;
    float* P0 = Qs + AF_Q * dh + warp * 2 * mk;
    float* P1 = P0 + mk;
    const int q4 = dh >> 2;                              // a power of two up to 32
    const int sh = 31 - __clz(q4);
    auto load_keys = [&](int lo, int hi) {
        for (int i = (lo << sh) + tid; i < hi << sh; i += AF_WARPS * 32) {
            const int t = i >> sh, c = (i & (q4 - 1)) * 4;
            const size_t off = (PAGED ? a.pg.row(b, t) : (size_t)(kv0 + t)) * a.kv_stride + h * dh + c;
            cp_async16(smem_u32(Ks + t * KP + c), a.k + off);
            cp_async16(smem_u32(Vs + t * KP + c), a.v + off);
        }
    };
    load_keys(0, pre);
    int nk[2], nkmax = 0;
#pragma unroll
    for (int i = 0; i < 2; ++i) nk[i] = warp + AF_WARPS * i < nq ? min(a.nkeys[r0 + warp + AF_WARPS * i], a.max_keys) : 0;
    for (int r = lane; r < nq; r += 32) nkmax = max(nkmax, min(a.nkeys[r0 + r], a.max_keys));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nkmax = max(nkmax, __shfl_xor_sync(0xffffffffu, nkmax, o));
    // where this thread's first piece of the keys behind the wait lies: the page table predates the step, its round trip does not belong there
    const int first = min(pre, nkmax), i0 = (first << sh) + tid;
    const bool has = i0 < nkmax << sh;
    const size_t off0 = has ? (PAGED ? a.pg.row(b, i0 >> sh) : (size_t)(kv0 + (i0 >> sh))) * a.kv_stride + h * dh + (i0 & (q4 - 1)) * 4 : 0;
    pdl_wait();
    for (int i = tid; i < nq << sh; i += AF_WARPS * 32) {
        const int r = i >> sh, c = (i & (q4 - 1)) * 4;
        const size_t qr = a.q_index ? (size_t)a.q_index[r0 + r] : (size_t)(r0 + r);
        cp_async16(smem_u32(Qs + r * dh + c), a.q + qr * a.q_stride + h * dh + c);
    }
    if (has) {
        const uint32_t at = ((i0 >> sh) * KP + (i0 & (q4 - 1)) * 4) * 4;
        cp_async16(smem_u32(Ks) + at, a.k + off0);
        cp_async16(smem_u32(Vs) + at, a.v + off0);
    }
    load_keys(first + ((AF_WARPS * 32) >> sh), nkmax);  // (the others')
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (warp >= nq) return;
    const int n = max(nk[0], nk[1]);
    const float* qa = Qs + warp * dh;
    const float* qb = warp + AF_WARPS < nq ? qa + AF_WARPS * dh : qa;
    float m0 = -CUDART_INF_F, m1 = -CUDART_INF_F;
    for (int t = lane; t < n; t += 32) {
        const float* kp = Ks + t * KP;
        float s0 = 0.f, s1 = 0.f;
#pragma unroll 4
        for (int e = 0; e < dh; e += 4) {
            const float4 k4 = *reinterpret_cast<const float4*>(kp + e), x = *reinterpret_cast<const float4*>(qa + e), y = *reinterpret_cast<const float4*>(qb + e);
            s0 = fmaf(x.x, k4.x, s0); s0 = fmaf(x.y, k4.y, s0); s0 = fmaf(x.z, k4.z, s0); s0 = fmaf(x.w, k4.w, s0);
            s1 = fmaf(y.x, k4.x, s1); s1 = fmaf(y.y, k4.y, s1); s1 = fmaf(y.z, k4.z, s1); s1 = fmaf(y.w, k4.w, s1);
        }
        s0 = t < nk[0] ? s0 * a.scale : -CUDART_INF_F;
        s1 = t < nk[1] ? s1 * a.scale : -CUDART_INF_F;
        P0[t] = s0; P1[t] = s1;
        m0 = fmaxf(m0, s0); m1 = fmaxf(m1, s1);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) { m0 = fmaxf(m0, __shfl_xor_sync(0xffffffffu, m0, o)); m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, o)); }
    float l0 = 0.f, l1 = 0.f;
    for (int t = lane; t < n; t += 32) {                  // (a masked score is -inf and gives 0; a row without keys keeps sum 0)
        const float e0 = m0 == -CUDART_INF_F ? 0.f : expf(P0[t] - m0), e1 = m1 == -CUDART_INF_F ? 0.f : expf(P1[t] - m1);
        l0 += e0; l1 += e1;
        P0[t] = e0; P1[t] = e1;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) { l0 += __shfl_xor_sync(0xffffffffu, l0, o); l1 += __shfl_xor_sync(0xffffffffu, l1, o); }
    __syncwarp();
    const int c = (lane & (q4 - 1)) * 4, grp = lane >> sh, ng = 32 >> sh;
    float4 o0 = make_float4(0.f, 0.f, 0.f, 0.f), o1 = o0;
    for (int t = grp; t < n; t += ng) {
        const float4 v4 = *reinterpret_cast<const float4*>(Vs + t * KP + c);
        const float p0 = P0[t], p1 = P1[t];
        o0.x = fmaf(p0, v4.x, o0.x); o0.y = fmaf(p0, v4.y, o0.y); o0.z = fmaf(p0, v4.z, o0.z); o0.w = fmaf(p0, v4.w, o0.w);
        o1.x = fmaf(p1, v4.x, o1.x); o1.y = fmaf(p1, v4.y, o1.y); o1.z = fmaf(p1, v4.z, o1.z); o1.w = fmaf(p1, v4.w, o1.w);
    }
    for (int o = q4; o < 32; o <<= 1) {
        o0.x += __shfl_xor_sync(0xffffffffu, o0.x, o); o0.y += __shfl_xor_sync(0xffffffffu, o0.y, o);
        o0.z += __shfl_xor_sync(0xffffffffu, o0.z, o); o0.w += __shfl_xor_sync(0xffffffffu, o0.w, o);
        o1.x += __shfl_xor_sync(0xffffffffu, o1.x, o); o1.y += __shfl_xor_sync(0xffffffffu, o1.y, o);
        o1.z += __shfl_xor_sync(0xffffffffu, o1.z, o); o1.w += __shfl_xor_sync(0xffffffffu, o1.w, o);
    }
    if (grp == 0) {
        float* op = a.out + (size_t)(r0 + warp) * a.out_stride + h * dh + c;
        *reinterpret_cast<float4*>(op) = l0 > 0.f ? make_float4(o0.x / l0, o0.y / l0, o0.z / l0, o0.w / l0) : make_float4(0.f, 0.f, 0.f, 0.f);
        if (warp + AF_WARPS < nq)
            *reinterpret_cast<float4*>(op + (size_t)AF_WARPS * a.out_stride) = l1 > 0.f ? make_float4(o1.x / l1, o1.y / l1, o1.z / l1, o1.w / l1) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

bool af_supported(int d_head, int max_keys) {
    return d_head >= 4 && d_head <= 128 && (d_head & (d_head - 1)) == 0 && af_smem(d_head, max_keys) <= RF_MAX_SMEM;
}
cudaError_t af_launch(bool paged, const AttnF32Args& a, int q_ub, int n_heads, int slots, bool pdl, cudaStream_t st) {
    auto go = [&](auto* kernel) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((q_ub + AF_Q - 1) / AF_Q, n_heads, slots); cfg.blockDim = dim3(AF_WARPS * 32);
        cfg.dynamicSmemBytes = af_smem(a.d_head, a.max_keys); cfg.stream = st;      // (allowed by rf_init)
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr; cfg.numAttrs = pdl ? 1 : 0;
        return cudaLaunchKernelEx(&cfg, kernel, a);
    };
    return paged ? go(k_attn_f32<true>) : go(k_attn_f32<false>);
}

// Shared-memory limits of everything launched above: the same for every handle, since they belong to the kernels in the whole process.
cudaError_t rf_init() {
    cudaError_t e = cudaSuccess;
    auto room = [&](auto* kernel) { if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RF_MAX_SMEM); };
#define RF_ROOM(EPI, BN) room(k_rows_f32<EPI, BN, 0>); room(k_rows_f32<EPI, BN, 4>); room(k_rows_f32<EPI, BN, 16>)
    RF_ROOM(EPI_STORE, 32); RF_ROOM(EPI_RELU, 32); RF_ROOM(EPI_QKV, 32); RF_ROOM(EPI_STATS, 64);
#undef RF_ROOM
    room(k_rows_f32<EPI_RESID, 32, 0>);
    room(k_attn_f32<true>); room(k_attn_f32<false>);
    return e;
}

}  // namespace sd
