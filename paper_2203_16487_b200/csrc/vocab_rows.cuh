// Vocabulary projection of a few rows with the final LayerNorm inside:  per row of x, statistics of LN(x) E^T over one tile of 224 vocabulary columns,
//     x fp32 [R, 512], R <= 32, E bf16 [N, 512]; one tile per CTA, one CTA per SM (32768 columns: 147).
//
// Bound by the chain of one CTA, not by the 33 MB of E, most of which is requested ahead of the dependency wait: rows and LayerNorm 2.2 us (1.1 for up to 16
// rows), 32 MMAs of 112 clocks 1.8 to 2.6, the accumulators' way through shared memory 0.4, statistics 0.9; some CTAs begin a microsecond late, where a
// predecessor held the SM's shared memory.  As two launches the step paid another boundary, the normalised rows' way through memory, and one warp's walk over 112 columns of 32
// rows (2.1 us: an accumulator row belongs to a lane of one TMEM quadrant, so with few rows two warps of eight had all the work).  Here
//   * the eight epilogue warps normalise the rows themselves, in every CTA (52 KB of rows each), and write them to shared memory as the MMA wants them;
//   * the draft's logit of each row is computed under the MMAs (same sum in every CTA); its embedding row, behind a chain of three round trips, is on its way
//     under the LayerNorm (requested ahead of the dependency wait it kept late CTAs from their rows: 126.3 -> 125.8 us a step);
//   * the two warps that can read the accumulators hand them over through shared memory, and each of the eight takes 28 columns.
// Both launches 10.8 us, this one 8.3 to 8.9 (26 rows); verify step of 26 rows 128.2 -> 125.8, of 11 rows 118 -> 115.3, greedy pass over 16 sequences 5680 -> 5570.
#pragma once
#include "gemm_tc.cuh"

namespace sd {

constexpr int VR_BN = 224, VR_K = 512, VR_NKB = VR_K / TC_BK;
template <int AR> struct VrCfg {                                      // AR: rows that the operand tiles hold (the MMA reads on into what follows, for lanes that nobody reads)
    static constexpr int A_BYTES = AR * 128, STAGE = VR_BN * 128;
    static constexpr int FIT = (232448 - 1024 - 512 - VR_NKB * A_BYTES) / STAGE, STAGES = FIT > VR_NKB ? VR_NKB : FIT;
    static constexpr int SMEM = VR_NKB * A_BYTES + STAGES * STAGE + 1024;
    static constexpr int PITCH = VR_BN + 4;                            // floats per row of the accumulators on their way through shared memory
    static_assert(32 * PITCH * 4 + 8 * 32 * 16 <= STAGES * STAGE, "they reuse the ring");
    static_assert(VR_NKB * A_BYTES + STAGES * STAGE >= (VR_NKB - 1) * A_BYTES + 128 * 128, "the MMA's 128 rows stay inside");
};

struct VocabRowsArgs {
    const float* x; const float* ln_g; const float* ln_b; float eps;
    const bf16* E; int N;
    const int* n_rows; int rows_static;
    const int* draft; const int* slot_seq; int k;                      // verify: row slot (k + 1) + c checks draft c of the slot's sequence; draft null (or k = 0): no drafts
    float* ld; int* ld_id;                                             // the logit and id of every row's draft (+inf, -1: none) go here; null: the drafter's pass
    bf16* y;                                                           // the normalised rows, for whoever replays the projection
    RowPart* part;                                                     // [rows, tiles]
    int want_sum;                                                      // also accumulate sum exp(l - max)
};

template <int AR>
__global__ void __launch_bounds__(TC_THREADS, 1) k_vocab_rows(const __grid_constant__ CUtensorMap tmW, VocabRowsArgs a, int* err_word) {
    using C = VrCfg<AR>;
    constexpr int RW = AR / 8, NC = VR_K / 128;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_full[C::STAGES], bar_empty[C::STAGES], bar_rows, bar_acc;
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s;
    __shared__ float s_ld[32];
    __shared__ int s_id[32];
    const int R = min(a.rows_static >= 0 ? a.rows_static : *a.n_rows, AR);                    // (a device-side count predates the step's chain)
    const uint32_t At = (smem_u32(smem_raw) + 1023u) & ~1023u, ring = At + VR_NKB * C::A_BYTES;
    uint8_t* At_p = smem_raw + (At - smem_u32(smem_raw));
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31, n0 = blockIdx.x * VR_BN;
    if (threadIdx.x == 0) {
        abort_s = 0;
        for (int s = 0; s < C::STAGES; ++s) { mbar_init(smem_u32(&bar_full[s]), 1); mbar_init(smem_u32(&bar_empty[s]), 1); }
        mbar_init(smem_u32(&bar_rows), TC_EPI_WARPS);
        mbar_init(smem_u32(&bar_acc), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32(&tmem_base_s), 256);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_d = __shfl_sync(0xffffffffu, tmem_base_s, 0);
    volatile int* abort_flag = &abort_s;
    const uint32_t full0 = smem_u32(&bar_full[0]), empty0 = smem_u32(&bar_empty[0]);
    if (warp == 0) {
        for (int s = 0; s < C::STAGES; ++s)
            if (elect_one()) {
                mbar_expect_tx(full0 + 8 * s, C::STAGE);
                tma_load_2d(ring + s * C::STAGE, &tmW, s * TC_BK, n0, full0 + 8 * s);
            }
    }
    pdl_launch_dependents();
    if (warp == 0) {
        pdl_wait();                                                   // (the waits below are bounded: they begin when the rows are on their way)
        bool ok = true;
        for (int kb = C::STAGES; kb < VR_NKB && ok; ++kb) {
            const int s = kb % C::STAGES;
            ok = mbar_wait_warp(empty0 + 8 * s, (kb / C::STAGES - 1) & 1, abort_flag, err_word, 1);
            if (ok && elect_one()) {
                mbar_expect_tx(full0 + 8 * s, C::STAGE);
                tma_load_2d(ring + s * C::STAGE, &tmW, kb * TC_BK, n0, full0 + 8 * s);
            }
        }
    } else if (warp == 1) {
        pdl_wait();
        constexpr uint32_t idesc = umma_idesc_bf16(TC_BM, VR_BN);
        bool ok = mbar_wait_warp(smem_u32(&bar_rows), 0, abort_flag, err_word, 13);
        tc_fence_after();
        for (int kb = 0; kb < VR_NKB && ok; ++kb) {
            const int s = kb % C::STAGES;
            ok = mbar_wait_warp(full0 + 8 * s, (kb / C::STAGES) & 1, abort_flag, err_word, 2);
            if (ok && elect_one()) {
                const uint64_t ad = umma_desc_k_sw128(At + kb * C::A_BYTES), wd = umma_desc_k_sw128(ring + s * C::STAGE);
                umma_bf16(tmem_d, ad, wd, idesc, kb ? 1u : 0u);
                umma_bf16(tmem_d, ad + 2, wd + 2, idesc, 1u);
                umma_bf16(tmem_d, ad + 4, wd + 4, idesc, 1u);
                umma_bf16(tmem_d, ad + 6, wd + 6, idesc, 1u);
                umma_commit(empty0 + 8 * s);
            }
        }
        if (ok && elect_one()) umma_commit(smem_u32(&bar_acc));
    } else {
        const int e = warp - 2;
        // ---- rows e, e + 8, ...
        float4 gm[NC], bt[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            gm[c] = ldg_pinned(reinterpret_cast<const float4*>(a.ln_g + lane * 4 + c * 128));
            bt[c] = ldg_pinned(reinterpret_cast<const float4*>(a.ln_b + lane * 4 + c * 128));
        }
        int slot[RW];                                                  // (row metadata and drafts predate the step's kernel chain)
#pragma unroll
        for (int i = 0; i < RW; ++i) slot[i] = a.draft && e + 8 * i < R ? a.slot_seq[(e + 8 * i) / (a.k + 1)] : -1;
        pdl_wait();
        float4 v[RW][NC];
#pragma unroll
        for (int i = 0; i < RW; ++i)
#pragma unroll
            for (int c = 0; c < NC; ++c)
                v[i][c] = e + 8 * i < R ? *reinterpret_cast<const float4*>(a.x + (size_t)(e + 8 * i) * VR_K + lane * 4 + c * 128) : make_float4(0.f, 0.f, 0.f, 0.f);
        // the drafts' embedding rows, a chain of three round trips, are fetched under the LayerNorm: a CTA that begins late would wait for them ahead of its rows
        int tok[RW];
#pragma unroll
        for (int i = 0; i < RW; ++i) {
            const int c0 = (e + 8 * i) % (a.k + 1);
            tok[i] = slot[i] >= 0 && c0 < a.k ? ld_pinned(a.draft + (size_t)slot[i] * a.k + c0) : -1;
        }
        float s[RW];
#pragma unroll
        for (int i = 0; i < RW; ++i) {
            s[i] = 0.f;
#pragma unroll
            for (int c = 0; c < NC; ++c) s[i] += v[i][c].x + v[i][c].y + v[i][c].z + v[i][c].w;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int i = 0; i < RW; ++i) s[i] += __shfl_xor_sync(0xffffffffu, s[i], o);
#pragma unroll
        for (int i = 0; i < RW; ++i) {
            const float mu = s[i] / VR_K;
            s[i] = 0.f;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                v[i][c].x -= mu; v[i][c].y -= mu; v[i][c].z -= mu; v[i][c].w -= mu;
                s[i] += v[i][c].x * v[i][c].x + v[i][c].y * v[i][c].y + v[i][c].z * v[i][c].z + v[i][c].w * v[i][c].w;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int i = 0; i < RW; ++i) s[i] += __shfl_xor_sync(0xffffffffu, s[i], o);
        uint2 ev[RW][NC], pk[RW][NC];
#pragma unroll
        for (int i = 0; i < RW; ++i)
#pragma unroll
            for (int c = 0; c < NC; ++c) ev[i][c] = (unsigned)tok[i] < (unsigned)a.N ? ldg_pinned(reinterpret_cast<const uint2*>(a.E + (size_t)tok[i] * VR_K + lane * 4 + c * 128)) : make_uint2(0u, 0u);
#pragma unroll
        for (int i = 0; i < RW; ++i) {
            const float rstd = 1.0f / sqrtf(s[i] / VR_K + a.eps);
            const int r = e + 8 * i;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                __nv_bfloat162 p0 = __floats2bfloat162_rn(v[i][c].x * rstd * gm[c].x + bt[c].x, v[i][c].y * rstd * gm[c].y + bt[c].y);
                __nv_bfloat162 p1 = __floats2bfloat162_rn(v[i][c].z * rstd * gm[c].z + bt[c].z, v[i][c].w * rstd * gm[c].w + bt[c].w);
                pk[i][c] = make_uint2(*reinterpret_cast<uint32_t*>(&p0), *reinterpret_cast<uint32_t*>(&p1));
                // column 4 lane + 128 c: K block 2 c + lane / 16, 16-byte chunk (lane % 16) / 2 of its 128-byte row, XOR-swizzled by the row
                *reinterpret_cast<uint2*>(At_p + (2 * c + (lane >> 4)) * C::A_BYTES + r * 128 + ((((lane & 15) >> 1) ^ (r & 7)) << 4) + (lane & 1) * 8) = pk[i][c];
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bar_rows));
        // under the MMAs: the drafts' logits
        float dot[RW];
#pragma unroll
        for (int i = 0; i < RW; ++i) {
            const int r = e + 8 * i;
            dot[i] = 0.f;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                if (r == (int)blockIdx.x && r < R) *reinterpret_cast<uint2*>(a.y + (size_t)r * VR_K + lane * 4 + c * 128) = pk[i][c];      // (CTA r of the grid stores row r)
                const float2 f0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&pk[i][c].x)), f1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&pk[i][c].y));
                const float2 w0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&ev[i][c].x)), w1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&ev[i][c].y));
                dot[i] = fmaf(f0.x, w0.x, dot[i]); dot[i] = fmaf(f0.y, w0.y, dot[i]); dot[i] = fmaf(f1.x, w1.x, dot[i]); dot[i] = fmaf(f1.y, w1.y, dot[i]);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int i = 0; i < RW; ++i) dot[i] += __shfl_xor_sync(0xffffffffu, dot[i], o);
        if (lane == 0) {
#pragma unroll
            for (int i = 0; i < RW; ++i) {
                const int r = e + 8 * i;
                const bool ok = (unsigned)tok[i] < (unsigned)a.N, checks = slot[i] >= 0 && r % (a.k + 1) < a.k;
                const float l = !checks ? CUDART_INF_F : ok ? dot[i] : -CUDART_INF_F;
                const int id = !checks ? -1 : ok ? tok[i] : -2;
                s_ld[r] = l; s_id[r] = id;
                if (a.ld && r == (int)blockIdx.x && r < R) { a.ld[r] = l; a.ld_id[r] = id; }
            }
        }
        // ---- the accumulators: rows 0..31 are the lanes of quadrant 0, which two of the eight warps can read
        const bool live = mbar_wait(smem_u32(&bar_acc), 0, abort_flag, err_word, 3);
        tc_fence_after();
        float* acc = reinterpret_cast<float*>(At_p + VR_NKB * C::A_BYTES);       // (all operands have been read)
        RowPart* parts = reinterpret_cast<RowPart*>(acc + 32 * C::PITCH);
        if ((warp & 3) == 0 && __all_sync(0xffffffffu, live)) {
            constexpr int H = VR_BN / 2;
            const int half = e >> 2;
#pragma unroll
            for (int c = 0; c < H / 16; c += 4) {
                uint32_t vr[4][16];
#pragma unroll
                for (int u = 0; u < 4; ++u) if (c + u < H / 16) tmem_ld_issue<16>(tmem_d + half * H + (c + u) * 16, vr[u]);
#pragma unroll
                for (int u = 0; u < 4; ++u) if (c + u < H / 16) {
                    tmem_ld_done<16>(vr[u]);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        *reinterpret_cast<uint4*>(acc + lane * C::PITCH + half * H + (c + u) * 16 + j * 4) = make_uint4(vr[u][4 * j], vr[u][4 * j + 1], vr[u][4 * j + 2], vr[u][4 * j + 3]);
                }
            }
        }
        asm volatile("bar.sync 1, %0;" ::"n"(TC_EPI_WARPS * 32) : "memory");     // the eight epilogue warps only
        // ---- warp e: columns 28 e .. + 27, a row per lane
        constexpr int CW = VR_BN / TC_EPI_WARPS;
        const float ld = lane < AR ? s_ld[lane] : 0.f;
        const int id = lane < AR ? s_id[lane] : -1, nb = n0 + e * CW;
        float x[CW];
#pragma unroll
        for (int j = 0; j < CW; j += 4) {
            const float4 t = *reinterpret_cast<const float4*>(acc + lane * C::PITCH + e * CW + j);
            x[j] = t.x; x[j + 1] = t.y; x[j + 2] = t.z; x[j + 3] = t.w;
        }
        if (nb + CW > a.N || __any_sync(0xffffffffu, (unsigned)(id - nb) < (unsigned)CW)) {          // warp-uniform, rare
#pragma unroll
            for (int j = 0; j < CW; ++j) x[j] = nb + j >= a.N ? -CUDART_INF_F : nb + j == id ? ld : x[j];      // draft column: pre-pass value
        }
        // maximum, its lowest column and the count as separate short chains
        RowPart p;
        float m4[4] = {x[0], x[1], x[2], x[3]};
        int c4[4] = {0, 0, 0, 0}, a4[4];
#pragma unroll
        for (int j = 4; j < CW; ++j) m4[j & 3] = fmaxf(m4[j & 3], x[j]);
        p.mx = fmaxf(fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])), -CUDART_INF_F);      // (28 NaN columns lose every comparison of the merge)
#pragma unroll
        for (int u = 0; u < 4; ++u) a4[u] = CW;
#pragma unroll
        for (int j = CW - 1; j >= 0; --j) { c4[j & 3] += x[j] > ld ? 1 : 0; a4[j & 3] = x[j] == p.mx ? j : a4[j & 3]; }
        const int at = min(min(a4[0], a4[1]), min(a4[2], a4[3]));
        p.arg = at < CW && p.mx > -CUDART_INF_F ? nb + at : 0x7fffffff;
        p.cnt = (c4[0] + c4[1]) + (c4[2] + c4[3]);
        p.sum = 0.f;
        if (a.want_sum) {
#pragma unroll 1
            for (int j = 0; j < CW; ++j)
                if (nb + j < a.N) p.sum += expf((nb + j == id ? ld : acc[lane * C::PITCH + e * CW + j]) - p.mx);
        }
        parts[e * 32 + lane] = p;
        asm volatile("bar.sync 1, %0;" ::"n"(TC_EPI_WARPS * 32) : "memory");
        if (e == 0 && lane < R) {
            RowPart q[TC_EPI_WARPS];
#pragma unroll
            for (int w = 0; w < TC_EPI_WARPS; ++w) q[w] = parts[w * 32 + lane];
            if (a.want_sum) {
#pragma unroll 1
                for (int w = 1; w < TC_EPI_WARPS; ++w) part_merge(q[0], parts[w * 32 + lane]);
            } else {
#pragma unroll
                for (int o = TC_EPI_WARPS / 2; o > 0; o >>= 1)
#pragma unroll
                    for (int w = 0; w < o; ++w) part_merge_nosum(q[w], q[w + o]);
            }
            a.part[(size_t)lane * gridDim.x + blockIdx.x] = q[0];
        }
        tc_fence_before();
    }
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_d, 256);
}

// Where this kernel is used: widths and vocabularies whose 224-column tiles are one wave, and few enough rows that every CTA can normalise them all and
// each row has a CTA that stores it (a device of a few SMs would have fewer tiles than rows).
constexpr int VR_MAX_ROWS = 32;
inline bool vr_supported(const TmaEncoder& enc, int N, int K, int rows_ub) {
    const int tiles = (N + VR_BN - 1) / VR_BN;
    return enc.ready && K == VR_K && rows_ub <= VR_MAX_ROWS && (N + 127) / 128 > enc.n_sm && tiles <= enc.n_sm && tiles >= rows_ub;
}
inline cudaError_t vr_init() {
    const cudaError_t e = cudaFuncSetAttribute(k_vocab_rows<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, VrCfg<16>::SMEM);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(k_vocab_rows<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, VrCfg<32>::SMEM);
}
inline int vr_launch(TmaEncoder& enc, const VocabRowsArgs& a, int rows_ub, cudaStream_t st) {
    CUtensorMap tw;
    if (!enc.get(tw, a.E, a.N, VR_K, VR_K, VR_BN)) return -1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((a.N + VR_BN - 1) / VR_BN); cfg.blockDim = dim3(TC_THREADS); cfg.stream = st;
    cfg.dynamicSmemBytes = rows_ub <= 16 ? VrCfg<16>::SMEM : VrCfg<32>::SMEM;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = enc.pdl ? 1 : 0;
    cudaError_t e = cudaLaunchKernelEx(&cfg, rows_ub <= 16 ? k_vocab_rows<16> : k_vocab_rows<32>, tw, a, enc.err_word);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) { enc.err = std::string("launch (vocabulary projection of few rows): ") + cudaGetErrorString(e); return -1; }
    return 0;
}

}  // namespace sd
