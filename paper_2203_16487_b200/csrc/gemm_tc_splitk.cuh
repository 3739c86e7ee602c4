// Residual GEMM over a few 128-row tiles with a long reduction (FFN2: K = 4 d), split along K inside a cluster:
//     resid[r, n] += x[r, :] . W[n, :] + bias[n],   x bf16 [R, K], W bf16 [N, K], resid fp32 [R, N],
// for row counts whose tiles x N / 64 (or N / 128) x SPLIT CTAs still fit one wave.
//
// Bound by the serial walk over K: with 64-wide column tiles there are N / 64 CTAs per row tile (8 for d = 512), and 32 k-blocks at 0.2 us are two thirds
// of the launch (9.4 us).  Here SPLIT CTAs of a cluster take a K slice of one tile each and then an equal share of its rows: every epilogue warp copies its
// 32 x 32 block of partial sums to the rows' owner (one 4 KB bulk copy, counted on the owner's mbarrier), which adds the slices in rank order -- fixed,
// so the result does not depend on timing -- then bias and residual.  Everybody finishes 128 / SPLIT rows; with one CTA collecting all
// partial tiles from 16-byte remote stores the exchange cost more than the walk it saved (11.4 us).  Verify step, unsplit / split:
// 286 rows at 512 columns 290 / 269 us, 494 rows 300 / 282, 832 rows 328 / 316; 208 rows at 768 columns 367 / 325.
#pragma once
#include "gemm_tc.cuh"

namespace sd {

// AR = rows of a tile.  Of a 64-row box the MMA reads 64 rows more, which are the stage's weights, into accumulator lanes that nobody reads.
template <int AR, int BN> struct SpkCfg {
    static constexpr int STAGES = BN == 128 ? 5 : AR == 128 ? 7 : 8;           // ring depth: the receive buffer takes the rest of shared memory
    static constexpr int A_KB = AR * TC_BK * 2, STAGE = A_KB + BN * TC_BK * 2;
    static constexpr int RECV = AR * BN * 4;               // SPLIT slices of AR / SPLIT rows
    static constexpr int SMEM = STAGES * STAGE + RECV + 1024;
    static_assert(STAGES * STAGE >= TC_EPI_WARPS * (BN / 64) * 4096, "the outgoing blocks reuse the ring");
    static_assert(AR == 128 || AR + BN >= 128, "the 128-row MMA read stays inside the stage");
};

// CTAs per tile: 4 while all clusters run at once, else 2, else none (0).  Shorter reductions gain less than the exchange costs (verify step, us, unsplit / split:
// K = 768 in four 208 rows 318 / 310, in two 520 rows 399 / 403; K = 512 416 rows 279 / 286).  (Clusters of 4 do not use every SM: 36 of them on 148 SMs took two waves,
// 392 us a verify
// step of 312 rows at 768 columns where clusters of 2 take 361.)
// 64-row tiles while their clusters run at once, too: half of the activations to fetch behind the wait (182 rows 197 -> 194.5, 234 rows 208.8 -> 204.5, 104 rows at 768 columns
// 258 -> 250), unless another stream's kernels share the SMs (two encoders over 144 rows 307 -> 315).
// Where two slices of 64-column tiles are more clusters than run at once, two of 128 columns, up to twice the rows: unsplit these are at most 72 CTAs that walk the whole K
// (verify step of 1248 rows, us, unsplit / split: 354.4 / 348.2, 1408 rows 387 / 379, 1664 rows 385 / 379, 2048 rows 426 / 420; drafts over 2160 rows 137.4 / 134.5).  Beside
// another stream's kernels (encoders) the unsplit ones stay, and for reductions that gain less than the exchange costs (two layers, 512 columns, verify / draft step of 1248 and of 2080 rows:
// K = 1024 287.2 / 295.3, 291 / 299 and 323 / 330, 325.5 / 334.4; 1536 300 / 300.5, 302 / 304.8 and 339 / 341, 341 / 346; 1664 302 / 302, 307 / 308 and 348 / 349.5, 351.4 / 352.5;
// 1792 308 / 305, 309.6 / 310.8 and 352 / 350, 354 / 355.3; 1024-wide output projections of 1040 rows 402 / 415, 408.5 / 423).
struct SpkPlan { int split, rows, cols; };
inline SpkPlan spk_plan(const TmaEncoder& enc, int N, int K, int rows_ub, bool shared) {
    if (N % 64 || K < 768) return {0, 0, 0};
    const long long n = N / 64, m = (rows_ub + TC_BM - 1) / TC_BM;
    if (K % (4 * TC_BK) == 0 && !shared && (rows_ub + 63) / 64 * n <= enc.spk_clusters4_64) return {4, 64, 64};
    if (K % (4 * TC_BK) == 0 && m * n <= enc.spk_clusters4) return {4, TC_BM, 64};
    if (K % (2 * TC_BK) || K < 1024) return {0, 0, 0};
    if (m * n <= enc.spk_clusters2) return {2, TC_BM, 64};
    return {!shared && K >= 1792 && N % 128 == 0 && m * (N / 128) <= enc.spk_clusters2_128 ? 2 : 0, TC_BM, 128};
}

template <int SPLIT, int AR, int BN>
__global__ void __launch_bounds__(TC_THREADS, 1)
k_gemm_tc_splitk(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW, GemmArgs<bf16> g, int* err_word) {
    using C = SpkCfg<AR, BN>;
    constexpr int NB = BN / 64;                                // 64-column blocks, one after the other in the outgoing and the receive buffer
    constexpr int SPK_STAGES = C::STAGES, SPK_A_KB = C::A_KB, SPK_STAGE = C::STAGE, SPK_RECV = C::RECV;
    constexpr int OWN = AR / SPLIT, RB = OWN < 32 ? OWN : 32;  // rows that a CTA finishes; rows that a warp sends to one owner
    static_assert(OWN % 16 == 0, "rows of 16 threads");
    const int m0 = blockIdx.y * AR, R = g.rows_static >= 0 ? g.rows_static : *g.n_rows;     // (a device-side count predates the step's chain)
    if (m0 >= R && m0 > 0) return;                             // the whole cluster leaves; the first row tile always waits for the predecessor
    const int nkb = g.K / TC_BK / SPLIT;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_full[SPK_STAGES], bar_empty[SPK_STAGES], bar_acc, bar_part;
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s;
    const uint32_t ring = (smem_u32(smem_raw) + 1023u) & ~1023u, recv = ring + SPK_STAGES * SPK_STAGE;
    uint8_t* ring_p = smem_raw + (ring - smem_u32(smem_raw));
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    uint32_t rank;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int n0 = (int)(blockIdx.x / SPLIT) * BN, kb0 = (int)rank * nkb;

    if (threadIdx.x == 0) {
        abort_s = 0;
        for (int s = 0; s < SPK_STAGES; ++s) { mbar_init(smem_u32(&bar_full[s]), 1); mbar_init(smem_u32(&bar_empty[s]), 1); }
        mbar_init(smem_u32(&bar_acc), 1);
        mbar_init(smem_u32(&bar_part), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(smem_u32(&bar_part), SPK_RECV);
    }
    if (warp == 1) tmem_alloc(smem_u32(&tmem_base_s), BN);
    tc_fence_before();
    tc_cluster_sync();                                         // every CTA's barriers exist before anybody sends
    tc_fence_after();
    const uint32_t tmem_d = __shfl_sync(0xffffffffu, tmem_base_s, 0);
    volatile int* abort_flag = &abort_s;
    const uint32_t full0 = smem_u32(&bar_full[0]), empty0 = smem_u32(&bar_empty[0]);
    const int pre = min(SPK_STAGES, nkb);                      // stages whose weight half is requested before the wait
    if (warp == 0) {
        for (int st = 0; st < pre; ++st)
            if (elect_one()) {
                mbar_expect_tx(full0 + 8 * st, SPK_STAGE);
                tma_load_2d(ring + st * SPK_STAGE + SPK_A_KB, &tmW, (kb0 + st) * TC_BK, n0, full0 + 8 * st);
            }
    }
    pdl_launch_dependents();
    if (threadIdx.x == 0) tma_prefetch_map(&tmA);
    pdl_wait();
    if (warp == 0) {
        int s = 0; uint32_t par = 1;                           // (a fresh barrier counts as past the phase before its first)
        for (int kb = 0; kb < nkb; ++kb) {
            if (!mbar_wait_warp(empty0 + 8 * s, par, abort_flag, err_word, 1)) break;
            const uint32_t dst = ring + s * SPK_STAGE, bar = full0 + 8 * s;
            if (elect_one()) {
                if (kb >= pre) {
                    mbar_expect_tx(bar, SPK_STAGE);
                    tma_load_2d(dst + SPK_A_KB, &tmW, (kb0 + kb) * TC_BK, n0, bar);
                }
                tma_load_2d(dst, &tmA, (kb0 + kb) * TC_BK, m0, bar);
            }
            if (++s == SPK_STAGES) { s = 0; par ^= 1u; }
        }
    } else if (warp == 1) {
        constexpr uint32_t idesc = umma_idesc_bf16(TC_BM, BN);
        int s = 0; uint32_t par = 0; bool ok = true;
        for (int kb = 0; kb < nkb; ++kb) {
            ok = mbar_wait_warp(full0 + 8 * s, par, abort_flag, err_word, 2);
            if (!ok) break;
            tc_fence_after();
            const uint32_t a_src = ring + s * SPK_STAGE, bar = empty0 + 8 * s;
            if (elect_one()) {
                const uint64_t ad = umma_desc_k_sw128(a_src), wd = umma_desc_k_sw128(a_src + SPK_A_KB);
                umma_bf16(tmem_d, ad, wd, idesc, kb ? 1u : 0u);
                umma_bf16(tmem_d, ad + 2, wd + 2, idesc, 1u);
                umma_bf16(tmem_d, ad + 4, wd + 4, idesc, 1u);
                umma_bf16(tmem_d, ad + 6, wd + 6, idesc, 1u);
                umma_commit(bar);
            }
            if (++s == SPK_STAGES) { s = 0; par ^= 1u; }
        }
        if (ok && elect_one()) umma_commit(smem_u32(&bar_acc));
    } else {
        const int q = warp & 3, half = (warp - 2) >> 2, e = (int)threadIdx.x - 64;
        // the residual and bias of the outputs that this thread will finish: rows e / 16 + 16 i of the CTA's share, four columns of each block
        const int c = (e & 15) * 4, row0 = m0 + (int)rank * OWN + (e >> 4);
        float4 x[NB][OWN / 16], bz[NB];
#pragma unroll
        for (int n = 0; n < NB; ++n) {
            bz[n] = g.bias ? __ldg(reinterpret_cast<const float4*>(g.bias + n0 + n * 64 + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int i = 0; i < OWN / 16; ++i)
                x[n][i] = row0 + 16 * i < R ? *reinterpret_cast<const float4*>(g.resid + (size_t)(row0 + 16 * i) * g.N + n0 + n * 64 + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        bool ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_acc), 0, abort_flag, err_word, 3));      // the MMAs are done: the ring is free
        tc_fence_after();
        if (ok && q * 32 < AR) {
#pragma unroll
            for (int n = 0; n < NB; ++n) {
                float v[32];
                tmem_ld32(tmem_d + ((uint32_t)(q * 32) << 16) + (uint32_t)(n * 64 + half * 32), v);
                // a row per lane, its 16-byte chunks XOR-swizzled by the row
                const int out = (n * TC_EPI_WARPS + warp - 2) * 4096;
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    *reinterpret_cast<float4*>(ring_p + out + lane * 128 + ((j ^ (lane & 7)) << 4)) = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane < 32 / RB) {
                    const uint32_t row = q * 32 + lane * RB, owner = row / OWN,
                                   dst = recv + n * (AR * 256) + ((rank * (OWN / RB) + row % OWN / RB) * 2 + half) * (RB * 128);
                    uint32_t ra, rb;
                    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(dst), "r"(owner));
                    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rb) : "r"(smem_u32(&bar_part)), "r"(owner));
                    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                 ::"r"(ra), "r"(ring + out + lane * (RB * 128)), "r"(RB * 128), "r"(rb) : "memory");
                }
                __syncwarp();
            }
        }
        ok = ok && mbar_wait(smem_u32(&bar_part), 0, abort_flag, err_word, 10);          // all slices of this CTA's rows have landed
        if (ok) {
            const uint8_t* src = ring_p + SPK_STAGES * SPK_STAGE + ((e & 15) >> 3) * (RB * 128);
#pragma unroll
            for (int n = 0; n < NB; ++n)
#pragma unroll
                for (int i = 0; i < OWN / 16; ++i) {
                    const int row = (e >> 4) + 16 * i;
                    const uint8_t* p = src + n * (AR * 256) + row / RB * (RB * 256) + row % RB * 128 + (((e & 7) ^ (row & 7)) << 4);
                    float4 a = *reinterpret_cast<const float4*>(p);
#pragma unroll
                    for (int s = 1; s < SPLIT; ++s) {                                    // rank order: fixed summation order
                        const float4 t = *reinterpret_cast<const float4*>(p + s * (OWN * 256));
                        a.x += t.x; a.y += t.y; a.z += t.z; a.w += t.w;
                    }
                    a.x += bz[n].x; a.y += bz[n].y; a.z += bz[n].z; a.w += bz[n].w;
                    a.x += x[n][i].x; a.y += x[n][i].y; a.z += x[n][i].z; a.w += x[n][i].w;
                    if (row0 + 16 * i < R) *reinterpret_cast<float4*>(g.resid + (size_t)(row0 + 16 * i) * g.N + n0 + n * 64 + c) = a;
                }
        }
    }
    tc_fence_before();
    __syncwarp();
    tc_cluster_sync();                                         // nobody leaves while a copy from its shared memory may be under way
    if (warp == 1) tmem_dealloc(tmem_d, BN);
}

template <int SPLIT, int AR, int BN>
inline cudaLaunchConfig_t spk_config(cudaLaunchAttribute* attr, dim3 grid, bool pdl, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = dim3(TC_THREADS); cfg.dynamicSmemBytes = SpkCfg<AR, BN>::SMEM; cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = SPLIT; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = pdl ? 2 : 1;
    return cfg;
}
template <int SPLIT, int AR, int BN>
inline cudaError_t spk_init_one(int* clusters) {
    cudaError_t e = cudaFuncSetAttribute(k_gemm_tc_splitk<SPLIT, AR, BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, SpkCfg<AR, BN>::SMEM);
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = spk_config<SPLIT, AR, BN>(attr, dim3(SPLIT), false, nullptr);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(clusters, k_gemm_tc_splitk<SPLIT, AR, BN>, &cfg);
    return e;
}
inline cudaError_t spk_init(TmaEncoder& enc) {
    cudaError_t e = spk_init_one<4, TC_BM, 64>(&enc.spk_clusters4);
    if (e == cudaSuccess) e = spk_init_one<4, 64, 64>(&enc.spk_clusters4_64);
    if (e == cudaSuccess) e = spk_init_one<2, TC_BM, 64>(&enc.spk_clusters2);
    return e == cudaSuccess ? spk_init_one<2, TC_BM, 128>(&enc.spk_clusters2_128) : e;
}

template <int SPLIT, int AR, int BN>
inline int spk_launch_one(TmaEncoder& enc, GemmArgs<bf16>& g, int rows_ub, cudaStream_t st) {
    CUtensorMap ta, tw;
    if (!enc.get(ta, g.A, rows_ub, g.K, g.lda, AR) || !enc.get(tw, g.W, g.N, g.K, g.K, BN)) return -1;
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = spk_config<SPLIT, AR, BN>(attr, dim3(g.N / BN * SPLIT, (rows_ub + AR - 1) / AR), enc.pdl, st);
    cudaError_t e = cudaLaunchKernelEx(&cfg, k_gemm_tc_splitk<SPLIT, AR, BN>, ta, tw, g, enc.err_word);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) { enc.err = std::string("launch (split-K): ") + cudaGetErrorString(e); return -1; }
    return 0;
}
inline int spk_launch(TmaEncoder& enc, SpkPlan plan, GemmArgs<bf16>& g, int rows_ub, cudaStream_t st) {
    if (!enc.ready) return -1;
    if (plan.rows == 64) return spk_launch_one<4, 64, 64>(enc, g, rows_ub, st);
    if (plan.cols == 128) return spk_launch_one<2, TC_BM, 128>(enc, g, rows_ub, st);
    return plan.split == 4 ? spk_launch_one<4, TC_BM, 64>(enc, g, rows_ub, st) : spk_launch_one<2, TC_BM, 64>(enc, g, rows_ub, st);
}

}  // namespace sd
