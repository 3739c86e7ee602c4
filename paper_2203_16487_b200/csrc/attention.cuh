// Attention for bf16 operands and head size 64: one CTA per (tile of 16 MT queries, head, sequence).  Used for the verifier's
// causal attention over the paged cache, both cross-attentions, the drafter's bidirectional attention and the encoders.
//
// K and V walk through a ring of NS cp.async stages (128-byte rows, XOR-swizzled 16-byte chunks).  Warp (row tile mt, key group
// kg) takes KW keys of every block for 16 queries: S = Q K^T (mma.sync m16n8k16, fp32 accumulation), running row maximum and
// sum in registers, P (bf16, relative to the running maximum); the result is divided by the fp32 sum of the unrounded exponentials.  (A bf16 value keeps its relative precision whatever the
// maximum it is taken relative to: against 64 bits the result is 1.0e-3 off with the running maximum where it is 1.2e-3 with the row's, 512 keys.)
// P goes straight from the score registers into the second contraction, and with KG > 1 the partial outputs of a row tile's key groups meet in shared memory at the
// end, added in group order; or, over one block of keys (SHARE), every group leaves its P in shared memory where its keys were, and each warp contracts all groups' P with its own
// slice of V's columns.  Work per CTA is 64 keys x 64 x 16 MT x 4 flops a block: too little to
// fill a 128-row tcgen05 tile, which is why this contraction uses warp-level MMA (8 clocks each per scheduler, measured).
//
// What bounds it.  Few CTAs: the chain of round trips of one CTA.  Everything that predates the step -- row counts, the page
// table's rows of all keys, the cached keys themselves -- is fetched ahead of the dependency wait, so that one round trip (queries and
// new keys) is left behind it, and the keys are spread over four or eight warps (verify step at 26 rows: 176 us with the one-shot
// kernel this one replaces, 161 with MT = 1, KG = 4).  Many CTAs: the fixed-latency chain inside a warp, so
// warps per SM and whole waves count: 16 of them, in CTAs of 64 queries with a ring of two 64-key blocks (128 sequences x 51 queries x 307 keys, verify
// step with 12 warps and a ring of three 1107 us, now 1055-1075) or of 32 queries with 32-key blocks (x 26 x 90: 555 with 8 warps and
// 64-key blocks, now 514).  Both are cut to 128 registers; with 64 queries that leaves 16 bytes a thread in local memory.  The tensor
// pipe is active 26 % of the time there, shared memory 41 %, and a warp waits 8.8 cycles for each instruction.  Below four CTAs an SM there is nothing to
// fill the SMs with, and 64-key blocks have more independent work per barrier: 32 queries take those, at 174 registers and 8 warps an SM.
#pragma once
#include "barriers.cuh"
#include "kernels.cuh"

namespace sd {

struct AttnTcArgs {
    const bf16* q; int q_stride; const int* q_index;     // query row r reads q + (q_index ? q_index[r] : r) * q_stride
    const bf16* k; const bf16* v; int kv_stride;         // contiguous: key t of sequence b at row kv_off[b] + t
    const int* kv_off;
    Paged pg;                                             // paged: row pg.row(b, t)
    const int* q_off; const int* q_cnt;                   // per sequence: first query row, number of query rows
    const int* seq_of;                                    // the sequence of grid slice z (-1: none), or null: slice z is sequence z
    const int* nkeys;                                     // per query row: visible keys (0..nkeys-1)
    const int* pre_keys;                                  // per sequence (or null): keys 0..pre-1 were written before this
                                                          // step began, so they may be fetched before the dependency wait
    bf16* out; int out_stride;
    int max_keys;                                         // upper bound on nkeys
    float scale;
};

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// byte offset of 16-byte chunk c (0..7) of row r in a tile of 128-byte rows
__device__ __forceinline__ uint32_t swz(int r, int c) { return (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4)); }
// 2^x for x <= 0: results below 2^-126 are 0.
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ void cp_wait_pending(int n) {       // cp.async.wait_group takes an immediate
    if (n <= 0) asm volatile("cp.async.wait_group 0;" ::: "memory");
    else if (n == 1) asm volatile("cp.async.wait_group 1;" ::: "memory");
    else if (n == 2) asm volatile("cp.async.wait_group 2;" ::: "memory");
    else asm volatile("cp.async.wait_group 3;" ::: "memory");
}

// The query projection inside the attention kernel (cross-attention of few rows): q = LN(x) Wq^T + bq for the CTA's 16 rows and head.
struct QueryArgs {
    const float* x;                                       // fp32 rows [rows, K]
    const float* ln_g; const float* ln_b; float eps;
    const bf16* w; const float* b;                        // [n_heads * 64, K]
};
template <int QNC> struct QueryCfg {                      // K = 128 QNC
    static constexpr int K = 128 * QNC, PITCH = K * 2 + 16;                           // bytes per row
    static constexpr int OPS = QNC ? (16 + 64) * PITCH : 0;
};

// The output projection and the residual sum inside the attention kernel (few rows): x_out[r] = x_in[x_index ? x_index[r] : r] + O Wo^T + bo.
struct OutArgs {
    const bf16* w; const float* b;                        // [K, K], K = 64 n_heads
    const float* x_in; const int* x_index; float* x_out;  // fp32 rows [rows, K]
    int* err_word;                                        // raised when the bounded wait for the other heads gives up
};
// Bytes behind the ring: 16 rows and 64 rows of weights for each projection that runs inside.
template <int QNC, int ON> struct ProjCfg { static constexpr int OPS = QueryCfg<QNC>::OPS + QueryCfg<ON / 2>::OPS; };

// 16 x 64 partial products of a CTA's eight warps: warp = (K slice of four, half of the columns); A: 16 rows, W: 64 rows of PITCH bytes.
// The slices meet in `red` ([4][16][72] floats); thread t then holds row t / 16, columns 4 (t % 16) .. + 3 of the sum.
template <int K>
struct Proj64 {
    static constexpr int PITCH = K * 2 + 16, RP = 72, STEPS = K / 64;
    uint32_t bfr[STEPS][4][2];
    __device__ __forceinline__ void load_w(uint32_t ws, int warp, int lane) {
        const uint32_t bp = ws + ((warp & 1) * 32 + (lane & 7) + (lane >> 4) * 8) * PITCH + (warp >> 1) * STEPS * 32 + ((lane >> 3) & 1) * 16;
#pragma unroll
        for (int s = 0; s < STEPS; ++s) {
            ldsm_x4(bp + s * 32, bfr[s][0][0], bfr[s][0][1], bfr[s][1][0], bfr[s][1][1]);
            ldsm_x4(bp + 16 * PITCH + s * 32, bfr[s][2][0], bfr[s][2][1], bfr[s][3][0], bfr[s][3][1]);
        }
    }
    // BLOCKED: A as 8-column chunks of 16 rows of 16 bytes, the way the heads send them; else rows of PITCH bytes
    template <bool BLOCKED>
    __device__ __forceinline__ void multiply(uint32_t as, float* red, int warp, int lane) {
        float c[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) c[j][e] = 0.f;
        const uint32_t ap = BLOCKED ? as + ((warp >> 1) * STEPS * 2 + (lane >> 4)) * 256 + (lane & 15) * 16
                                    : as + (lane & 15) * PITCH + (warp >> 1) * STEPS * 32 + (lane >> 4) * 16;
#pragma unroll
        for (int s = 0; s < STEPS; ++s) {
            uint32_t af[4];
            ldsm_x4(ap + s * (BLOCKED ? 512 : 32), af[0], af[1], af[2], af[3]);
#pragma unroll
            for (int j = 0; j < 4; ++j) mma_bf16(c[j], af, bfr[s][j][0], bfr[s][j][1]);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float* p = red + ((warp >> 1) * 16 + (lane >> 2)) * RP + (warp & 1) * 32 + j * 8 + (lane & 3) * 2;
            *reinterpret_cast<float2*>(p) = make_float2(c[j][0], c[j][1]);
            *reinterpret_cast<float2*>(p + 8 * RP) = make_float2(c[j][2], c[j][3]);
        }
    }
    static __device__ __forceinline__ float4 sum(const float* red, int tid) {
        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            const float4 u = *reinterpret_cast<const float4*>(red + (s * 16 + (tid >> 4)) * RP + (tid & 15) * 4);
            t.x += u.x; t.y += u.y; t.z += u.z; t.w += u.w;
        }
        return t;
    }
};

constexpr int SHARE_KEYS = 128;                           // up to so many keys the groups share probabilities: the one block of every SHARE kernel
constexpr int ATTN_SMEM = 227 * 1024 - 2048;              // dynamic shared memory of a CTA; the rest is for what the kernel declares

// MT row tiles of 16 queries x KG key groups = MT KG warps; a key block holds KW keys for each group; NS stages.
template <int MT, int KG, int KW>
struct AttnCfg {
    static constexpr int KB = KG * KW;                                    // keys per block
    static constexpr int STAGE = KB * 256;                                // K and V of a block
    static constexpr int PP = KW * 2 + 16;                                // bytes per row of a key group's probabilities: 16 rows, in place of the group's keys
    static constexpr int MERGE = KG > 1 ? MT * KG * 16 * (72 + 2) * 4 : 0;     // partial outputs (padded rows) and (maximum, sum); reuses the stages
    // queries, ring (or merge buffers), operands of the projections, and for paged keys the table of their rows
    static constexpr size_t smem(int max_keys, int ns, bool paged, int query_bytes = 0) {
        const int nb = (max_keys + KB - 1) / KB;
        const size_t ring = (size_t)(nb < ns ? (nb < 1 ? 1 : nb) : ns) * STAGE;
        return (size_t)MT * 2048 + (ring > MERGE ? ring : MERGE) + query_bytes + (paged ? (size_t)((max_keys + 3) & ~3) * 4 : 0);
    }
};

// CTAs per SM that the registers are cut for; 0 leaves it to the compiler (told 1, it takes 148 registers for MT = 1, KG = 4 where 100 do, and the
// verify step of 832 rows 334 us instead of 316; MT = 2 with 64-key blocks is better with its 174 than with 129: 1664 rows 388 / 400 us).  Four groups that share are told 5
// (86 registers; left to itself it takes 59: verify steps of 26 rows 112.9 / 115.0, 416 rows of 768 columns 364.4 / 367.5, encoder of 64 ids 215.8 / 219.7, others level to 1 %).
constexpr int attn_ctas(int mt, int kg, int kw, bool share) { return kg > 1 ? (share && kg == 4 ? 5 : 0) : mt == 4 ? 4 : kw == 32 ? 8 : 1; }

// QNC > 0: the queries are projected here (QueryArgs; MT = 1, KG = 8).  The CTA's 64 rows of Wq are requested ahead of the wait, the
// 16 rows normalised behind it; one launch and its round trip through memory less per layer (26 rows, K = 512: 5.5 -> 4.4 us).
//
// ON > 0: the heads of a query tile are a cluster of ON CTAs, and the output projection runs here too (OutArgs).  Bound by the same chain of round trips:
// every CTA sends its head's 16 rows (bf16, as they would go to memory) to the shared memory of all, multiplies the 16 whole rows by its own 64 rows
// of Wo and adds the residual.  A launch and its round trip less (verify step of 26 rows, both attentions of six layers: 156.5 -> 147.2 us).
//   * Wo, and Wq with QNC, are requested ahead of the wait and are register fragments by the time it returns (fetched behind it 155.2 us; turned into fragments
//     behind it, while the rows arrive, their 128 KB from shared memory delayed the LayerNorm: rows and LayerNorm 1.5 us, now 1.0);
//   * the head's 16 rows, 2 KB, go to each CTA as one bulk copy, every copy issued by another warp and counted on the receiver's mbarrier.  (As eight copies of 256
//     bytes from the lanes of every warp their issue alone took 790 clocks, one lane after the other; 16-byte asynchronous remote stores 0.85 us, plain ones behind a
//     cluster barrier more.)
//
// SHARE: the keys are one block (at most SHARE_KEYS), and the groups do not add up partial outputs of all 64 columns through shared memory (35 KB written and read for
// eight groups: 990 + 910 clocks) but leave their probabilities there, where their keys were (6 KB); every warp then multiplies those of all groups by its own
// 64 / KG columns of the values.  The groups' shares are scaled and added in the same order with the same roundings: results are the same to the bit.
// us a pass, in turn: before | with the 2 KB copies above and the pitch below | sharing as well.
//   verify  5 rows 104.9 | 100.8 | 98.9    16 rows 107.9 | 104.9 | 103.6    26 rows 115.1 | 113.2 | 112.9    416 rows 249.1 | 245.2 | 234.0    624 rows 284.8 | 280.4 | 276.4
//           832 rows 311.5 | 304.9 | 306.1 (sharing itself loses 0.4 % there)       768 columns, 416 rows 370.7 | 363.4 | 364.4
//   drafts of 8 x (21 + 16) rows 83.9 | - | 81.4;  encoders of 64 ids 218.7 | 217.9 | 215.8, of 120 268.9 | 266.0 | 262.0, of 480 417.8 | 411.1 | 409.9
// Over several blocks every warp would read the probabilities of eight groups once a block (2 sequences, 512 keys: 691 / 714 us an encode
// pass): those add partial outputs, in rows of 72 floats, which keep stores and loads out of each other's banks (68 | 72: 26 rows over 276 keys 133.5 | 130.1, 4 x 26 rows
// 175.1 | 172.0, encoders of 2 x 512 ids 693.4 | 685.7; no pass of 22 got slower).
// (QNC and ON stay the last two: the test of the routes reads them off the kernel's name.)
template <bool PAGED, int MT, int KG, int KW, int NS, bool SHARE = false, int QNC = 0, int ON = 0>
__global__ void __launch_bounds__(MT * KG * 32, attn_ctas(MT, KG, KW, SHARE)) k_attn(AttnTcArgs a, QueryArgs qa, OutArgs oa) {
    using C = AttnCfg<MT, KG, KW>;
    static_assert((QNC == 0 && ON == 0) || (MT == 1 && KG == 8), "the projections are laid out for eight warps and 16 rows");
    static_assert(QNC == 0 || ON == 0 || ON == 2 * QNC, "one width");
    static_assert(NS >= 1 && NS <= 4 && KW % 16 == 0, "ring depth, keys per warp");
    static_assert(!SHARE || C::KB >= SHARE_KEYS, "one block holds all keys: there is no second pass");
    static_assert(!SHARE || ((KG == 4 || KG == 8) && MT == 1 && 16 * C::PP <= KW * 128), "a warp's one or two 8-column tiles, one row tile, probabilities where the keys were");
    constexpr int THREADS = MT * KG * 32, KB = C::KB, NT = KW / 8, BM = MT * 16;
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ int s_nk[BM];
    __shared__ int s_nkmax;
    __shared__ __align__(8) uint64_t heads_bar;               // ON: counts the heads' rows as they arrive
    __shared__ int abort_s;
    __shared__ float2 s_ml[SHARE ? KG : 1][16];                // (maximum, sum) of every key group and row
    const int b = a.seq_of ? a.seq_of[blockIdx.z] : (int)blockIdx.z, h = blockIdx.y, qt = blockIdx.x;
    if (b < 0) return;
    // Row metadata, page table and sequence lengths are written at the start of the step, before the first
    // kernel of the programmatic-launch chain can begin, so they may be read before the dependency wait.
    const int cnt = a.q_cnt[b], q_first = a.q_off[b];
    const int pre = a.pre_keys ? min(a.pre_keys[b], a.max_keys) : 0, kv0 = PAGED ? 0 : a.kv_off[b];
    if (qt * BM >= cnt) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int r0 = q_first + qt * BM, nq = min(BM, cnt - qt * BM);
    const int nb_cap = (a.max_keys + KB - 1) / KB, ring = nb_cap < NS ? max(nb_cap, 1) : NS;        // stages that shared memory was sized for
    const uint32_t Qs = (uint32_t)__cvta_generic_to_shared(sm), St = Qs + BM * 128;
    unsigned char* Sp = sm + BM * 128;
    using QC = QueryCfg<QNC>;
    unsigned char* qops = Sp + max(ring * C::STAGE, C::MERGE);             // QNC: 16 rows, then 64 weight rows, of QC::PITCH bytes
    float4 lgam[QNC ? QNC : 1], lbet[QNC ? QNC : 1];
    if constexpr (QNC > 0) {
        const uint32_t ws = (uint32_t)__cvta_generic_to_shared(qops) + 16 * QC::PITCH;
        const bf16* w = qa.w + (size_t)h * 64 * QC::K;
        for (int i = tid; i < 64 * (QC::K / 8); i += THREADS) {
            const int r = i / (QC::K / 8), c = i % (QC::K / 8);
            cp_async16(ws + r * QC::PITCH + c * 16, w + (size_t)r * QC::K + c * 8);
        }
#pragma unroll
        for (int c = 0; c < QNC; ++c) {
            lgam[c] = ldg_pinned(reinterpret_cast<const float4*>(qa.ln_g + lane * 4 + c * 128));
            lbet[c] = ldg_pinned(reinterpret_cast<const float4*>(qa.ln_b + lane * 4 + c * 128));
        }
    }
    using OC = QueryCfg<ON ? ON / 2 : 2>;
    const uint32_t oops = (uint32_t)__cvta_generic_to_shared(qops) + QC::OPS;   // ON: 16 rows that the cluster's CTAs fill, this head's 64 rows of Wo
    Proj64<OC::K> wo;
    float4 res = make_float4(0.f, 0.f, 0.f, 0.f), ob = res;              // ON: the residual and the bias of this thread's four outputs
    if constexpr (ON > 0) {
        const bf16* w = oa.w + (size_t)h * 64 * OC::K;
        for (int i = tid; i < 64 * (OC::K / 8); i += THREADS) {
            const int r = i / (OC::K / 8), c = i % (OC::K / 8);
            cp_async16(oops + (16 + r) * OC::PITCH + c * 16, w + (size_t)r * OC::K + c * 8);
        }
        if (tid == 0) {
            abort_s = 0;
            mbar_init(smem_u32(&heads_bar), 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            mbar_expect_tx(smem_u32(&heads_bar), 16 * OC::K * 2);           // all heads' columns of the 16 rows, this CTA's own among them
        }
        __syncwarp();
        cluster_arrive();
        ob = ldg_pinned(reinterpret_cast<const float4*>(oa.b + h * 64 + (tid & 15) * 4));
    }
    int* s_row = reinterpret_cast<int*>(qops + ProjCfg<QNC, ON>::OPS);            // paged: K / V row of every key
    if (PAGED) {
        for (int t = tid; t < a.max_keys; t += THREADS) s_row[t] = (int)a.pg.row(b, t);
        __syncthreads();
    }
    const int c8 = tid & 7, t0 = tid >> 3;      // a thread keeps its 16-byte chunk of the 128-byte head slice and walks the keys
    const bf16* kcol = a.k + h * 64 + c8 * 8;
    const bf16* vcol = a.v + h * 64 + c8 * 8;
    // keys [blk KB + lo, blk KB + hi) of a block into its stage; rows past the last key (n) are zeroed
    auto load_keys = [&](int blk, int lo, int hi, int n) {
        const uint32_t Ks = St + (blk % ring) * C::STAGE, Vs = Ks + KB * 128;
        for (int t = lo + t0; t < hi; t += THREADS / 8) {
            const int key = blk * KB + t;
            if (key < n) {
                const size_t off = (size_t)(PAGED ? s_row[key] : kv0 + key) * a.kv_stride;
                cp_async16(Ks + swz(t, c8), kcol + off);
                cp_async16(Vs + swz(t, c8), vcol + off);
            } else {
                *reinterpret_cast<uint4*>(sm + (Ks - Qs) + swz(t, c8)) = make_uint4(0, 0, 0, 0);
                *reinterpret_cast<uint4*>(sm + (Vs - Qs) + swz(t, c8)) = make_uint4(0, 0, 0, 0);
            }
        }
    };
    // keys that predate this step (cached prefix, encoder memory) are requested before the wait, as far as the ring reaches ...
    const int npre = min(pre, ring * KB);
    for (int blk = 0; blk * KB < npre; ++blk) load_keys(blk, 0, min(npre - blk * KB, KB), npre);
    if (tid < 32) {
        int m = 0;
#pragma unroll
        for (int i = 0; i < (BM + 31) / 32; ++i) {
            const int r = tid + i * 32;
            const int nk = r < nq ? min(a.nkeys[r0 + r], a.max_keys) : 0;
            if (r < BM) s_nk[r] = nk;
            m = max(m, nk);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (tid == 0) s_nkmax = m;
    }
    if constexpr (ON > 0 || QNC > 0) asm volatile("cp.async.commit_group;" ::: "memory");
    __syncthreads();
    const int nkmax = s_nkmax, nblk = max((nkmax + KB - 1) / KB, 1);
    pdl_launch_dependents();
    // the weights become fragments as soon as they are here, still ahead of the wait
    Proj64<QNC ? QC::K : 256> pj;
    if constexpr (ON > 0 || QNC > 0) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        if constexpr (QNC > 0) pj.load_w((uint32_t)__cvta_generic_to_shared(qops) + 16 * QC::PITCH, warp, lane);
        if constexpr (ON > 0) wo.load_w(oops + 16 * OC::PITCH, warp, lane);
    }
    pdl_wait();                                  // ... and everything the predecessor kernels wrote after it
    if constexpr (ON > 0) {
        const int r = tid >> 4;
        if (r < nq) res = *reinterpret_cast<const float4*>(oa.x_in + (size_t)(oa.x_index ? oa.x_index[r0 + r] : r0 + r) * OC::K + h * 64 + (tid & 15) * 4);
    }
    if constexpr (QNC == 0) {
        for (int r = t0; r < BM; r += THREADS / 8) {
            if (r < nq) {
                const size_t qr = a.q_index ? (size_t)a.q_index[r0 + r] : (size_t)(r0 + r);
                cp_async16(Qs + swz(r, c8), a.q + qr * a.q_stride + h * 64 + c8 * 8);
            } else {
                *reinterpret_cast<uint4*>(sm + swz(r, c8)) = make_uint4(0, 0, 0, 0);
            }
        }
    } else {
        constexpr float INV_K = 1.0f / QC::K;
        float4 xv[2][QNC];
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int c = 0; c < QNC; ++c) {
                const int m = warp + 8 * s;
                xv[s][c] = m < nq ? *reinterpret_cast<const float4*>(qa.x + (size_t)(r0 + m) * QC::K + lane * 4 + c * 128) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        const float4 v = __ldg(reinterpret_cast<const float4*>(qa.b + h * 64 + (tid & 15) * 4));
        float mu[2] = {0.f, 0.f}, rs[2] = {0.f, 0.f};
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int c = 0; c < QNC; ++c) mu[s] += (xv[s][c].x + xv[s][c].y) + (xv[s][c].z + xv[s][c].w);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { mu[0] += __shfl_xor_sync(0xffffffffu, mu[0], o); mu[1] += __shfl_xor_sync(0xffffffffu, mu[1], o); }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            mu[s] *= INV_K;
#pragma unroll
            for (int c = 0; c < QNC; ++c) {
                xv[s][c].x -= mu[s]; xv[s][c].y -= mu[s]; xv[s][c].z -= mu[s]; xv[s][c].w -= mu[s];
                rs[s] = fmaf(xv[s][c].x, xv[s][c].x, rs[s]); rs[s] = fmaf(xv[s][c].y, xv[s][c].y, rs[s]);
                rs[s] = fmaf(xv[s][c].z, xv[s][c].z, rs[s]); rs[s] = fmaf(xv[s][c].w, xv[s][c].w, rs[s]);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { rs[0] += __shfl_xor_sync(0xffffffffu, rs[0], o); rs[1] += __shfl_xor_sync(0xffffffffu, rs[1], o); }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            rs[s] = 1.0f / sqrtf(rs[s] * INV_K + qa.eps);
            const int m = warp + 8 * s;
#pragma unroll
            for (int c = 0; c < QNC; ++c) {
                const float4 v = xv[s][c];
                __nv_bfloat162 p0 = __floats2bfloat162_rn(fmaf(v.x * rs[s], lgam[c].x, lbet[c].x), fmaf(v.y * rs[s], lgam[c].y, lbet[c].y));
                __nv_bfloat162 p1 = __floats2bfloat162_rn(fmaf(v.z * rs[s], lgam[c].z, lbet[c].z), fmaf(v.w * rs[s], lgam[c].w, lbet[c].w));
                *reinterpret_cast<uint2*>(qops + m * QC::PITCH + (lane * 4 + c * 128) * 2) =
                    m < nq ? make_uint2(*reinterpret_cast<uint32_t*>(&p0), *reinterpret_cast<uint32_t*>(&p1)) : make_uint2(0u, 0u);
            }
        }
        __syncthreads();
        const uint32_t ops = (uint32_t)__cvta_generic_to_shared(qops);
        float* red = reinterpret_cast<float*>(Sp + max(ring * C::STAGE, C::MERGE) + 16 * QC::PITCH);        // (weights that are dead by then)
        pj.template multiply<false>(ops, red, warp, lane);
        __syncthreads();
        const int r = tid >> 4, c = (tid & 15) * 4;
        const float4 t = Proj64<QC::K>::sum(red, tid);
        __nv_bfloat162 p0 = __floats2bfloat162_rn(t.x + v.x, t.y + v.y), p1 = __floats2bfloat162_rn(t.z + v.z, t.w + v.w);
        *reinterpret_cast<uint2*>(sm + swz(r, c >> 3) + (c & 7) * 2) = make_uint2(*reinterpret_cast<uint32_t*>(&p0), *reinterpret_cast<uint32_t*>(&p1));
    }
    int issued = 0;
    auto issue = [&]() {                         // the rest of block `issued`, one commit group per block
        load_keys(issued, min(max(npre - issued * KB, 0), KB), KB, nkmax);
        asm volatile("cp.async.commit_group;" ::: "memory");
        ++issued;
    };

    const int g = lane >> 2, t4 = lane & 3;
    const int mt = warp % MT, kg = warp / MT;    // query rows 16 mt .. + 15, keys KW kg .. + KW - 1 of every block
    const int nk0 = s_nk[mt * 16 + g], nk1 = s_nk[mt * 16 + g + 8];
    uint32_t qf[4][4];
    float m_run[2] = {-CUDART_INF_F, -CUDART_INF_F}, l_run[2] = {0.f, 0.f};   // rows g, g + 8 (sums: this lane's share)
    constexpr int NJ = SHARE ? 8 / KG : 8;       // 8-column tiles of a warp: all of them, or its share for every key group
    float acc[8][4];                             // [column tile], [key group * NJ + column tile]
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[j][e] = 0.f;
    const float sl = a.scale * 1.4426950408889634f;      // exp(scale (s - max)) as 2^(sl s - sl max)
    // keys that every row of this warp sees (rows past the last query see none and are never stored)
    int nkall = mt * 16 + g < nq ? nk0 : 0x7fffffff;
    if (mt * 16 + g + 8 < nq) nkall = min(nkall, nk1);
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) nkall = min(nkall, __shfl_xor_sync(0xffffffffu, nkall, o));

    while (issued < min(ring, nblk)) issue();
    for (int blk = 0; blk < (SHARE ? 1 : nblk); ++blk) {
        cp_wait_pending(issued - blk - 1);
        __syncthreads();
        if (blk == 0) {
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
                const int r = mt * 16 + (lane & 7) + ((lane >> 3) & 1) * 8, c = ks * 2 + (lane >> 4);
                ldsm_x4(Qs + swz(r, c), qf[ks][0], qf[ks][1], qf[ks][2], qf[ks][3]);
            }
        }
        const uint32_t Ks = St + (blk % ring) * C::STAGE + kg * KW * 128, Vs = Ks + KB * 128;
        const int kbase = blk * KB + kg * KW;
        if (kbase < nkmax && mt * 16 < nq) {       // warp-uniform: a visible key, a live query
            float sc[NT][4];
            float bm0 = -CUDART_INF_F, bm1 = -CUDART_INF_F;
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                uint32_t kf[2][4];
#pragma unroll
                for (int kk = 0; kk < 2; ++kk)
                    ldsm_x4(Ks + swz(nt * 8 + (lane & 7), kk * 4 + (lane >> 3)), kf[kk][0], kf[kk][1], kf[kk][2], kf[kk][3]);
                float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) mma_bf16(s4, qf[ks], kf[ks >> 1][(ks & 1) * 2], kf[ks >> 1][(ks & 1) * 2 + 1]);
#pragma unroll
                for (int e = 0; e < 4; ++e) sc[nt][e] = s4[e];
            }
            if (kbase + KW > nkall) {              // a block at some row's last key
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) {
                    const int col = kbase + nt * 8 + t4 * 2;
                    if (col >= nk0) sc[nt][0] = -CUDART_INF_F;
                    if (col + 1 >= nk0) sc[nt][1] = -CUDART_INF_F;
                    if (col >= nk1) sc[nt][2] = -CUDART_INF_F;
                    if (col + 1 >= nk1) sc[nt][3] = -CUDART_INF_F;
                }
            }
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                bm0 = fmaxf(bm0, fmaxf(sc[nt][0], sc[nt][1]));
                bm1 = fmaxf(bm1, fmaxf(sc[nt][2], sc[nt][3]));
            }
            bm0 = fmaxf(bm0, __shfl_xor_sync(0xffffffffu, bm0, 1)); bm1 = fmaxf(bm1, __shfl_xor_sync(0xffffffffu, bm1, 1));
            bm0 = fmaxf(bm0, __shfl_xor_sync(0xffffffffu, bm0, 2)); bm1 = fmaxf(bm1, __shfl_xor_sync(0xffffffffu, bm1, 2));
            const float mn0 = fmaxf(m_run[0], bm0), mn1 = fmaxf(m_run[1], bm1);
            // a row with no visible key so far keeps maximum -inf: its terms are 0 against a base of 0
            const float mb0 = (mn0 == -CUDART_INF_F) ? 0.f : mn0 * sl, mb1 = (mn1 == -CUDART_INF_F) ? 0.f : mn1 * sl;
            if (!SHARE && blk > 0) {
                const float al0 = ex2(fmaf(m_run[0], sl, -mb0)), al1 = ex2(fmaf(m_run[1], sl, -mb1));      // (maximum -inf: 0, on sums that are 0)
                l_run[0] *= al0; l_run[1] *= al1;
#pragma unroll
                for (int j = 0; j < 8; ++j) { acc[j][0] *= al0; acc[j][1] *= al0; acc[j][2] *= al1; acc[j][3] *= al1; }
            }
            m_run[0] = mn0; m_run[1] = mn1;
#pragma unroll
            for (int kt = 0; kt < NT / 2; ++kt) {
                uint32_t pf[4];
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    const float* s = sc[2 * kt + hf];
                    const float e0 = ex2(fmaf(s[0], sl, -mb0)), e1 = ex2(fmaf(s[1], sl, -mb0));      // -inf scores give 0
                    const float e2 = ex2(fmaf(s[2], sl, -mb1)), e3 = ex2(fmaf(s[3], sl, -mb1));
                    l_run[0] += e0 + e1; l_run[1] += e2 + e3;
                    __nv_bfloat162 p01 = __floats2bfloat162_rn(e0, e1), p23 = __floats2bfloat162_rn(e2, e3);
                    // accumulator layout of an 8-key tile = half of the A fragment of a 16-key step
                    pf[hf * 2] = *reinterpret_cast<uint32_t*>(&p01);
                    pf[hf * 2 + 1] = *reinterpret_cast<uint32_t*>(&p23);
                }
                if constexpr (SHARE) {
                    unsigned char* pr = sm + (Ks - Qs) + g * C::PP + kt * 32 + t4 * 4;
                    if (kt == 0) __syncwarp();       // (all lanes' keys have been read)
                    *reinterpret_cast<uint32_t*>(pr) = pf[0]; *reinterpret_cast<uint32_t*>(pr + 8 * C::PP) = pf[1];
                    *reinterpret_cast<uint32_t*>(pr + 16) = pf[2]; *reinterpret_cast<uint32_t*>(pr + 8 * C::PP + 16) = pf[3];
                } else {
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        uint32_t vf[4];
                        ldsm_x4_t(Vs + swz(kt * 16 + (lane & 7) + ((lane >> 3) & 1) * 8, v * 2 + (lane >> 4)), vf[0], vf[1], vf[2], vf[3]);
                        mma_bf16(acc[2 * v], pf, vf[0], vf[1]);
                        mma_bf16(acc[2 * v + 1], pf, vf[2], vf[3]);
                    }
                }
            }
        }
        if (!SHARE && (issued < nblk || (KG > 1 && blk + 1 == nblk))) __syncthreads();       // the stage is about to be overwritten (by a later block, or by the merge)
        if (issued < nblk) issue();
    }

    l_run[0] += __shfl_xor_sync(0xffffffffu, l_run[0], 1); l_run[1] += __shfl_xor_sync(0xffffffffu, l_run[1], 1);
    l_run[0] += __shfl_xor_sync(0xffffffffu, l_run[0], 2); l_run[1] += __shfl_xor_sync(0xffffffffu, l_run[1], 2);
    if constexpr (KG == 1) {
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const int r = mt * 16 + g + half * 8;
            if (r < nq) {
                const float inv = l_run[half] > 0.f ? 1.0f / l_run[half] : 0.f;
                bf16* o = a.out + (size_t)(r0 + r) * a.out_stride + h * 64 + t4 * 2;
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    *reinterpret_cast<__nv_bfloat162*>(o + j * 8) = __floats2bfloat162_rn(acc[j][half * 2] * inv, acc[j][half * 2 + 1] * inv);
            }
        }
    } else {
        [[maybe_unused]] float* mO = reinterpret_cast<float*>(Sp);       // [MT][KG][16 rows][72]
        if constexpr (SHARE) {
            // ---- every warp takes the probabilities of all groups, and of the values its own 64 / KG columns; the groups' shares are added in group order
            if (t4 == 0) { s_ml[kg][g] = make_float2(m_run[0], l_run[0]); s_ml[kg][g + 8] = make_float2(m_run[1], l_run[1]); }
            __syncthreads();
            const uint32_t Vb = St + KB * 128;
#pragma unroll
            for (int q = 0; q < KG; ++q) {
                if (q * KW >= nkmax) break;
#pragma unroll
                for (int kt = 0; kt < KW / 16; ++kt) {
                    uint32_t pf[4], vf[4];
                    ldsm_x4(St + q * KW * 128 + (lane & 15) * C::PP + kt * 32 + (lane >> 4) * 16, pf[0], pf[1], pf[2], pf[3]);
                    const int t = q * KW + kt * 16 + (lane & 15);
                    if constexpr (NJ == 1) {
                        asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];" : "=r"(vf[0]), "=r"(vf[1]) : "r"(Vb + swz(t, kg)));
                        mma_bf16(acc[q], pf, vf[0], vf[1]);
                    } else {
                        ldsm_x4_t(Vb + swz(t, kg * 2 + (lane >> 4)), vf[0], vf[1], vf[2], vf[3]);
                        mma_bf16(acc[q * NJ], pf, vf[0], vf[1]);
                        mma_bf16(acc[q * NJ + 1], pf, vf[2], vf[3]);
                    }
                }
            }
            float2 ma[KG], mb[KG];
            float m0 = -CUDART_INF_F, m1 = -CUDART_INF_F, den0 = 0.f, den1 = 0.f;
#pragma unroll
            for (int q = 0; q < KG; ++q) { ma[q] = s_ml[q][g]; mb[q] = s_ml[q][g + 8]; m0 = fmaxf(m0, ma[q].x); m1 = fmaxf(m1, mb[q].x); }
            float x[NJ][4];
#pragma unroll
            for (int j = 0; j < NJ; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) x[j][e] = 0.f;
#pragma unroll
            for (int q = 0; q < KG; ++q) {
                const float f0 = ma[q].x == -CUDART_INF_F ? 0.f : ex2((ma[q].x - m0) * sl), f1 = mb[q].x == -CUDART_INF_F ? 0.f : ex2((mb[q].x - m1) * sl);
                den0 = fmaf(ma[q].y, f0, den0); den1 = fmaf(mb[q].y, f1, den1);
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                    const float* t = acc[q * NJ + j];
                    x[j][0] = fmaf(t[0], f0, x[j][0]); x[j][1] = fmaf(t[1], f0, x[j][1]); x[j][2] = fmaf(t[2], f1, x[j][2]); x[j][3] = fmaf(t[3], f1, x[j][3]);
                }
            }
            const float inv0 = den0 > 0.f ? 1.0f / den0 : 0.f, inv1 = den1 > 0.f ? 1.0f / den1 : 0.f;
            bf16* o = a.out + (size_t)(r0 + g) * a.out_stride + h * 64 + kg * 8 * NJ + t4 * 2;
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                const __nv_bfloat162 p0 = __floats2bfloat162_rn(x[j][0] * inv0, x[j][1] * inv0), p1 = __floats2bfloat162_rn(x[j][2] * inv1, x[j][3] * inv1);
                if constexpr (ON > 0) {              // eight columns of the 16 rows, in place of the queries
                    *reinterpret_cast<__nv_bfloat162*>(sm + kg * 256 + g * 16 + t4 * 4) = p0;
                    *reinterpret_cast<__nv_bfloat162*>(sm + kg * 256 + (g + 8) * 16 + t4 * 4) = p1;
                } else {
                    if (g < nq) *reinterpret_cast<__nv_bfloat162*>(o + j * 8) = p0;
                    if (g + 8 < nq) *reinterpret_cast<__nv_bfloat162*>(o + (size_t)8 * a.out_stride + j * 8) = p1;
                }
            }
        } else {
            // ---- the key groups of a row tile meet in shared memory; each of its warps combines 64 / KG columns, in group order.  (Rows 72 floats apart: neither
            // the stores of the groups nor the loads across them meet in a bank.)
            float* mML = mO + MT * KG * 16 * 72;                         // [MT][KG][16 rows][maximum, sum]
            float* po = mO + (mt * KG + kg) * 16 * 72;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                *reinterpret_cast<float2*>(po + g * 72 + j * 8 + t4 * 2) = make_float2(acc[j][0], acc[j][1]);
                *reinterpret_cast<float2*>(po + (g + 8) * 72 + j * 8 + t4 * 2) = make_float2(acc[j][2], acc[j][3]);
            }
            if (t4 == 0) {
                float* ml = mML + (mt * KG + kg) * 32;
                ml[g * 2] = m_run[0]; ml[g * 2 + 1] = l_run[0];
                ml[(g + 8) * 2] = m_run[1]; ml[(g + 8) * 2 + 1] = l_run[1];
            }
            __syncthreads();
            constexpr int CW = 64 / KG;                                  // columns per warp; two lanes per row take four of every eight
            const int rr = lane >> 1, c0 = kg * CW + (lane & 1) * 4, r = mt * 16 + rr;
            float m = -CUDART_INF_F;
            float f[KG];
#pragma unroll
            for (int q = 0; q < KG; ++q) { f[q] = mML[(mt * KG + q) * 32 + rr * 2]; m = fmaxf(m, f[q]); }
            float den = 0.f;
#pragma unroll
            for (int q = 0; q < KG; ++q) {
                f[q] = (f[q] == -CUDART_INF_F) ? 0.f : ex2((f[q] - m) * sl);
                den = fmaf(mML[(mt * KG + q) * 32 + rr * 2 + 1], f[q], den);
            }
            const float inv = den > 0.f ? 1.0f / den : 0.f;
#pragma unroll
            for (int c = 0; c < CW; c += 8) {
                float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int q = 0; q < KG; ++q) {
                    const float4 t = *reinterpret_cast<const float4*>(mO + ((mt * KG + q) * 16 + rr) * 72 + c0 + c);
                    x.x = fmaf(t.x, f[q], x.x); x.y = fmaf(t.y, f[q], x.y); x.z = fmaf(t.z, f[q], x.z); x.w = fmaf(t.w, f[q], x.w);
                }
                __nv_bfloat162 p0 = __floats2bfloat162_rn(x.x * inv, x.y * inv), p1 = __floats2bfloat162_rn(x.z * inv, x.w * inv);
                const uint2 pk = make_uint2(*reinterpret_cast<uint32_t*>(&p0), *reinterpret_cast<uint32_t*>(&p1));
                if constexpr (ON > 0) *reinterpret_cast<uint2*>(sm + kg * 256 + lane * 8) = pk;          // eight columns of the 16 rows, in place of the queries
                else if (r < nq) *reinterpret_cast<uint2*>(a.out + (size_t)(r0 + r) * a.out_stride + h * 64 + c0 + c) = pk;
            }
        }
        if constexpr (ON > 0) {
            static_assert(KG == 8, "eight key groups: eight columns a warp");
            // the head's 64 columns, 2 KB, go to every CTA of the cluster as one copy, each issued by a warp of its own
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            cluster_wait();                          // every CTA of the cluster has begun and its barrier exists
            __syncthreads();                         // (all warps' columns are there; what the stages held is dead)
            if (warp < ON && lane == 0) {
                uint32_t ra, rb;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(oops + h * 2048), "r"(warp));
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rb) : "r"(smem_u32(&heads_bar)), "r"(warp));
                asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], 2048, [%2];"
                             ::"r"(ra), "r"(Qs), "r"(rb) : "memory");
            }
            __syncwarp();
            mbar_wait(smem_u32(&heads_bar), 0, &abort_s, oa.err_word, 12);
            __syncwarp();
            cluster_arrive_relaxed();                // this thread has seen what was sent to its CTA
            wo.template multiply<true>(oops, mO, warp, lane);
            __syncthreads();
            const float4 t = Proj64<OC::K>::sum(mO, tid);
            if ((tid >> 4) < nq)
                *reinterpret_cast<float4*>(oa.x_out + (size_t)(r0 + (tid >> 4)) * OC::K + h * 64 + (tid & 15) * 4) =
                    make_float4(t.x + ob.x + res.x, t.y + ob.y + res.y, t.z + ob.z + res.z, t.w + ob.w + res.w);
            cluster_wait();                          // nobody leaves while a copy from its shared memory may be under way
        }
    }
}

}  // namespace sd
