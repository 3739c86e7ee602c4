// GEMM for passes of few activation rows (see rows_gemm.cuh for where it is used).
#include "attention.cuh"
#include "barriers.cuh"
#include "rows_gemm.cuh"

namespace sd {

__device__ __forceinline__ void rg_stamp(long long* trace, int slot) {
    if (trace && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) { long long t; asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t)); trace[slot] = t; }
}

constexpr int RG_WARPS = 8, RG_THREADS = RG_WARPS * 32;
template <int MT, int NT, int WN, int CS>
struct RgCfg {
    static constexpr int BM = 16 * MT, NB = 8 * NT, WK = RG_WARPS / WN, RP = NB + 8;     // RP: pitch of a partial row (floats)
    static constexpr size_t red_bytes = (size_t)WK * BM * RP * 4;
    static int kpad(int Kc) { return (Kc + 16 * WK - 1) / (16 * WK) * (16 * WK); }               // whole MMA steps for every K slice
    static size_t smem(int Kc, bool fragments = false) {
        size_t ops = (size_t)(BM + NB) * (kpad(Kc) * 2 + 16);
        if (fragments && (size_t)BM * (kpad(Kc) * 2 + 16) + red_bytes > ops) ops = (size_t)BM * (kpad(Kc) * 2 + 16) + red_bytes;
        return (ops > red_bytes ? ops : red_bytes) + (CS > 1 ? (size_t)BM * NB * 4 : 0);
    }
};

// One CTA = 16 MT rows x 8 NT columns, K walked by the warps side by side (WN warps across the columns, 8 / WN K slices).
//
// Bound: latency.  A decoding step of few rows is a chain of 39 launches, 24 of them these, each over 0.5-2 MB of weights, so what counts is the
// time from the predecessor's last store to this kernel's.  Hence:
//   * everything that does not depend on the predecessor -- the CTA's whole weight tile into shared memory, LayerNorm
//     parameters, cache rows -- is requested before the dependency wait;
//   * 256 threads of at most 80 registers (118 to 120 where a LayerNorm of 768 columns runs inside; with fragments see below) and 20-100 KB of shared memory, so that the next two kernels of the chain are resident
//     (their weights landed) while this one runs.  A 512-thread version with the weights in registers had shorter phases and a
//     longer step (240 against 218 us), because its successors could not start early;
//   * after the wait one round trip brings the rows; with NC > 0 they are normalised on the way (K = 128 NC, two rows per
//     warp: 1.3 us against 2.3 us when a cluster of 8 shared the normalised rows through distributed shared memory);
//   * where the reduction's length is one of the usual ones (ST > 0: ST MMA steps a warp) the weights have also become register fragments by then,
//     so that behind the rows there are only ST loads of A and the MMAs: shared memory handed over 96 KB a CTA before (0.39 of the 0.75 us between the
//     rows' arrival and the partial sums), 16 KB now, and the partial sums go where the weights were, without a barrier in between;
//   * K is split over the warps (and, for long reductions, over a cluster of CS CTAs whose partial tiles meet in the owner's
//     shared memory), the slices are added in a fixed order: results do not depend on timing.
// Measured inside a verify step at 26 rows: 2.8 us for QKV and FFN1 with their LayerNorm (3.5 with the weights read from shared memory behind the
// rows), 2.6 us for FFN2 (3.5); the step 145.1 -> 131, a greedy pass over 16 sequences 6262 -> 5680 us.  The fragments cost registers (up to 158 a
// thread, 768 columns 221): beyond three row tiles with a LayerNorm inside too few of the successors' CTAs are resident (52 rows: 154 / 161 us a step), those keep the variant without.
template <int EPI, int NC, int MT, int NT, int WN, int CS, int ST>
__global__ void __launch_bounds__(RG_THREADS, (NC > 0 && ST >= 8) || MT * ST > 16 ? 1 : NC > 4 || ST > 0 ? 2 : 3) k_rows(RowsArgs a) {
    using C = RgCfg<MT, NT, WN, CS>;
    constexpr int BM = C::BM, NB = C::NB, WK = C::WK, RP = C::RP, TN = NT / WN;      // TN = 8-column tiles per warp
    static_assert(TN % 2 == 0 || TN == 1, "B fragments come in pairs");
    static_assert(ST == 0 || TN > 1, "weights as fragments: column tiles in pairs");
    constexpr bool LN = NC > 0;
    extern __shared__ __align__(16) unsigned char rg_sm[];
    __shared__ int s_kv[BM];
    __shared__ __align__(16) float s_bias[NB];
    __shared__ __align__(8) uint64_t part_bar;
    __shared__ int abort_s;
    const GemmArgs<bf16>& g = a.g;
    const int K = LN ? NC * 128 : g.K, N = g.N, Kc = ST > 0 ? ST * 16 * WK : CS > 1 ? K / CS : K;
    const int Kp = (Kc + 16 * WK - 1) / (16 * WK) * (16 * WK), pitch = Kp * 2 + 16;                // Kp: padded with zeros; pitch in bytes
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    uint32_t rank = 0;
    if (CS > 1) asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int n0 = (CS > 1 ? (int)blockIdx.x / CS : (int)blockIdx.x) * NB, kb = (int)rank * Kc, m0 = blockIdx.y * BM;
    const int R = min((g.rows_static >= 0 ? g.rows_static : *g.n_rows) - m0, BM);
    if (R <= 0 && blockIdx.y > 0) return;
    const uint32_t As = smem_u32(rg_sm), Ws = As + BM * pitch;
    float* red = reinterpret_cast<float*>(rg_sm + (ST > 0 ? BM * pitch : 0));        // (in place of the operands; with fragments, of the weights)
    const size_t ops = ST > 0 ? BM * pitch + ((size_t)NB * pitch > C::red_bytes ? (size_t)NB * pitch : C::red_bytes) : (size_t)(BM + NB) * pitch;
    float* inbox = reinterpret_cast<float*>(rg_sm + (ops > C::red_bytes ? ops : C::red_bytes));     // CS > 1: [rank][BM][NB / CS]
    rg_stamp(a.trace, 0);
    // ---- before the dependency wait: weights, bias, LayerNorm parameters, cache rows
    const int cpr = Kp >> 3, cv = Kc >> 3;                    // 16-byte pieces per row, and those that hold values
    {
        int r = tid / cpr, c = tid % cpr;                     // one division; then walk
        const int dr = RG_THREADS / cpr, dc = RG_THREADS % cpr;
        const bf16* w = g.W + (size_t)n0 * K + kb;
        while (r < NB) {
            if (n0 + r < N && c < cv) cp_async16(Ws + r * pitch + c * 16, w + (size_t)r * K + c * 8);
            else *reinterpret_cast<uint4*>(rg_sm + (BM + r) * pitch + c * 16) = make_uint4(0, 0, 0, 0);
            r += dr; c += dc;
            if (c >= cpr) { c -= cpr; ++r; }
        }
        // The bias as well, in shared memory where registers are short: fetched where it is added, it cost 0.3 us at the end of every launch (verify step
        // of 26 rows 120.4 -> 117.3 us, of 104 rows 176 -> 171, greedy pass over 16 sequences 5570 -> 5280)
        if (ST == 0 && tid < NB / 4) {
            if (g.bias && n0 + tid * 4 < N) cp_async16(smem_u32(s_bias + tid * 4), g.bias + n0 + tid * 4);
            else *reinterpret_cast<float4*>(s_bias + tid * 4) = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    constexpr int ITEMS = BM * NB / 4, IPT = (ITEMS + RG_THREADS - 1) / RG_THREADS;                 // float4 outputs
    constexpr int OW = NB / CS, OITEMS = BM * OW / 4;                                               // ... that a rank owns
    static_assert(CS == 1 || (OW % 4 == 0 && OITEMS <= RG_THREADS), "ownership");
    float4 lgam[LN ? NC : 1], lbet[LN ? NC : 1];
    if (LN) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            lgam[c] = ldg_pinned(reinterpret_cast<const float4*>(a.ln_g + lane * 4 + c * 128));
            lbet[c] = ldg_pinned(reinterpret_cast<const float4*>(a.ln_b + lane * 4 + c * 128));
        }
    }
    // every float4 of outputs that a thread finishes lies in the same four columns
    const int bn = n0 + (CS > 1 ? (int)rank * OW + (tid % (OW / 4)) * 4 : (tid % (NB / 4)) * 4);
    float4 bzr = make_float4(0.f, 0.f, 0.f, 0.f);
    if (ST > 0 && g.bias && bn < N) bzr = ldg_pinned(reinterpret_cast<const float4*>(g.bias + bn));
    if (EPI == EPI_QKV && tid < BM) s_kv[tid] = tid < R ? (int)g.pg.row(g.seq[m0 + tid], g.pos[m0 + tid]) : 0;
    if (CS > 1) {
        if (tid == 0) {
            abort_s = 0;
            mbar_init(smem_u32(&part_bar), 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            mbar_expect_tx(smem_u32(&part_bar), (uint32_t)(CS - 1) * max(R, 0) * OW * 4);
        }
        tc_cluster_sync();                                    // every peer's barrier exists before anybody sends
    }
    rg_stamp(a.trace, 1);
    pdl_launch_dependents();
    const int wk = warp / WN, wn = warp % WN, steps = Kp / (16 * WK);
    // A: rows lane % 16, k half lane / 16.  B: with two column tiles, rows (lane & 7) + 8 (lane >> 4), k half (lane >> 3) & 1
    uint32_t ap = As + (lane & 15) * pitch + wk * steps * 32 + (lane >> 4) * 16;
    uint32_t bp = Ws + (wn * TN * 8 + (lane & 7) + (TN > 1 ? (lane >> 4) * 8 : 0)) * pitch + wk * steps * 32 + ((lane >> 3) & 1) * 16;
    uint32_t wf[ST > 0 ? ST : 1][TN][2];
    if constexpr (ST > 0) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
#pragma unroll
        for (int s = 0; s < ST; ++s)
#pragma unroll
            for (int j = 0; j < TN; j += 2) ldsm_x4(bp + s * 32 + j * 8 * pitch, wf[s][j][0], wf[s][j][1], wf[s][j + 1][0], wf[s][j + 1][1]);
    }
    pdl_wait();
    rg_stamp(a.trace, 2);
    // ---- activation rows
    if constexpr (LN) {
        constexpr int RW = BM / RG_WARPS;                     // rows per warp
        float4 xv[RW][NC];
#pragma unroll
        for (int s = 0; s < RW; ++s)
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const int m = warp + RG_WARPS * s;
                xv[s][c] = m < R ? *reinterpret_cast<const float4*>(a.ln_x + (size_t)(m0 + m) * K + lane * 4 + c * 128) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        float mu[RW], rs[RW];
#pragma unroll
        for (int s = 0; s < RW; ++s) {
            mu[s] = 0.f;
#pragma unroll
            for (int c = 0; c < NC; ++c) mu[s] += (xv[s][c].x + xv[s][c].y) + (xv[s][c].z + xv[s][c].w);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int s = 0; s < RW; ++s) mu[s] += __shfl_xor_sync(0xffffffffu, mu[s], o);
#pragma unroll
        for (int s = 0; s < RW; ++s) {
            mu[s] *= 1.0f / K; rs[s] = 0.f;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                xv[s][c].x -= mu[s]; xv[s][c].y -= mu[s]; xv[s][c].z -= mu[s]; xv[s][c].w -= mu[s];
                rs[s] = fmaf(xv[s][c].x, xv[s][c].x, rs[s]); rs[s] = fmaf(xv[s][c].y, xv[s][c].y, rs[s]);
                rs[s] = fmaf(xv[s][c].z, xv[s][c].z, rs[s]); rs[s] = fmaf(xv[s][c].w, xv[s][c].w, rs[s]);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int s = 0; s < RW; ++s) rs[s] += __shfl_xor_sync(0xffffffffu, rs[s], o);
#pragma unroll
        for (int s = 0; s < RW; ++s) {
            rs[s] = 1.0f / sqrtf(rs[s] * (1.0f / K) + a.ln_eps);
            const int m = warp + RG_WARPS * s;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const float4 v = xv[s][c];
                __nv_bfloat162 p0 = __floats2bfloat162_rn(fmaf(v.x * rs[s], lgam[c].x, lbet[c].x), fmaf(v.y * rs[s], lgam[c].y, lbet[c].y));
                __nv_bfloat162 p1 = __floats2bfloat162_rn(fmaf(v.z * rs[s], lgam[c].z, lbet[c].z), fmaf(v.w * rs[s], lgam[c].w, lbet[c].w));
                *reinterpret_cast<uint2*>(rg_sm + m * pitch + (lane * 4 + c * 128) * 2) =
                    m < R ? make_uint2(*reinterpret_cast<uint32_t*>(&p0), *reinterpret_cast<uint32_t*>(&p1)) : make_uint2(0u, 0u);
            }
        }
    } else {
        int r = tid / cpr, c = tid % cpr;
        const int dr = RG_THREADS / cpr, dc = RG_THREADS % cpr;
        const bf16* A = g.A + (size_t)m0 * g.lda + kb;
        while (r < BM) {
            if (r < R && c < cv) cp_async16(As + r * pitch + c * 16, A + (size_t)r * g.lda + c * 8);
            else *reinterpret_cast<uint4*>(rg_sm + r * pitch + c * 16) = make_uint4(0, 0, 0, 0);
            r += dr; c += dc;
            if (c >= cpr) { c -= cpr; ++r; }
        }
    }
    // residual values of this thread's outputs
    const int own_r = tid / (OW / 4), own_n = n0 + (int)rank * OW + (tid % (OW / 4)) * 4;               // CS > 1
    const bool mine = CS > 1 && tid < OITEMS && own_r < R && own_n < N;
    float4 own_x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (EPI == EPI_RESID && mine) own_x = *reinterpret_cast<const float4*>(g.resid + (size_t)(m0 + own_r) * N + own_n);
    float4 xo[IPT];
    if (EPI == EPI_RESID && CS == 1) {
#pragma unroll
        for (int i = 0; i < IPT; ++i) {
            const int o = tid + i * RG_THREADS, r = o / (NB / 4), n = n0 + (o % (NB / 4)) * 4;
            xo[i] = (o < ITEMS && r < R && n < N) ? *reinterpret_cast<const float4*>(g.resid + (size_t)(m0 + r) * N + n) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    rg_stamp(a.trace, 3);
    // ---- products: warp (wk, wn) takes K slice wk and TN column tiles of every row tile
    float acc[MT][TN][4];
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;
    if constexpr (ST > 0) {
#pragma unroll
        for (int s = 0; s < ST; ++s) {
            uint32_t af[MT][4];
#pragma unroll
            for (int i = 0; i < MT; ++i) ldsm_x4(ap + i * 16 * pitch + s * 32, af[i][0], af[i][1], af[i][2], af[i][3]);
#pragma unroll
            for (int i = 0; i < MT; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) mma_bf16(acc[i][j], af[i], wf[s][j][0], wf[s][j][1]);
        }
    } else {
#pragma unroll 8
        for (int s = 0; s < steps; ++s, ap += 32, bp += 32) {
            uint32_t af[MT][4], bf[TN][2];
#pragma unroll
            for (int i = 0; i < MT; ++i) ldsm_x4(ap + i * 16 * pitch, af[i][0], af[i][1], af[i][2], af[i][3]);
            if constexpr (TN == 1) asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];" : "=r"(bf[0][0]), "=r"(bf[0][1]) : "r"(bp));
            else {
#pragma unroll
                for (int j = 0; j < TN; j += 2) ldsm_x4(bp + j * 8 * pitch, bf[j][0], bf[j][1], bf[j + 1][0], bf[j + 1][1]);
            }
#pragma unroll
            for (int i = 0; i < MT; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) mma_bf16(acc[i][j], af[i], bf[j][0], bf[j][1]);
        }
        __syncthreads();                                      // the operands are dead: partial sums take their place
    }
    {
        const int gq = lane >> 2, t4 = lane & 3;
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) {
                float* p = red + (wk * BM + i * 16 + gq) * RP + (wn * TN + j) * 8 + t4 * 2;
                *reinterpret_cast<float2*>(p) = make_float2(acc[i][j][0], acc[i][j][1]);
                *reinterpret_cast<float2*>(p + 8 * RP) = make_float2(acc[i][j][2], acc[i][j][3]);
            }
    }
    __syncthreads();
    rg_stamp(a.trace, 4);
    // ---- fixed-order sum over the K slices, then the epilogue
    auto emit = [&](int r, int n, float4 v, float4 x) {
        const float4 bz = ST > 0 ? bzr : *reinterpret_cast<const float4*>(s_bias + (n - n0));
        v.x += bz.x; v.y += bz.y; v.z += bz.z; v.w += bz.w;
        if (EPI == EPI_RELU) { v.x = fmaxf(v.x, 0.f); v.y = fmaxf(v.y, 0.f); v.z = fmaxf(v.z, 0.f); v.w = fmaxf(v.w, 0.f); }
        if (EPI == EPI_GELU) { v.x = ffn_act(v.x, 1); v.y = ffn_act(v.y, 1); v.z = ffn_act(v.z, 1); v.w = ffn_act(v.w, 1); }
        if (EPI == EPI_RESID) {
            *reinterpret_cast<float4*>(g.resid + (size_t)(m0 + r) * N + n) = make_float4(x.x + v.x, x.y + v.y, x.z + v.z, x.w + v.w);
            return;
        }
        bf16* o = g.out + (size_t)(m0 + r) * g.ldo + n;
        if (EPI == EPI_QKV && n >= g.kv_d) {
            const size_t row = (size_t)s_kv[r] * g.kv_d;
            o = n < 2 * g.kv_d ? g.kc + row + (n - g.kv_d) : g.vc + row + (n - 2 * g.kv_d);
        }
        __nv_bfloat162 p0 = __floats2bfloat162_rn(v.x, v.y), p1 = __floats2bfloat162_rn(v.z, v.w);
        *reinterpret_cast<uint2*>(o) = make_uint2(*reinterpret_cast<uint32_t*>(&p0), *reinterpret_cast<uint32_t*>(&p1));
    };
#pragma unroll
    for (int i = 0; i < IPT; ++i) {
        const int o = tid + i * RG_THREADS;
        if (o >= ITEMS) break;
        const int r = o / (NB / 4), cn = (o % (NB / 4)) * 4;
        if (r >= R) continue;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int s = 0; s < WK; ++s) { const float4 t = *reinterpret_cast<const float4*>(red + (s * BM + r) * RP + cn); v.x += t.x; v.y += t.y; v.z += t.z; v.w += t.w; }
        if (CS == 1) { if (n0 + cn < N) emit(r, n0 + cn, v, xo[i]); }
        else {
            const uint32_t own = cn / OW;
            float* slot = inbox + ((int)rank * BM + r) * OW + cn % OW;
            if (own == rank) *reinterpret_cast<float4*>(slot) = v;
            else st_peer16(smem_u32(slot), smem_u32(&part_bar), own, make_uint4(__float_as_uint(v.x), __float_as_uint(v.y), __float_as_uint(v.z), __float_as_uint(v.w)));
        }
    }
    if (CS > 1) {
        __syncthreads();
        mbar_wait(smem_u32(&part_bar), 0, &abort_s, a.err_word, 8);
        if (mine) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int s = 0; s < CS; ++s) { const float4 t = *reinterpret_cast<const float4*>(inbox + (s * BM + own_r) * OW + (tid % (OW / 4)) * 4); v.x += t.x; v.y += t.y; v.z += t.z; v.w += t.w; }
            emit(own_r, own_n, v, own_x);
        }
    }
    rg_stamp(a.trace, 5);
}

template <int EPI, int NC, int MT, int NT, int WN, int CS, int ST = 0>
inline cudaError_t rg_launch_one(const RowsArgs& a, int rows_ub, bool pdl, cudaStream_t st) {
    using C = RgCfg<MT, NT, WN, CS>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((a.g.N + C::NB - 1) / C::NB * CS, (rows_ub + C::BM - 1) / C::BM); cfg.blockDim = dim3(RG_THREADS);
    cfg.dynamicSmemBytes = C::smem(a.g.K / CS, ST > 0); cfg.stream = st;       // (allowed by rg_init)
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (CS > 1) { attr[n].id = cudaLaunchAttributeClusterDimension; attr[n].val.clusterDim.x = CS; attr[n].val.clusterDim.y = 1; attr[n].val.clusterDim.z = 1; ++n; }
    if (pdl) { attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization; attr[n].val.programmaticStreamSerializationAllowed = 1; ++n; }
    cfg.attrs = attr; cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, k_rows<EPI, NC, MT, NT, WN, CS, ST>, a);
}

constexpr int RG_MAX_SMEM = 227 * 1024 - 1024;

// K slices (CTAs of a cluster) per output tile: reductions of 1024 and more are split (26 rows, K = 2048: 2 slices 180 us per verify step,
// 4 slices 186, 1 slice of 32 rows 186; 208 rows: 4 slices 284, 2 slices 304).
static int rg_split(int N, int K, int rows_ub, bool cluster) {
    if (K < 1024 || !cluster) return 1;
    if (rows_ub > rg_ln_rows(min(N, K)) && K % 32 == 0) return 4;
    return K % 16 == 0 ? 2 : 1;       // (the reductions whose weights become fragments take four: rg_launch_resid)
}
// 16-row tiles read the weights once more for every 16 rows, so they stop first; what counts is whether all CTAs are resident at once next to their
// predecessors' and successors', hence limits in CTAs per SM.  Width 512 (84 KB and 100 KB a CTA, two to an SM), verify step, us, tcgen05 tiles / 16 rows / 32 rows
// of the output projections: 208 rows 223 / 204 / 214, 312 rows 258 / 235 / 244, 416 rows 277 / 269 / 270, 520 rows 289 / 280 / 275, 624 rows 295 / 295 / 291.5, 832 rows
// 312 / 333 / 312; the QKV projection: 182 rows 203 / - / 195, 208 rows 204 / - / 199.6, 312 rows 235 / - / 245.  Width 768 (50 KB, 32 columns; 149 KB, one to an SM): 130
// rows 275 / 258 / 265, 156 rows 281 / 265 / 269, 208 rows 307 / 325 / 296, 312 rows 360 / 373 / 350, 364 rows 343 / - / 346.  The two encoders share the SMs (512: 144 rows
// 316 / 273, 200 rows 324 / 299; 768: 96 rows 203 / 193, 200 rows 270 / 260, 296 rows 303 / 314), so output projections with K = 512 stop sooner there: 16-row tiles at
// 7/8 CTA per SM (256 rows at 512 columns), 32-row ones at 5/9 (320 rows): 6 + 12 layers, whole tiles / 16 rows / 32 rows: 256 rows 186.5 / 185 / -, 260 rows 225 / 229.5 / 221, 288 rows 226 /
// 231 / 223, 320 rows 229 / - / 230, 360 rows 231 / - / 237.8, 512 rows 271.8 / - / 276, 560 rows 256.7 / - / 265.8.  They begin where the few-rows ones end, at 73 (768: 41) rows: from 97 on
// left whole tiles in between (512: 80 rows 165 / 145, 96 rows 167 / 148; 768: 60 rows 204 / 189).
int rg_frag_rows(int epi, int N, int K, int rows_ub, int n_sm, bool enc) {
    const bool resid = epi == EPI_RESID;
    if (N % 64 || !(K == 512 || (K == 768 && resid)) || rows_ub <= (enc ? rg_tile_rows_enc(min(N, K)) : K == 512 ? 96 : 80)) return 0;
    const long long sm = n_sm, t16 = (rows_ub + 15) / 16, t32 = (rows_ub + 31) / 32;
    if (resid && t16 * (K == 512 ? N / 64 : N / 32) <= (!enc ? K == 512 ? sm * 3 / 2 : sm * 5 / 3 : K == 512 ? sm * 7 / 8 : sm)) return 16;
    return t32 * (N / 64) <= (K == 512 ? (enc && resid ? sm * 5 / 9 : sm * 5 / 4) : enc ? sm * 2 / 3 : sm * 7 / 8) ? 32 : 0;
}
bool rg_supported(int epi, int N, int K, int lda, int rows_ub, bool cluster) {
    if (rows_ub > RG_MAX_ROWS || K % 16 || N % 16 || lda % 8) return false;
    if (epi != EPI_STORE && epi != EPI_RELU && epi != EPI_GELU && epi != EPI_RESID && epi != EPI_QKV) return false;
    const int Kc = K / (epi == EPI_RESID ? rg_split(N, K, rows_ub, cluster) : 1);
    return (int)RgCfg<2, 8, 2, 4>::smem(Kc) <= RG_MAX_SMEM;                     // (the largest tile any of the launches below uses)
}

// Tile shapes: 16 rows where the LayerNorm runs inside (each CTA repeats its rows' normalisation: few rows, wide column tiles), 32 rows
// beyond; columns so that a projection of a 512-wide model still spreads over 24-96 CTAs.
template <int EPI, int NC>
inline cudaError_t rg_launch_out(const RowsArgs& a, int rows_ub, int frag, bool pdl, cudaStream_t st) {
    const bool wide = a.g.N >= 1024;
    if constexpr (NC == 0) { if (frag) return rg_launch_one<EPI, 0, 2, 8, 2, 1, 8>(a, rows_ub, pdl, st); }
    // Weights as fragments.  One row tile: 32 columns a CTA (greedy pass over 16 sequences 6090 -> 5700 us; with two row tiles these are too many CTAs: one
    // sentence 902 -> 973); up to three: 64 columns (verify step, us, without / with: 26 rows 136.4 / 129.6, 44 rows 139.8 / 136.7, 52 rows 154 / 161).
    // 768 columns take 96 registers of fragments next to the 96 of the rows: 11 rows 190.6 / 183.6, 26 rows 195 / 201.5, 41 rows 205 / 212.
    if constexpr (NC == 2 || NC == 4) {
        if (wide && rows_ub <= 16) return rg_launch_one<EPI, NC, 1, 4, 1, 1, NC>(a, rows_ub, pdl, st);
        if (wide && rows_ub <= 48) return rg_launch_one<EPI, NC, 1, 8, 2, 1, 2 * NC>(a, rows_ub, pdl, st);
    }
    if constexpr (NC == 6) { if (wide && rows_ub <= 16) return rg_launch_one<EPI, NC, 1, 8, 2, 1, 2 * NC>(a, rows_ub, pdl, st); }
    if constexpr (NC == 0) { if (rows_ub > rg_ln_rows(min(a.g.N, a.g.K))) return rg_launch_one<EPI, 0, 2, 8, 2, 1>(a, rows_ub, pdl, st); }
    if (wide) return rg_launch_one<EPI, NC, 1, 8, 2, 1>(a, rows_ub, pdl, st);
    if constexpr (EPI == EPI_STORE) { if (rows_ub > 32) return rg_launch_one<EPI, NC, 1, 4, 1, 1>(a, rows_ub, pdl, st); }
    return rg_launch_one<EPI, NC, 1, 2, 1, 1>(a, rows_ub, pdl, st);
}
static cudaError_t rg_launch_resid(const RowsArgs& a, int rows_ub, int frag, bool cluster, bool pdl, cudaStream_t st) {
    if (frag && a.g.K == 512) return frag == 16 ? rg_launch_one<EPI_RESID, 0, 1, 8, 2, 1, 8>(a, rows_ub, pdl, st) : rg_launch_one<EPI_RESID, 0, 2, 8, 2, 1, 8>(a, rows_ub, pdl, st);
    if (frag) return frag == 16 ? rg_launch_one<EPI_RESID, 0, 1, 4, 1, 1, 6>(a, rows_ub, pdl, st) : rg_launch_one<EPI_RESID, 0, 2, 8, 2, 1, 12>(a, rows_ub, pdl, st);
    const int split = rg_split(a.g.N, a.g.K, rows_ub, cluster);
    if (rows_ub > rg_ln_rows(min(a.g.N, a.g.K))) {
        if (split == 4) return rg_launch_one<EPI_RESID, 0, 2, 8, 2, 4>(a, rows_ub, pdl, st);
        return rg_launch_one<EPI_RESID, 0, 2, 8, 2, 1>(a, rows_ub, pdl, st);
    }
    // Weights as fragments where K is one of these (verify step, us, without / with: K = 2048 26 rows 143 / 137.5 with two slices of 32 columns, 136.7 with
    // four of 64; 104 rows 188 / 184, 183; K = 3072 26 rows 194.9 / 190 with two slices, 195 with four; 63 rows 247 / 243.6; K = 512 52 rows 154 / 152).
    if (split == 2) {
        switch (a.g.K) {
            case 1024: return rg_launch_one<EPI_RESID, 0, 1, 4, 1, 2, 4>(a, rows_ub, pdl, st);
            case 2048: return rg_launch_one<EPI_RESID, 0, 1, 8, 2, 4, 8>(a, rows_ub, pdl, st);
            case 3072: return rg_launch_one<EPI_RESID, 0, 1, 4, 1, 2, 12>(a, rows_ub, pdl, st);
            default: return rg_launch_one<EPI_RESID, 0, 1, 4, 1, 2>(a, rows_ub, pdl, st);
        }
    }
    switch (split == 1 ? a.g.K : 0) {
#define RG_RESID(ST) return rows_ub > 32 ? rg_launch_one<EPI_RESID, 0, 1, 4, 1, 1, ST>(a, rows_ub, pdl, st) : rg_launch_one<EPI_RESID, 0, 1, 2, 1, 1, ST>(a, rows_ub, pdl, st)
        case 256: RG_RESID(2);
        case 512: RG_RESID(4);
        case 768: RG_RESID(6);
        default: RG_RESID(0);
#undef RG_RESID
    }
}
template <int EPI>
inline cudaError_t rg_launch_nc(const RowsArgs& a, int rows_ub, int frag, bool pdl, cudaStream_t st) {
    if (!a.ln_x) return rg_launch_out<EPI, 0>(a, rows_ub, frag, pdl, st);
    switch (a.g.K) {
        case 256: return rg_launch_out<EPI, 2>(a, rows_ub, 0, pdl, st);
        case 512: return rg_launch_out<EPI, 4>(a, rows_ub, 0, pdl, st);
        default: return rg_launch_out<EPI, 6>(a, rows_ub, 0, pdl, st);
    }
}
cudaError_t rg_launch(int epi, const RowsArgs& a, int rows_ub, int frag, bool cluster, bool pdl, cudaStream_t st) {
    switch (epi) {
        case EPI_STORE: return rg_launch_nc<EPI_STORE>(a, rows_ub, frag, pdl, st);
        case EPI_RELU: return rg_launch_nc<EPI_RELU>(a, rows_ub, frag, pdl, st);
        case EPI_GELU: return rg_launch_nc<EPI_GELU>(a, rows_ub, frag, pdl, st);
        case EPI_QKV: return rg_launch_nc<EPI_QKV>(a, rows_ub, frag, pdl, st);
        default: return rg_launch_resid(a, rows_ub, frag, cluster, pdl, st);
    }
}


// Shared-memory limits of everything launched above.  The limit belongs to the kernel in the whole process: one that followed the launch would
// be another handle's by the time of the launch, if that handle decodes on another host thread.
template <int EPI, int NC, int MT, int NT, int WN, int CS, int ST = 0>
static void rg_room(cudaError_t& e) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_rows<EPI, NC, MT, NT, WN, CS, ST>, cudaFuncAttributeMaxDynamicSharedMemorySize, RG_MAX_SMEM);
}
template <int EPI, int NC>
static void rg_room_out(cudaError_t& e) {
    if constexpr (NC == 0) { rg_room<EPI, 0, 2, 8, 2, 1>(e); rg_room<EPI, 0, 2, 8, 2, 1, 8>(e); }
    if constexpr (NC == 2 || NC == 4) rg_room<EPI, NC, 1, 4, 1, 1, NC>(e);
    if constexpr (NC > 0) rg_room<EPI, NC, 1, 8, 2, 1, 2 * NC>(e);
    rg_room<EPI, NC, 1, 8, 2, 1>(e);
    if constexpr (EPI == EPI_STORE) rg_room<EPI, NC, 1, 4, 1, 1>(e);
    rg_room<EPI, NC, 1, 2, 1, 1>(e);
}
template <int EPI>
static void rg_room_nc(cudaError_t& e) { rg_room_out<EPI, 0>(e); rg_room_out<EPI, 2>(e); rg_room_out<EPI, 4>(e); rg_room_out<EPI, 6>(e); }
cudaError_t rg_init() {
    cudaError_t e = cudaSuccess;
    rg_room_nc<EPI_STORE>(e); rg_room_nc<EPI_RELU>(e); rg_room_nc<EPI_GELU>(e); rg_room_nc<EPI_QKV>(e);
    rg_room<EPI_RESID, 0, 1, 8, 2, 1, 8>(e); rg_room<EPI_RESID, 0, 2, 8, 2, 1, 8>(e); rg_room<EPI_RESID, 0, 2, 8, 2, 1, 12>(e);
    rg_room<EPI_RESID, 0, 2, 8, 2, 4>(e); rg_room<EPI_RESID, 0, 2, 8, 2, 1>(e); rg_room<EPI_RESID, 0, 1, 4, 1, 2>(e);
    rg_room<EPI_RESID, 0, 1, 4, 1, 2, 4>(e); rg_room<EPI_RESID, 0, 1, 8, 2, 4, 8>(e); rg_room<EPI_RESID, 0, 1, 4, 1, 2, 12>(e);
    rg_room<EPI_RESID, 0, 1, 4, 1, 1>(e); rg_room<EPI_RESID, 0, 1, 4, 1, 1, 2>(e); rg_room<EPI_RESID, 0, 1, 4, 1, 1, 4>(e); rg_room<EPI_RESID, 0, 1, 4, 1, 1, 6>(e);
    rg_room<EPI_RESID, 0, 1, 2, 1, 1>(e); rg_room<EPI_RESID, 0, 1, 2, 1, 1, 2>(e); rg_room<EPI_RESID, 0, 1, 2, 1, 1, 4>(e); rg_room<EPI_RESID, 0, 1, 2, 1, 1, 6>(e);
    return e;
}

}  // namespace sd
