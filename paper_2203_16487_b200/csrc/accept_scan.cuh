// The acceptance rule alone on caller-provided logits [B, k+1, V] (Section 3.2, Eq. 7-9): one launch, no scratch memory.
//
// Bound: HBM latency, then bandwidth, over the rows up to the first rejected draft.  One thread-block cluster per sequence; the
// cluster's CTAs split a row's columns and the warps of a CTA take GR rows at once (W / GR warps to a row), so a lane keeps
// eight 16-byte loads in flight.  After each group of GR rows every warp sends its (max, argmax, count) to the
// cluster's shared memories, and behind one cluster barrier each CTA merges them and finds the first rejected draft by
// itself; the rows of later groups are never read.  32 x 26 x 32768 logits, launched from the Python binding one after the other: 1001 -> 22 us
// (one CTA per sequence, a row at a time, 4 bytes a load, before); 128 sequences: 1010 -> 47 us.
#pragma once
#include "barriers.cuh"
#include "kernels.cuh"

namespace sd {

__device__ __forceinline__ void as_take(RowPart& m, float x, int v, float ld) {
    if (x > m.mx || (x == m.mx && v < m.arg)) { m.mx = x; m.arg = v; }
    m.cnt += (x > ld) ? 1 : 0;
}

// grid = B x CL CTAs of W warps, clusters of CL along x; W a multiple of GR, GR <= 32 a power of two.
template <int CL, int GR, int W>
__global__ void __launch_bounds__(W * 32, 48 / W)
k_accept_scan(const float* __restrict__ logits, const int* __restrict__ draft, int k, int V, int beta, float tau,
              int* __restrict__ accepted, int* __restrict__ bif) {
    constexpr int WPR = W / GR;                  // warps per row
    __shared__ __align__(16) RowPart inbox[2][CL * WPR][GR];   // [group parity][sender][row]: the next group never overwrites what is being read
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    uint32_t rank = 0;
    if (CL > 1) asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    if (CL > 1) cluster_arrive();                // waited for before anything is sent: a peer's shared memory is there once the peer has begun
    const int b = blockIdx.x / CL, part = (int)rank * WPR + warp % WPR, parts = CL * WPR;
    // the draft of this warp's row in the next group is fetched a group ahead, so that its logit does not wait for it
    int tok_next = (warp / WPR < k) ? draft[b * k + warp / WPR] : -1;
    for (int c0 = 0, it = 0; c0 <= k; c0 += GR, ++it) {
        const int c = c0 + warp / WPR;                   // this warp's row
        const int tok = tok_next;
        tok_next = (c + GR < k) ? draft[b * k + c + GR] : -1;
        RowPart m; m.mx = -CUDART_INF_F; m.arg = 0x7fffffff; m.sum = 0.f; m.cnt = 0;
        float ld = CUDART_INF_F;
        if (c <= k) {
            const float* l = logits + ((size_t)b * (k + 1) + c) * V;
            if (c < k) ld = (tok >= 0 && tok < V) ? __ldg(l + tok) : -CUDART_INF_F;
            // 16-byte pieces between the unaligned ends of the row (V need not be a multiple of 4)
            const int head = min(V, (int)((16 - ((uintptr_t)l & 15)) & 15) >> 2);
            const int n4 = (V - head) >> 2, tail = head + n4 * 4;
            const float4* l4 = reinterpret_cast<const float4*>(l + head);
            const int per = (n4 + parts - 1) / parts, i0 = min(n4, part * per), i1 = min(n4, i0 + per);
            int i = i0 + lane;
            for (; i + 7 * 32 < i1; i += 8 * 32) {
                float4 x[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) x[u] = __ldcs(l4 + i + u * 32);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int v = head + (i + u * 32) * 4;
                    as_take(m, x[u].x, v, ld); as_take(m, x[u].y, v + 1, ld); as_take(m, x[u].z, v + 2, ld); as_take(m, x[u].w, v + 3, ld);
                }
            }
            for (; i < i1; i += 32) {
                const float4 x = __ldcs(l4 + i);
                const int v = head + i * 4;
                as_take(m, x.x, v, ld); as_take(m, x.y, v + 1, ld); as_take(m, x.z, v + 2, ld); as_take(m, x.w, v + 3, ld);
            }
            if (part == 0) {
                if (lane < head) as_take(m, l[lane], lane, ld);
                if (tail + lane < V) as_take(m, l[tail + lane], tail + lane, ld);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                RowPart q;
                q.mx = __shfl_xor_sync(0xffffffffu, m.mx, o);
                q.arg = __shfl_xor_sync(0xffffffffu, m.arg, o);
                q.cnt = __shfl_xor_sync(0xffffffffu, m.cnt, o);
                part_merge_nosum(m, q);
            }
        }
        m.sum = ld;                                      // (the unused field carries the draft's logit)
        RowPart* slot = &inbox[it & 1][part][warp / WPR];
        __syncwarp();
        if (CL > 1 && it == 0) cluster_wait();
        if (lane < CL) {                                 // one lane per peer
            if (CL == 1) *slot = m;
            else {
                uint32_t ra;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(smem_u32(slot)), "r"(lane));
                asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};"
                             ::"r"(ra), "r"(__float_as_uint(m.mx)), "r"(m.arg), "r"(__float_as_uint(m.sum)), "r"(m.cnt) : "memory");
            }
        }
        __syncwarp();
        if (CL > 1) tc_cluster_sync(); else __syncthreads();
        // every warp merges the group by itself: 32 / GR lanes per row, each over its share of the senders
        constexpr int LPR = 32 / GR;
        const int r = lane / LPR;
        RowPart t; t.mx = -CUDART_INF_F; t.arg = 0x7fffffff; t.sum = 0.f; t.cnt = 0;
#pragma unroll 2
        for (int p = lane % LPR; p < CL * WPR; p += LPR) { const RowPart q = inbox[it & 1][p][r]; part_merge_nosum(t, q); t.sum = q.sum; }
#pragma unroll
        for (int o = 1; o < LPR; o <<= 1) {
            RowPart q;
            q.mx = __shfl_xor_sync(0xffffffffu, t.mx, o);
            q.arg = __shfl_xor_sync(0xffffffffu, t.arg, o);
            q.cnt = __shfl_xor_sync(0xffffffffu, t.cnt, o);
            part_merge_nosum(t, q);
        }
        // (t.sum = the draft's logit: every sender of a row carries the same; lane 0 of the row has seen at least one)
        const bool stop = lane % LPR == 0 && c0 + r <= k && (c0 + r == k || !(t.cnt <= beta - 1 && (t.mx - t.sum) <= tau));
        const unsigned stops = __ballot_sync(0xffffffffu, stop);
        if (stops) {
            if (rank == 0 && warp == 0 && lane == __ffs(stops) - 1) { accepted[b] = c0 + r; bif[b] = t.arg; }
            break;
        }
    }
    // (a CTA may leave: its peers have sent everything that it read, and it sent everything before the last barrier)
}

template <int CL, int GR, int W>
inline cudaError_t as_launch_one(const float* logits, const int* draft, int B, int k, int V, int beta, float tau, int* acc, int* bif, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    if (CL > 8) {                                        // 16 CTAs are beyond the portable cluster size
        cudaError_t e = cudaFuncSetAttribute(k_accept_scan<CL, GR, W>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
    }
    cfg.gridDim = dim3((unsigned)B * CL); cfg.blockDim = dim3(W * 32); cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = CL > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k_accept_scan<CL, GR, W>, logits, draft, k, V, beta, tau, acc, bif);
}

// The split by size.  us between events around one launch, logits not in L2, a draft wrong once in seven, k = 25; the variants in the order of
// the rule (one CTA | 256 warps a sequence | 128 warps | 128 in small CTAs with groups of 8 rows), * = taken:
//   V = 1000    16 sequences  14* 12 10 14      64  16* 23 14 19     128  16* 40 20 31
//   V = 4096    16            18* 14 12 14      64  23* 25 16 21     128  23* 41 23 31
//   V = 8192    16  31 13* 12 16    32  32 19 14* 18    33  33 20 14 18*    64  33 29 21 25*    128  33 43 29 33*
//   V = 32768   16  94 21* 23 25    17  94 21 23* 25    27  96 29 27* 27    33  74 29 28 27*    64  96 45 42 35*    128  99 72 64 55*
//   V = 50265   16 147 25* 32 33    17 147 27 33* 35    27 147 37 37* 37    33 115 39 39 34*    64 150 60 61 53*    128 154 100 94 78*
// The wider the row, the longer 256 warps pay, until their CTAs (three of 16 warps to an SM) no longer run at once, from 28 sequences on; the
// groups of 8 read fewer rows past a rejection, which counts once memory is busy.  Short blocks prefer groups of 16 longer (k = 8, V = 32768:
// 64 sequences 53 35 27 31*).  Between neighbouring variants the lines cost at most 7 us where they are not best.
inline cudaError_t as_launch(const float* logits, const int* draft, int B, int k, int V, int beta, float tau, int* acc, int* bif, cudaStream_t st) {
    if (V <= 4096) return as_launch_one<1, 8, 16>(logits, draft, B, k, V, beta, tau, acc, bif, st);
    if (B <= 16) return as_launch_one<16, 16, 16>(logits, draft, B, k, V, beta, tau, acc, bif, st);
    if (B <= 32) return as_launch_one<8, 16, 16>(logits, draft, B, k, V, beta, tau, acc, bif, st);
    return as_launch_one<16, 8, 8>(logits, draft, B, k, V, beta, tau, acc, bif, st);
}

}  // namespace sd
