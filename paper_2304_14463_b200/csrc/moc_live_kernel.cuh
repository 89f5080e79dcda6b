// Evaluator for small graphs and large batches (n <= 128, C <= 4): a lane per sequence, walked from its last
// step to its first with the set of resident outputs as a bit mask in registers.
//
// Walking backwards turns the interval ends of Section 2 into liveness: a copy is resident from its own step to
// the last step that consumes it before its node is computed again (Eqs. 2, 3, 5), so that going backwards an
// output becomes live at the first consumer met and stops being live at the copy that serves it.  With
// L = the nodes live behind step t and v = seq[t]
//     usage(t) = m(L) + m({v} + preds(v) not in L)                        (Eq. 4)
//     L <- (L without v) + preds(v)
// and L starts as the sinks (results stay to the end).  A node still live in front of the first step has a
// consumer without an earlier copy (Eq. 5 violated).  No positions, no scatter, no prefix sum: one addition per
// copy and four bit operations per mask word and step, whatever C is.  Copies are counted bit-sliced: plane k holds the
// nodes with more than k copies; the sequence is well-formed iff plane 0 is full, the planes together hold T bits
// (no further copy) and no node exceeds its cap (Eq. 7, C_v).
//
// Memory.  A step looks up its node's predecessor mask and record, and m of the outputs that become live, at
// addresses the data decide.  The tables are replicated so that every lane has banks of its own (128 bytes per
// row), which makes those reads conflict-free; one block per SM holds them (66 KB at n = 128) and the sequence is
// read in place, 32 bytes per lane and eight steps, the next sixteen on their way (eight: 42.0 us at the size below).
//
// Latency.  A lane's steps follow one another, and a batch of 65536 is only 14 warps per SM.  So the part of a
// step that depends on the step before is kept to the mask operations; m of what becomes live is
// fetched without a branch, one set bit (two, three for fewer words) of every mask word at a time, an empty word reading
// a row of zeros.  The host deals the nodes to the words so that the predecessors of a node lie in
// different words where possible, and more bits than that are left to a loop that few steps need.  (A loop
// over the set bits of each word instead: 69 us at the size below, 1200 cycles per step.)
//
// n = 100, B = 65536, C = 2: 36.2 to 37.0 us (one launch) against 84 us for the warp-per-sequence kernel behind the offsets kernel.
// The range of a block from the host and sums by warp reductions instead of 64-bit divisions, shuffles and loops over the warps:
// kernel time 39.3 -> 37.2 us (ncu, caches kept), n = 34, B = 65536 15.8 -> 14.9, n = 46, B = 32100 16.1 -> 14.6.  Eight steps at a time instead of four: + 1.5.
// Bound: the integer pipe, about 87 warp instructions per step of 32 sequences (issue slots 65 %, ALU pipe 55 %), a fifth of them for bits beyond one per word.
// The warp-per-sequence kernel pays a warp's fixed costs (clearing, scans, reductions) per sequence, which a
// sequence of 120 steps does not repay; at n > 128 the masks outgrow the registers.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "moc_pair_kernel.cuh"

namespace moc {

constexpr int kLiveMaxN = 128;
constexpr int kLiveThreads = 512;   // 16 warps with up to 128 registers: two vectors of steps in flight per lane
constexpr int kLivePlanes = 4;     // C <= 4

struct LiveParams {
    int32_t n, C;
    int32_t B;
    int32_t per_block, spare;      // block c takes per_block groups of 32 sequences, one more when c < spare
    int64_t M;
    const uint4* image;            // the tables as they lie in shared memory (live_image)
    uint32_t sinks[kLiveMaxN / 32];
    int64_t sink_m;                // sum of m over the sinks
    uint32_t allow[kLivePlanes - 1][kLiveMaxN / 32];   // nodes that may have a 2nd, 3rd, 4th copy
    const int32_t* seqs;
    const int32_t* lens;
    const int64_t* offs;           // row offsets, or nullptr: packed rows, found from the lengths
    int64_t* out_peak;
    int64_t* out_dur;
    int32_t* out_status;
};

constexpr int kLiveWordRows = 33;  // rows of m per mask word: zero, then bit 0 .. 31

__host__ __device__ inline size_t live_smem_bytes(int32_t n, int words) { return ((size_t)(n + 1) * 3 + (size_t)words * kLiveWordRows) * 128; }

// The tables, 128 bytes a row: [node] mask of the node and its predecessors, [node] mask of the node, [node] (m, w),
// [word][1 + bit] m; the node rows n and the first row of a word are empty.  place[v] = mask word << 5 | bit of node v,
// preds: n rows of `words` words.
inline std::vector<uint32_t> live_image(int32_t n, int words, bool wide, const std::vector<int32_t>& place, const std::vector<uint32_t>& preds,
                                        const int64_t* m, const int64_t* w) {
    std::vector<uint32_t> t(live_smem_bytes(n, words) / 4, 0u);
    uint32_t *own = t.data() + (size_t)(n + 1) * 32, *mw = own + (size_t)(n + 1) * 32, *bit_m = mw + (size_t)(n + 1) * 32;
    for (int32_t v = 0; v < n; ++v) {
        const uint32_t word = (uint32_t)place[v] >> 5, bit = (uint32_t)place[v] & 31u;
        const uint32_t narrow[2] = {(uint32_t)m[v], (uint32_t)w[v]};
        const uint32_t full[4] = {(uint32_t)m[v], (uint32_t)((uint64_t)m[v] >> 32), (uint32_t)w[v], (uint32_t)((uint64_t)w[v] >> 32)};
        for (uint32_t i = 0; i < 32; ++i) {
            const uint32_t k = i & (uint32_t)(words - 1), mine = k == word ? 1u << bit : 0u;
            t[(size_t)v * 32 + i] = preds[(size_t)v * words + k] | mine;
            own[(size_t)v * 32 + i] = mine;
            mw[(size_t)v * 32 + i] = wide ? full[i & 3] : narrow[i & 1];
            bit_m[((size_t)word * kLiveWordRows + 1 + bit) * 32 + i] = full[wide ? i & 1 : 0];
        }
    }
    return t;
}

// Table reads: free to move between the steps (the tables do not change), as lds_u32_nv.
__device__ __forceinline__ uint2 live_lds_v2(uint32_t addr) {
    uint2 v;
    asm("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint4 live_lds_v4(uint32_t addr) {
    uint4 v;
    asm("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}

template <int W>
__device__ __forceinline__ void live_lds_words(uint32_t addr, uint32_t (&x)[W]) {
    if constexpr (W == 1) { x[0] = lds_u32_nv(addr); }
    else if constexpr (W == 2) { const uint2 v = live_lds_v2(addr); x[0] = v.x; x[1] = v.y; }
    else { const uint4 v = live_lds_v4(addr); x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w; }
}
// highest set bit, -1 without one
__device__ __forceinline__ int live_top_bit(uint32_t x) {
    int u;
    asm("bfind.u32 %0, %1;" : "=r"(u) : "r"(x));
    return u;
}

// W: mask words (n <= 32 W).  K: copy planes (C <= K).  SumT: int32_t when C * sum(m) and C * sum(w) are below 2^31.
template <typename SumT, int W, int K>
__global__ void __launch_bounds__(kLiveThreads, 1) eval_live_kernel(const LiveParams p) {
    extern __shared__ __align__(16) char smem[];
    __shared__ int64_t s_part[32];
    constexpr uint32_t kFull = 0xFFFFFFFFu;
    constexpr bool kWide = sizeof(SumT) == 8;
    constexpr int kPops = W == 4 ? 1 : (W == 2 ? 2 : 3);
    const int tid = threadIdx.x, lane = tid & 31, wpb = blockDim.x >> 5;
    const int warp = __shfl_sync(kFull, tid >> 5, 0);
    const int n = p.n;
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem);
    // ---- tables: asynchronous copies, complete behind the search for the rows
    {
        const int n16 = (int)(live_smem_bytes(n, W) / 16);
        for (int i = tid; i < n16; i += blockDim.x)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sbase + 16u * (uint32_t)i), "l"(p.image + i) : "memory");
    }
    uint32_t pa = sbase + (uint32_t)(4 * W * (lane % (32 / W)));                                  // this lane's column of each table
    uint32_t ra = sbase + (uint32_t)(n + 1) * 256u + (kWide ? 16u * (lane & 7) : 8u * (lane & 15));
    uint32_t ma = sbase + (uint32_t)(n + 1) * 384u + 128u + (kWide ? 8u * (lane & 15) : 4u * lane);    // row of bit 0 of word 0
    uint32_t own = (uint32_t)(n + 1) * 128u;                                                          // from a mask row to the node's own

    // ---- rows: block c takes a contiguous range of the groups of 32 consecutive sequences
    const int g_begin = (int)blockIdx.x * p.per_block + min((int)blockIdx.x, p.spare), g_end = g_begin + p.per_block + ((int)blockIdx.x < p.spare ? 1 : 0);
    int64_t base = 0;              // offset of the first row of the groups at hand
    if (p.offs == nullptr) {
        const uint64_t sum = warp_sum_u59(lengths_before<8>(p.lens, 32 * g_begin, tid, blockDim.x));
        if (lane == 0) s_part[warp] = (int64_t)sum;
        __syncthreads();
        base = (int64_t)warp_sum_u59(lane < wpb ? (uint64_t)s_part[lane] : 0);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    for (int g0 = g_begin; g0 < g_end; g0 += wpb) {
        const int b = 32 * (g0 + warp) + lane;
        const bool mine = g0 + warp < g_end && b < p.B;
        const int32_t len = mine ? __ldg(p.lens + b) : 0;
        int64_t off;
        if (p.offs == nullptr) {
            const int64_t l = max(len, 0), incl = warp_inclusive_sum(l, lane);
            __syncthreads();       // the last readers of s_part are done (and the tables stand)
            if (lane == 31) s_part[warp] = incl;
            __syncthreads();
            const uint64_t part = lane < wpb ? (uint64_t)s_part[lane] : 0;
            off = base + incl - l + (int64_t)warp_sum_u59(lane < warp ? part : 0);
            base += (int64_t)warp_sum_u59(part);
        } else {
            off = mine ? __ldg(p.offs + b) : 0;
            if (g0 == g_begin) __syncthreads();
        }
        MOC_STAGED(pa);                        // the tables are read behind the barrier
        MOC_STAGED(ra);
        MOC_STAGED(ma);
        MOC_STAGED(own);
        const int32_t T = (len >= n && (int64_t)len <= (int64_t)p.C * n) ? len : 0;
        // ---- the walk.  Vectors of four steps between 16-byte boundaries; steps outside the row count as the empty node n.
        const int32_t* row = p.seqs + off;
        const int a = (int)((reinterpret_cast<uintptr_t>(row) & 15) >> 2);
        auto fetch = [&](int i) -> int4 {       // steps 4 i - a .. + 3
            int4 v = make_int4(n, n, n, n);
            const int t0 = 4 * i - a;
            if (i >= 0 && t0 < T) {
                if (t0 >= 0 && t0 + 4 <= T) {
                    v = __ldg(reinterpret_cast<const int4*>(row + t0));
                } else {
                    if (t0 >= 0) v.x = __ldg(row + t0);
                    if (t0 + 1 >= 0 && t0 + 1 < T) v.y = __ldg(row + t0 + 1);
                    if (t0 + 2 >= 0 && t0 + 2 < T) v.z = __ldg(row + t0 + 2);
                    if (t0 + 3 >= 0 && t0 + 3 < T) v.w = __ldg(row + t0 + 3);
                }
            }
            return v;
        };
        uint32_t live[W], seen[K][W];
#pragma unroll
        for (int k = 0; k < W; ++k) {
            live[k] = p.sinks[k];
#pragma unroll
            for (int c = 0; c < K; ++c) seen[c][k] = 0;
        }
        SumT cur = (SumT)p.sink_m, peak = 0, dur = 0;
        auto m_of = [&](int u, int k) -> SumT {          // bit u of word k; u = -1: the word's row of zeros
            const uint32_t mu = ma + (uint32_t)(u * 128 + k * (kLiveWordRows * 128));
            if constexpr (kWide) { const uint2 y = live_lds_v2(mu); return (SumT)((uint64_t)y.x | (uint64_t)y.y << 32); }
            else return (SumT)lds_u32_nv(mu);
        };
        // Four steps, last one first.  What depends on the step before is two or three operations per mask word; the
        // table reads of the four steps, and then those of the outputs that become live, are in flight together.
        auto four = [&](const int4 q) {
            const int32_t id[4] = {q.w, q.z, q.y, q.x};
            uint32_t fresh[4][W], left[4];
            SumT mv[4], add[4];
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                // an id outside [0, n) and a filling step take the empty row n and set no bit
                const uint32_t v = min((uint32_t)id[s], (uint32_t)n);
                uint32_t pm[W], bit[W];            // the node with its predecessors, the node
                live_lds_words<W>(pa + v * 128u, pm);
                live_lds_words<W>(pa + v * 128u + own, bit);
                if constexpr (kWide) {
                    const uint4 x = live_lds_v4(ra + v * 128u);
                    mv[s] = (SumT)((uint64_t)x.x | (uint64_t)x.y << 32);
                    dur += (SumT)((uint64_t)x.z | (uint64_t)x.w << 32);
                } else {
                    const uint2 x = live_lds_v2(ra + v * 128u);
                    mv[s] = (SumT)x.x;
                    dur += (SumT)x.y;
                }
#pragma unroll
                for (int k = 0; k < W; ++k) {
#pragma unroll
                    for (int c = K - 1; c > 0; --c) seen[c][k] |= seen[c - 1][k] & bit[k];
                    seen[0][k] |= bit[k];
                    fresh[s][k] = pm[k] & ~live[k];
                    live[k] = (live[k] | pm[k]) & ~bit[k];
                }
            }
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                add[s] = 0;
                left[s] = 0;
#pragma unroll
                for (int k = 0; k < W; ++k) {
#pragma unroll
                    for (int z = 0; z < kPops; ++z) {
                        const int u = live_top_bit(fresh[s][k]);
                        add[s] += m_of(u, k);
                        if (z + 1 < kPops) fresh[s][k] &= ~(1u << (u & 31));
                    }
                    left[s] |= fresh[s][k] & (fresh[s][k] - 1u);          // more than the last one taken
                }
            }
            if (__any_sync(kFull, (left[0] | left[1] | left[2] | left[3]) != 0)) {
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    while (__any_sync(kFull, left[s] != 0)) {
                        left[s] = 0;
#pragma unroll
                        for (int k = 0; k < W; ++k) {
                            fresh[s][k] &= ~(1u << (live_top_bit(fresh[s][k]) & 31));      // taken already
                            add[s] += m_of(live_top_bit(fresh[s][k]), k);
                            left[s] |= fresh[s][k] & (fresh[s][k] - 1u);
                        }
                    }
                }
            }
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                cur += add[s];
                peak = cur > peak ? cur : peak;
                cur -= mv[s];
            }
        };
        // eight steps at a time (a 32-byte sector of the row), the next eight on their way
        int i = ((T + a + 3) >> 2) - 1;
        const int trips = (int)__reduce_max_sync(kFull, (unsigned)(T > 0 ? (i + 2) >> 1 : 0));
        int4 n1 = fetch(i), n0 = fetch(i - 1), f1 = fetch(i - 2), f0 = fetch(i - 3);
        i -= 2;
        for (int r = 0; r < trips; ++r) {
            const int4 q1 = n1, q0 = n0;
            n1 = f1;
            n0 = f0;
            i -= 2;
            f1 = fetch(i);
            f0 = fetch(i - 1);
            four(q1);
            four(q0);
        }
        if (mine) {
            int64_t pk = -1, du = -1;
            int32_t st = -2;
            if (T > 0) {
                uint32_t present = 0, total = 0, over = 0, missing = 0;
#pragma unroll
                for (int k = 0; k < W; ++k) {
                    present += __popc(seen[0][k]);
                    missing |= live[k];
#pragma unroll
                    for (int c = 0; c < K; ++c) total += __popc(seen[c][k]);
#pragma unroll
                    for (int c = 1; c < K; ++c) over |= seen[c][k] & ~p.allow[c - 1][k];
                }
                // every step that was not an invalid id set a bit of its own in some plane, or was one copy too many
                if (present == (uint32_t)n && total == (uint32_t)T && over == 0) {
                    du = (int64_t)dur;
                    st = -1;
                    if (missing == 0) {
                        pk = (int64_t)peak;
                        st = pk <= p.M ? 1 : 0;
                    }
                }
            }
            p.out_peak[b] = pk;
            p.out_dur[b] = du;
            p.out_status[b] = st;
        }
    }
}

}  // namespace moc
