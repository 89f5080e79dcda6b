// Fast path of the sequence evaluator for C <= 2 copies per node (the paper's experiments all use
// C_v = 2, Section 4.3): one warp evaluates one sequence, warp-synchronously, with the graph staged
// once per block in shared memory.
//
// Representation.  Positions are 1-based and 16 bits wide.  Each node owns one 32-bit word with
// its two positions in any order; a node computed once holds the same position in both halves, an
// absent node holds 0.  A consumer reads both copies of a successor with one load.  Lane l of a
// warp works on the nodes with id = l (mod 32): a node's word then sits in bank l, so the lanes'
// reads of their own words never collide.  The nodes of each residue class are sorted by out-degree
// (descending); "half" j holds the j-th node of every class and a tile is two consecutive halves,
// so a lane treats two nodes per tile.  The successor lists are stored per tile as a dense
// [rows][32] matrix of 32-bit entries: entry (k, l) packs the byte offsets of the words of the
// k-th successor of lane l's two nodes, 16 bits each; rows = largest out-degree in the tile; a list that is used
// up continues with the node's own word, which is neutral for both reductions below.  A sink has
// one made-up successor: a word that holds the sequence length T, which keeps its last copy to
// the end.  Every lane of a warp runs the same trip count.  Node slots beyond the last node of a
// class own a constant word (1, 1) and carry m = w = 0, so they need no special case.
//
// Stages for one sequence seq[0..T) (paper: Section 2, Eqs. 1-8):
//   1. occurrence words   step t exchanges (t+1, t+1) into its node's word; if the word was taken,
//                         the previous low half is stored into the high half.  An id outside
//                         [0, n) lands in a spare word.  A third copy, or an id out of range,
//                         loses a position: the sequence is well-formed (Eq. 7, C_v) iff no word
//                         is zero and the number of words with two positions is T - n.
//   2. free steps         one lane per node u with copies a <= b (a = b if computed once), one pass
//                         over its successors' words r with two packed 16-bit reductions (both
//                         halves of r take part in both):
//                           Ga = max (r - a) mod 2^16   a successor copy before a (Eq. 5 violated)
//                                                       makes it 2^15 or more; otherwise a + Ga is
//                                                       the latest successor copy: b is kept until
//                                                       there (seeded with b - a: at least b);
//                           Gb = max (r - b) mod 2^16   ranks the copies below b above all others,
//                                                       in order: the latest successor copy inside
//                                                       (a, b), until which the first copy a is kept
//                                                       (Eqs. 2, 3, 5); seeded with a - b, so that
//                                                       without such a copy the result is a itself.
//   3. memory profile     delta[p] += m_u, delta[free+1] -= m_u, prefix sum (Eq. 4).
//   4. reductions         peak (Section 2), duration = sum_v w_v + sum over second copies (Eq. 1).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "moc_kernels.cuh"

namespace moc {

struct PairParams {
    int32_t n;
    int32_t n_tiles;           // tiles of 64 node slots (two halves of 32)
    int32_t max_T;             // C * n
    const void* rec;           // 64 * n_tiles node records (8 bytes for 32-bit sums, 16 for 64-bit), slot = half * 32 + lane
    const uint64_t* wslot;     // 64 * n_tiles, same slots: w | 1 << 48 | (C_v == 1) << 63
    const uint32_t* sell;      // successor tiles: byte offsets of the successor words of a lane's two nodes, 16 bits each
    int64_t base_dur;          // sum of all w
    int32_t small_w;           // sum of all w below 2^32
    const int32_t* seqs;
    const int32_t* lens;
    const int64_t* offs;       // exclusive prefix sum of the lengths, or nullptr: the kernel finds the rows itself
    int32_t B;
    int32_t per_block, spare;  // rows found by the kernel: block c takes per_block sequences, one more when c < spare
    int32_t team;              // kTeam: warps per sequence (a divisor of the block's warps)
    int64_t M;
    int64_t* out_peak;
    int64_t* out_dur;
    int32_t* out_status;
    // shared-memory layout, bytes (multiples of 16)
    uint32_t rec_bytes, w_bytes, sell_bytes;     // graph, once per block
    uint32_t word_bytes, delta_bytes;            // per sequence in flight; 16 bytes after the words hold the constant (1, 1)
    int32_t split;                               // 64-bit sums: position k of the high part of an amount (below)
};

// Node record: {byte offset of the node's word | x << 16, m}, where x is, in a tile's first half, the rows of the tile and, in its
// second, its first row in `sell` (which has fewer than 2^15); m takes 32 bits, or, for 64-bit
// sums, two words after a pad word: m mod 2^32 and m >> k.
//
// 64-bit sums without 64-bit atomics (which shared memory emulates with compare-and-swap loops: twice the time
// of the whole kernel).  A delta entry is two 32-bit words that are added to separately: the amounts mod 2^32, and the
// amounts >> k.  A sum S of deltas up to some step is a difference of two sets of resident outputs, at most
// 2 n of them each, so that with L and H the sums of the two words
//     S = 2^k H + (something below 2 n 2^k in absolute value),   S = L (mod 2^32),
// which determines S when 2 n 2^k <= 2^31: S = 2^k H + sign-extended (L - 2^k H mod 2^32).  H itself fits 32 bits when
// 2 sum(m) < 2^(31 + k); graphs beyond that (sum(m) >= 2^51 at n = 442) use the general kernels.
template <typename MemT> struct Amount { MemT v; };
template <> struct Amount<int64_t> { uint32_t lo, hi; };
__device__ __forceinline__ int64_t split_value(uint32_t lo, uint32_t hi, int32_t k) {
    return ((int64_t)(int32_t)hi << k) + (int32_t)(lo - (hi << k));
}
constexpr uint64_t kPairDurMask = (uint64_t(1) << 48) - 1;   // bits 0..47 of the summed wslot entries: w of the second copies
constexpr int kPairCntShift = 48;                             // bits 48..62: number of nodes with two copies

constexpr int kPairDeltaFront = 16;  // bytes in front of delta[0]: lands writes of absent nodes
constexpr int kPairWordTail = 16;    // bytes after the words: the word read by empty node slots

__device__ __forceinline__ int64_t warp_sum64(int64_t v) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, d);
    return v;
}
__device__ __forceinline__ int32_t warp_max_t(int32_t v) { return __reduce_max_sync(0xFFFFFFFFu, v); }
__device__ __forceinline__ int64_t warp_max_t(int64_t v) { return warp_max(v); }

// per-halfword unsigned max of two packed 16-bit pairs (one instruction on sm_90 and later)
__device__ __forceinline__ uint32_t max_u16x2(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("max.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ uint32_t min_u16x2(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("min.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ uint32_t swap_halves(uint32_t a) { return __byte_perm(a, 0, 0x1032); }

// ---- shared-memory accesses by 32-bit shared address
__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void sts_u16(uint32_t addr, uint32_t v) {
    asm volatile("st.shared.u16 [%0], %1;" ::"r"(addr), "h"((uint16_t)v) : "memory");
}
__device__ __forceinline__ uint32_t exch_shared(uint32_t addr, uint32_t v) {
    uint32_t old;
    asm volatile("atom.shared.exch.b32 %0, [%1], %2;" : "=r"(old) : "r"(addr), "r"(v) : "memory");
    return old;
}
__device__ __forceinline__ void red_add_shared(uint32_t addr, int32_t v) {
    asm volatile("red.shared.add.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void red_add_shared(uint32_t addr, int64_t v) {
    asm volatile("red.shared.add.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ void red_add_amount(uint32_t addr, Amount<int32_t> a) { red_add_shared(addr, a.v); }
__device__ __forceinline__ void red_sub_amount(uint32_t addr, Amount<int32_t> a) { red_add_shared(addr, -a.v); }
__device__ __forceinline__ void red_add_amount(uint32_t addr, Amount<int64_t> a) {
    red_add_shared(addr, (int32_t)a.lo);
    red_add_shared(addr + 4u, (int32_t)a.hi);
}
__device__ __forceinline__ void red_sub_amount(uint32_t addr, Amount<int64_t> a) {
    red_add_shared(addr, (int32_t)(0u - a.lo));
    red_add_shared(addr + 4u, (int32_t)(0u - a.hi));
}
// Free to move, for tables that do not change once they stand: its address comes from a base that went through
// MOC_STAGED, without which nothing would keep the read behind the barrier that the table arrives with.
__device__ __forceinline__ uint32_t lds_u32_nv(uint32_t addr) {
    uint32_t v;
    asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint4 lds_v4(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint64_t lds_u64(uint32_t addr) {
    uint64_t v;
    asm volatile("ld.shared.u64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void sts_u32(uint32_t addr, uint32_t v) {
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ int32_t lds_mem(uint32_t addr, int32_t) { return (int32_t)lds_u32(addr); }
__device__ __forceinline__ int64_t lds_mem(uint32_t addr, int64_t) { return (int64_t)lds_u64(addr); }
__device__ __forceinline__ void sts_mem(uint32_t addr, int32_t v) { sts_u32(addr, (uint32_t)v); }
__device__ __forceinline__ void sts_mem(uint32_t addr, int64_t v) {
    asm volatile("st.shared.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}

__device__ __forceinline__ uint2 lds_v2(uint32_t addr) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr) : "memory");
    return v;
}
// st.shared.u16 [addr], v  if old != 0
__device__ __forceinline__ void sts_u16_if_nonzero(uint32_t old, uint32_t addr, uint32_t v) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %0, 0;\n\t@q st.shared.u16 [%1], %2;\n\t}" ::"r"(old), "r"(addr),
                 "h"((uint16_t)v) : "memory");
}
// Makes a value opaque to the compiler at this point: it is then kept in its register instead of
// being recomputed from the kernel parameters wherever it is used (the hot loops are short of
// instruction slots, not of registers).
#define MOC_KEEP(x) asm volatile("" : "+r"(x))
// The same for the address of a table in shared memory, at the point from which the table may be read (behind the barrier).
#define MOC_STAGED(x) asm volatile("" : "+r"(x) : : "memory")


// Barrier of the warps that share a sequence.
template <bool kTeam>
__device__ __forceinline__ void team_sync(int id, int threads) {
    if constexpr (kTeam) asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
    else __syncwarp();
}

// Warps per block, at most.
__host__ __device__ constexpr int pair_max_warps(int pre, bool team) { return pre == 0 && !team ? 19 : 16; }

// Bound, large batches: the shared-memory data pipe (three quarters of one wavefront per clock, 528 wavefronts per
// sequence) and instruction issue (68 %, 1795 instructions per sequence); DRAM traffic equals the rows.  n = 442, B = 16384: 41.9 -> 41.6 us
// of kernel time (ncu, caches kept), 40.95 -> 40.4 to 40.95 us a launch back to back, by four exchanges in flight before their results
// are looked at, ragged ends of a row through the same code, no second search for the end of the row.  Bound, small
// batches: a chain of latencies; the division for a block's range, the sums of the lengths by shuffles and loops, and the copy
// of the graph behind one another were part of it (kernel time at n = 20, B = 1024 5.4 -> 4.7 us, where a call takes 5.8 to 6.1;
// a call at n = 442, B = 592 10.2 -> 7.3, n = 1000, B = 592 12.3 -> 8.4, these two with kTeam).
//
// kPre: how many 16-byte vectors of the next row each lane fetches ahead (rows of about 128*kPre
// steps; 0 for short rows, where the extra registers cost more than the wait).  Blocks have up to 16
// warps and two of them share an SM (62 registers per thread, no spills); without fetched rows 48 registers do, and 19
// warps (n = 250, B = 25000 44.5 -> 42.2 us; n = 442 without fetching, 38 warps on an SM 41.2, 28 with it 40.7).
//
// kTeam: p.team warps share a sequence, for batches that leave most of an SM's warps without one: the latency of a
// sequence is then what counts, and the row, the tiles and the scan are dealt to the warps.
template <typename MemT, int kPre, bool kTeam>
__global__ void __launch_bounds__(32 * pair_max_warps(kPre, kTeam), 2) eval_pair_kernel(const PairParams p) {
    static_assert(!kTeam || kPre == 0, "a team has one sequence at a time and fetches nothing ahead");
    extern __shared__ __align__(16) char smem[];
    __shared__ int64_t s_part[19];
    __shared__ uint64_t s_acc[16];               // kTeam: what the warps of a sequence tell one another
    __shared__ uint32_t s_flag[16], s_lo[16], s_hi[16];
    __shared__ int64_t s_top[16];
    constexpr uint32_t kRecB = sizeof(MemT) == 4 ? 8u : 16u;
    constexpr uint32_t kFull = 0xFFFFFFFFu;
    // ---- graph -> shared memory, once per block: records | durations | successor tiles.  Asynchronous copies: they
    // complete behind the search for the rows (a launch of few sequences is a chain of such latencies).
    const uint32_t graph_bytes = p.rec_bytes + p.w_bytes + p.sell_bytes;
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem);
    {
        auto copy = [&](uint32_t to, const void* from, uint32_t bytes) {
            for (uint32_t i = 16u * threadIdx.x; i < bytes; i += 16u * blockDim.x)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + i), "l"(reinterpret_cast<const char*>(from) + i) : "memory");
        };
        copy(sbase, p.rec, p.rec_bytes);
        copy(sbase + p.rec_bytes, p.wslot, p.w_bytes);
        copy(sbase + p.rec_bytes + p.w_bytes, p.sell, p.sell_bytes);
    }
    const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
    // broadcast from lane 0 so that the compiler knows the warp index is uniform across the warp
    const int warp = __shfl_sync(kFull, (int)(threadIdx.x >> 5), 0);
    // sequences in flight per block, this warp's, and its place among the warps of that one
    const int tw = kTeam ? p.team : 1, group = kTeam ? warp / tw : warp, wt = kTeam ? warp - group * tw : 0, groups = kTeam ? wpb / tw : wpb;
    const int tl = 32 * wt + lane, tn = 32 * tw;
    char* ws = smem + graph_bytes + (size_t)group * (p.word_bytes + kPairWordTail + p.delta_bytes);
    uint32_t* word = reinterpret_cast<uint32_t*>(ws);
    char* delta_base = ws + p.word_bytes + kPairWordTail;          // includes the front pad
    uint32_t wa = (uint32_t)__cvta_generic_to_shared(word);
    uint32_t da = (uint32_t)__cvta_generic_to_shared(delta_base) + kPairDeltaFront;  // &delta[0]
    uint32_t da1 = da - (uint32_t)sizeof(MemT);                                     // &delta[-1]
    // this lane's entries of the first tile: record, duration, successor row
    uint32_t rec0 = sbase + kRecB * (uint32_t)lane, w0 = sbase + p.rec_bytes + 8u * (uint32_t)lane,
             sell0 = sbase + p.rec_bytes + p.w_bytes + 4u * (uint32_t)lane;
    int n_tiles = p.n_tiles;
    MOC_KEEP(wa);
    MOC_KEEP(da);
    MOC_KEEP(da1);
    MOC_KEEP(rec0);
    MOC_KEEP(w0);
    MOC_KEEP(n_tiles);

    const int n = p.n;
    // Two ways to find the rows.  With p.offs (written by the offsets kernel) warps stride over the
    // whole batch.  Without it (p.offs == nullptr) block c takes a contiguous range: it adds up the lengths in
    // front of its range once, and every warp then walks the range with the lengths themselves -- no scratch,
    // no second kernel.
    const bool self = p.offs == nullptr;
    int b, b_end, b_step;
    int64_t off = 0;
    int32_t T = 0;
    // self mode: lanes 0..groups-1 hold the lengths of sequences b .. b+groups-1 (next: of the following ones)
    int32_t len_raw = 0, len_c0 = 0;
    uint64_t sum = 0;
    auto group_sum = [&](int32_t raw, int lanes) -> int64_t {   // sum of max(raw, 0) over lanes < `lanes`
        const uint32_t v = (lane < lanes && raw > 0) ? (uint32_t)raw : 0u;
        const uint32_t lo = __reduce_add_sync(kFull, v & 0xFFFFu), hi = __reduce_add_sync(kFull, v >> 16);
        return (int64_t)lo + ((int64_t)hi << 16);
    };
    if (!self) {
        b = blockIdx.x + gridDim.x * group;      // a batch smaller than the grid's warps spreads over all blocks
        b_end = p.B;
        b_step = gridDim.x * groups;
        if (b < b_end) { off = __ldg(&p.offs[b]); T = __ldg(&p.lens[b]); }
    } else {
        const int c0 = (int)blockIdx.x * p.per_block + min((int)blockIdx.x, p.spare);
        b_end = c0 + p.per_block + ((int)blockIdx.x < p.spare ? 1 : 0);
        b_step = groups;
        b = c0 + group;
        // lengths of the first sequences of the range (this warp starts at the group-th of them), and of those from b on
        len_c0 = (c0 + lane < p.B) ? __ldg(p.lens + c0 + lane) : 0;
        len_raw = (b + lane < p.B) ? __ldg(p.lens + b + lane) : 0;
        sum = lengths_before(p.lens, c0, threadIdx.x, blockDim.x);
    }
    // words and deltas are zero when a sequence begins: the words are cleared behind stage 2, the deltas by the scan
    auto clear = [&](uint32_t at, uint32_t bytes) {
        for (uint32_t i = 16u * (uint32_t)tl; i < bytes; i += 16u * (uint32_t)tn)
            asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(at + i), "r"(0) : "memory");
    };
    auto clear_deltas = [&]() { clear(da - kPairDeltaFront, p.delta_bytes); };   // all of them, with the front pad
    clear(wa, p.word_bytes);
    clear_deltas();
    if (tl == 0) sts_u32(wa + p.word_bytes, 0x00010001u);   // owned by empty node slots
    if (self) {
        sum = warp_sum_u59(sum);
        if (lane == 0) s_part[warp] = (int64_t)sum;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();                        // the graph is there, the state is zero, the sums of the warps stand
    MOC_STAGED(sell0);
    if (self) {
        off = (int64_t)warp_sum_u59(lane < wpb ? (uint64_t)s_part[lane] : 0) + group_sum(len_c0, group);
        T = __shfl_sync(kFull, len_raw, 0);
    }
    constexpr int kPerVec = 16 / (int)sizeof(MemT);  // delta entries per 16-byte vector
    constexpr int kShift = sizeof(MemT) == 4 ? 2 : 3;

    // Vector i of a row: its steps 4 i - a .. + 3, where steps outside the row count as the spare id n.
    auto fetch = [&](const int32_t* row, int32_t len, int t0) -> int4 {
        if (t0 >= 0 && t0 + 4 <= len) return __ldg(reinterpret_cast<const int4*>(row + t0));
        int4 v = make_int4(n, n, n, n);
        if (t0 >= 0) v.x = __ldg(row + t0);
        if (t0 + 1 >= 0 && t0 + 1 < len) v.y = __ldg(row + t0 + 1);
        if (t0 + 2 >= 0 && t0 + 2 < len) v.z = __ldg(row + t0 + 2);
        if (t0 + 3 >= 0 && t0 + 3 < len) v.w = __ldg(row + t0 + 3);
        return v;
    };
    // The first kPre 16-byte vectors per lane of the NEXT row are loaded into registers while the
    // current sequence is still being worked on, so that stage 1 does not wait for HBM.
    int4 pre[kPre > 0 ? kPre : 1];
    bool have_pre = false;
    while (b < b_end) {
        // fetch the next sequence's place early: its latency hides behind this sequence's work
        const int b_next = b + b_step;
        int64_t off_next = 0;
        int32_t T_next = 0, len_next = 0;
        if (!self) {
            if (b_next < b_end) { off_next = __ldg(&p.offs[b_next]); T_next = __ldg(&p.lens[b_next]); }
        } else {
            if (b_next < b_end) len_next = (b_next + lane < p.B) ? __ldg(p.lens + b_next + lane) : 0;
            off_next = off + group_sum(len_raw, groups);   // skip the sequences b .. b+groups-1
        }

        const bool use_pre = have_pre;   // pre[] holds this row only if the previous iteration fetched it
        have_pre = false;
        int64_t out_pk = -1, out_du = -1;
        int32_t out_st = -2;
        if (T >= n && T <= p.max_T) {
            const int nvec_d = (T + 2 + kPerVec - 1) / kPerVec;        // vectors covering delta[0..T+1]
            const int V = kTeam ? ((nvec_d + tn - 1) / tn) | 1 : ((nvec_d + 31) >> 5) | 1;      // vectors per lane, odd

            // ---- stage 1: occurrence words
            if (tl == 0) sts_u32(wa + 4u * (uint32_t)(n + 1), (uint32_t)T * 0x10001u);   // the made-up successor of sinks
            {
                const int32_t* row = p.seqs + off;
                const int a = (int)((reinterpret_cast<uintptr_t>(row) & 15) >> 2);
                const int nvec = (T + a + 3) >> 2;
                // ids outside [0, n) and steps outside the row go to the spare word n; the copy count exposes the former
                auto put4 = [&](int4 v, int t0) {
                    const uint32_t t1 = (uint32_t)(t0 + 1) * 0x10001u;
                    const uint32_t a0 = wa + 4u * min((uint32_t)v.x, (uint32_t)n), a1 = wa + 4u * min((uint32_t)v.y, (uint32_t)n),
                                   a2 = wa + 4u * min((uint32_t)v.z, (uint32_t)n), a3 = wa + 4u * min((uint32_t)v.w, (uint32_t)n);
                    const uint32_t o0 = exch_shared(a0, t1), o1 = exch_shared(a1, t1 + 0x10001u), o2 = exch_shared(a2, t1 + 0x20002u),
                                   o3 = exch_shared(a3, t1 + 0x30003u);
                    sts_u16_if_nonzero(o0, a0 + 2, o0);
                    sts_u16_if_nonzero(o1, a1 + 2, o1);
                    sts_u16_if_nonzero(o2, a2 + 2, o2);
                    sts_u16_if_nonzero(o3, a3 + 2, o3);
                };
                // (the first kPre vectors per lane may already be here)
#pragma unroll
                for (int j = 0; j < kPre; ++j) {
                    const int i = lane + 32 * j;
                    if (i < nvec) {
                        int4 v = pre[j];
                        if (!use_pre) v = fetch(row, T, 4 * i - a);
                        put4(v, 4 * i - a);
                    }
                }
                for (int i = tl + 32 * kPre; i < nvec; i += tn) put4(fetch(row, T, 4 * i - a), 4 * i - a);
            }
            team_sync<kTeam>(group + 1, tn);

            // request the next row now: the loads complete behind stages 2-4
            if (kPre > 0 && b_next < b_end) {
                const int64_t off_n = off_next;
                const int32_t T_n = self ? __shfl_sync(kFull, len_next, 0) : T_next;
                if (T_n >= n && T_n <= p.max_T) {
                    const int32_t* nrow = p.seqs + off_n;
                    const int an = (int)((reinterpret_cast<uintptr_t>(nrow) & 15) >> 2);
                    const int nvn = (T_n + an + 3) >> 2;
#pragma unroll
                    for (int j = 0; j < kPre; ++j) {
                        const int i = lane + 32 * j;
                        if (i < nvn) pre[j] = fetch(nrow, T_n, 4 * i - an);
                    }
                    have_pre = true;
                }
            }

            if (kPre == 0 && !kTeam && b_next < b_end) {
                // short rows are read in place; ask for the next one to be brought into L2 meanwhile
                const int64_t off_n = off_next;
                const int32_t T_n = self ? __shfl_sync(kFull, len_next, 0) : T_next;
                if (T_n >= n && T_n <= p.max_T) {
                    const char* nrow = reinterpret_cast<const char*>(p.seqs + off_n);
                    const int bytes = 4 * T_n;
                    for (int i = 128 * lane; i < bytes; i += 4096) asm volatile("prefetch.global.L2 [%0];" ::"l"(nrow + i));
                    if (lane == 31) asm volatile("prefetch.global.L2 [%0];" ::"l"(nrow + bytes - 4));
                }
            }

            // ---- stage 2 and the scatter of stage 3: two node slots per lane and tile
            uint32_t vmin = 0xFFFFFFFFu, depw = 0, capw = 0;
            uint64_t acc = 0;
            {
                uint32_t prec = rec0 + 64u * kRecB * (uint32_t)wt, pw = w0 + 512u * (uint32_t)wt, ps = sell0;
                // rows read in place and teams, where a sequence's latency shows: successor entries one row ahead (behind the last one
                // lies the state of a sequence).  n = 20, B = 1024 6.8 -> 6.0 us; with rows fetched ahead n = 353, B = 12000 28.8 -> 29.1.
                constexpr bool kAhead = kPre == 0;
                uint32_t e = kAhead ? lds_u32_nv(ps) : 0u;
                for (int d = wt; d < n_tiles; d += tw, prec += 64u * kRecB * (uint32_t)tw, pw += 512u * (uint32_t)tw) {
                    uint32_t ab[2], naa[2], nbb[2], Ga[2], Gb[2];
                    Amount<MemT> m[2];
                    int rows = 0;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        uint32_t x;
                        if constexpr (sizeof(MemT) == 4) {
                            const uint2 r = lds_v2(prec + 32u * kRecB * h);
                            x = r.x;
                            m[h].v = (MemT)r.y;
                        } else {
                            const uint4 r = lds_v4(prec + 32u * kRecB * h);
                            x = r.x;
                            m[h].lo = r.z;
                            m[h].hi = r.w;
                        }
                        if (h == 0) rows = (int)(x >> 16);
                        if (kTeam && h == 1) {
                            ps = sell0 + ((x >> 16) << 7);
                            e = lds_u32_nv(ps);               // (a team fetches no rows ahead)
                        }
                        const uint32_t own = lds_u32(wa + (x & 0xFFFFu));
                        vmin = min(vmin, own);
                        const uint32_t sw = swap_halves(own);
                        const uint32_t mn = min_u16x2(own, sw), mx = max_u16x2(own, sw);   // (a, a), (b, b)
                        ab[h] = __byte_perm(mn, mx, 0x7610);   // (a, b)
                        naa[h] = 0x00010000u - mn;             // (-a, -a) mod 2^16 for a >= 1
                        nbb[h] = 0x00010000u - mx;
                        Ga[h] = mx - mn;                       // (b - a, b - a)
                        Gb[h] = 0x00010000u - Ga[h];           // (a - b, a - b) mod 2^16 when a < b
                    }
                    // successors of the tile: the same trip count in every lane, used-up lists read the node's own word
#pragma unroll 2
                    for (int k = 0; k < rows; ++k) {
                        if (!kAhead) e = lds_u32(ps);
                        ps += 128u;
                        const uint32_t e_next = kAhead ? lds_u32_nv(ps) : 0u;
                        const uint32_t r0 = lds_u32(wa + (e & 0xFFFFu));
                        const uint32_t r1 = lds_u32(wa + (e >> 16));
                        e = e_next;
                        Ga[0] = __viaddmax_u16x2(r0, naa[0], Ga[0]);
                        Ga[1] = __viaddmax_u16x2(r1, naa[1], Ga[1]);
                        Gb[0] = __viaddmax_u16x2(r0, nbb[0], Gb[0]);
                        Gb[1] = __viaddmax_u16x2(r1, nbb[1], Gb[1]);
                    }
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        depw |= Ga[h];                         // bit 15 or 31: a successor copy before a
                        const uint32_t gg = max_u16x2(__byte_perm(Ga[h], Gb[h], 0x5410), __byte_perm(Ga[h], Gb[h], 0x7632));
                        const uint32_t v = gg + ab[h];                           // (end of b, end of a) mod 2^16
                        const uint32_t a16 = ab[h] & 0xFFFFu, b16 = ab[h] >> 16;
                        red_add_amount(da1 + (b16 << kShift), m[h]);
                        red_sub_amount(da + ((v & 0xFFFFu) << kShift), m[h]);
                        if (a16 != b16) {
                            red_add_amount(da1 + (a16 << kShift), m[h]);
                            red_sub_amount(da + ((v >> 16) << kShift), m[h]);
                            // bit 63 of the duration marks a node that may have one copy only (C_v = 1)
                            const uint64_t wx = lds_u64(pw + 256u * h);
                            capw |= (uint32_t)(wx >> 32);
                            acc += wx;
                        }
                    }
                }
            }
            vmin = __reduce_min_sync(kFull, vmin);
            // the low words add up without a carry when all durations together fit 32 bits
            uint64_t acc_all = p.small_w ? (uint64_t)__reduce_add_sync(kFull, (uint32_t)(acc >> 32)) << 32 | __reduce_add_sync(kFull, (uint32_t)acc)
                                         : (uint64_t)warp_sum64((int64_t)acc);
            bool cap_ok = !__any_sync(kFull, (int32_t)capw < 0), dep = __any_sync(kFull, (depw & 0x80008000u) != 0);
            if constexpr (kTeam) {
                if (lane == 0) {
                    s_acc[warp] = acc_all;
                    s_flag[warp] = (vmin == 0 ? 1u : 0u) | (cap_ok ? 0u : 2u) | (dep ? 4u : 0u);
                }
                team_sync<kTeam>(group + 1, tn);
                const bool in = lane < tw;
                const uint32_t f = __reduce_or_sync(kFull, in ? s_flag[group * tw + lane] : 0u);
                acc_all = (uint64_t)warp_sum64(in ? (int64_t)s_acc[group * tw + lane] : 0);
                vmin = f & 1u ? 0u : 1u;
                cap_ok = !(f & 2u);
                dep = (f & 4u) != 0;
            } else {
                __syncwarp();
            }
            clear(wa, p.word_bytes);
            const bool well_formed = cap_ok && vmin != 0 && (int)((acc_all >> kPairCntShift) & 0x7FFFu) == T - n;
            const int64_t dur_extra = (int64_t)(acc_all & kPairDurMask);
            if (!well_formed || dep) clear_deltas();

            if (!well_formed) {
                // status -2, sentinels already set
            } else if (dep) {
                out_st = -1;
                out_du = p.base_dur + dur_extra;
            } else {
                // ---- stage 3 + 4: prefix sum and running maximum; lane owns V consecutive vectors
                // One pass: the lane's running prefix and the largest prefix it sees; the largest
                // usage inside the lane's chunk is then (sum of the chunks before it) + that maximum.
                const int v0 = tl * V, v1 = kTeam ? min(v0 + V, nvec_d) : v0 + V;     // (a team's arrays end with the last vector)
                uint32_t d4 = da + 16u * (uint32_t)v0;
                MemT peak;
                uint32_t lo = 0, hi = 0;
                auto take = [&](uint32_t at) -> int4 {
                    const uint4 q = lds_v4(at);
                    asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(at), "r"(0) : "memory");
                    return make_int4((int)q.x, (int)q.y, (int)q.z, (int)q.w);
                };
                if constexpr (sizeof(MemT) == 4) {
                    MemT run = 0, top = INT32_MIN;
                    for (int j = v0; j < v1; ++j, d4 += 16u) {
                        const int4 q = take(d4);
                        run += q.x; top = max(top, run);
                        run += q.y; top = max(top, run);
                        run += q.z; top = max(top, run);
                        run += q.w; top = max(top, run);
                    }
                    lo = warp_inclusive_sum((uint32_t)run, lane);
                    peak = (MemT)(lo - (uint32_t)run) + top;
                    if (kTeam && v0 >= v1) peak = INT32_MIN;
                } else {
                    int64_t top = INT64_MIN;
                    uint32_t l = 0, h = 0;
                    for (int j = v0; j < v1; ++j, d4 += 16u) {
                        const int4 q = take(d4);
                        l += (uint32_t)q.x; h += (uint32_t)q.y;
                        const int64_t u = split_value(l, h, p.split);
                        l += (uint32_t)q.z; h += (uint32_t)q.w;
                        const int64_t w = split_value(l, h, p.split);
                        top = u > top ? u : top;
                        top = w > top ? w : top;
                    }
                    lo = warp_inclusive_sum(l, lane);
                    hi = warp_inclusive_sum(h, lane);
                    peak = split_value(lo - l, hi - h, p.split) + top;
                    if (kTeam && v0 >= v1) peak = INT64_MIN;
                }
                out_pk = (int64_t)warp_max_t(peak);
                if constexpr (kTeam) {
                    // the warp's largest usage counts from the usage in front of it
                    if (lane == 31) { s_lo[warp] = lo; s_hi[warp] = hi; s_top[warp] = out_pk; }
                }
                out_du = p.base_dur + dur_extra;
                out_st = 1;
            }
            team_sync<kTeam>(group + 1, tn);
            if constexpr (kTeam) {
                if (out_st == 1 && wt == 0) {
                    const bool in = lane < tw;
                    const uint32_t l = in ? s_lo[group * tw + lane] : 0u, h = in ? s_hi[group * tw + lane] : 0u;
                    const int64_t top = in ? s_top[group * tw + lane] : 0;
                    MemT front;
                    if constexpr (sizeof(MemT) == 4) front = (MemT)(warp_inclusive_sum(l, lane) - l);
                    else front = split_value(warp_inclusive_sum(l, lane) - l, warp_inclusive_sum(h, lane) - h, p.split);
                    // usages are 0 or more: a warp without vectors counts as 0
                    const bool has = in && top != (sizeof(MemT) == 4 ? (int64_t)INT32_MIN : INT64_MIN);
                    out_pk = (int64_t)warp_max_t(has ? (MemT)(front + (MemT)top) : (MemT)0);
                }
            }
            if (out_st == 1) out_st = out_pk <= p.M ? 1 : 0;
        }
        if (tl == 0) {
            p.out_peak[b] = out_pk;
            p.out_dur[b] = out_du;
            p.out_status[b] = out_st;
        }
        if (self) {
            len_raw = len_next;
            T_next = __shfl_sync(kFull, len_next, 0);
        }
        b = b_next;
        off = off_next;
        T = T_next;
    }
}

}  // namespace moc
