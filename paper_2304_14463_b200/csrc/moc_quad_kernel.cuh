// Block-per-sequence path of the evaluator for up to four copies per node (the paper's cap C_v,
// Section 2; its experiments use 2, larger caps trade more recomputation for memory): a thread
// block evaluates one sequence at a time with the positions of a node's copies packed into one
// 64-bit word, so that a consumer reads all copies of a successor with one load and compares them
// two at a time with packed 16-bit arithmetic.
//
// Representation.  Positions are 1-based and 16 bits wide (sequences of at most 32766 steps: the packed
// comparisons tell earlier from later by the sign of a 16-bit difference).  After
// stage 1b a node's word holds its copies in order of arrival, and copies again in the quarters that are
// left, so that no quarter is empty; only the owner sorts them.
//
// Stages for one sequence seq[0..T) (paper: Section 2, Eqs. 1-8):
//   1a. occurrence words  step t takes the next free quarter of its node's word (a 16-bit counter per
//                         node, two counters per 32-bit atomic) and stores t + 1 there.
//   1b. per node          count in [1, min(C, C_v)] (Eq. 7 and the cap), duration of the further copies
//                         (Eq. 1); empty quarters filled; delta[p - 1] = m for every copy p ("+m at the copy's
//                         own step" of stage 3: a plain store, every step belongs to exactly one copy).
//   2.  free steps        one thread per node u with copies a_1 <= ... <= a_4, nodes taken in order of
//                         falling out-degree so that the lanes of a warp run about the same number of
//                         rounds; per successor word r (both halves, two packed operations each):
//                           G_0 = max (r - a_1) mod 2^16        2^15 or more: a successor copy before
//                                                               the first copy (Eq. 5 violated); else
//                                                               a_1 + G_0 is the latest successor copy,
//                                                               until which the last copy is kept;
//                           G_i = max (r - a_{i+1}) mod 2^16    ranks the successor copies below
//                                                               a_{i+1} above all others: the latest
//                                                               one inside (a_i, a_{i+1}), until which
//                                                               copy i is kept (Eqs. 2, 3, 5); seeded
//                                                               with a_i - a_{i+1}: else a_i itself.
//                         A sink's only successor is a made-up word that holds T in every quarter.
//   3.  memory profile    delta[free + 1] -= m_u per copy, prefix sum over the steps (Eq. 4).
//   4.  reductions        peak (Section 2), status against the budget.
//
// Stage 2 walks the successor tiles of the warp-per-sequence kernel (two node slots per lane, uniform trip counts, packed
// word offsets) where the graph has them, else a record per node with bounds tests.  Rows are found from the lengths (each
// block sums those in front of its range), or through `offs`.
//
// Who shares a sequence (quad_shape, from the size of the batch): a warp (kQuadWarps: large batches of graphs up to some 600 nodes), a
// team of warps (kQuadTeams), both with the graph copied into the block's shared memory once and several sequences in flight
// beside it, or the block (kQuadBlock: sequences whose state leaves no room for the graph, and large graphs).  Bound: instruction issue and
// the barriers between the stages (four per sequence: behind 1a, 1b, 2 and the prefix sum; the words are cleared for the next
// sequence behind stage 2); a small batch is a chain of latencies, of which a 64-bit division for the range of a
// block, sums of the lengths and of the chunks by shuffles and by loops over the warps (now warp reductions), the
// graph through L2 and three barriers were taken out.  n = 442, B = 148, C = 3 8.7 -> 6.2 us; n = 153, C = 3, B = 18944 68 -> 39 (a warp
// per sequence; a block of 64 threads spent most of its instructions on barriers and sums); n = 24 45 -> 21; n = 442, C = 3, B = 4736 33 -> 27 (teams of two);
// n = 2192, C = 2 (words of 32 bits), B = 1184 32.5 -> 24.9; n = 1000, C = 3, B = 4096 53.3 -> 45.3 (teams of four); n = 5000, B = 1024 80 -> 71.7 (one of 32); profile of n = 1000 8.2 -> 6.2, of n = 442 6.15 -> 5.6
// (no peak, no duration, first elements of the row requested before the state is clear).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "moc_pair_kernel.cuh"

namespace moc {

struct QuadParams {
    int32_t n;
    int32_t C;                 // 3 or 4 accumulators are compiled; C itself bounds the copy count
    int32_t max_T;             // C * n
    int32_t B;
    int32_t per_block, spare;  // rows found by the kernel: block c takes per_block sequences, one more when c < spare
    int64_t M;
    int32_t n_tiles, split, small_w;    // as in PairParams
    int32_t team;              // kQuadTeams: warps per sequence (a divisor of the block's warps; at most 16 teams)
    const void* rec;
    const uint32_t* sell;
    const int32_t* tile_row;   // first row of every tile in `sell`
    const uint64_t* wslot;     // durations by slot, as in PairParams
    uint32_t rec_bytes, w_bytes, sell_bytes, row_bytes;   // the block's copies of rec, wslot, sell and tile_row
    const uint4* order;        // without tiles: n records of 32 bytes in order of falling out-degree (below)
    const uint16_t* succ;      // ... and the successors beyond the eighth of the nodes that have more
    const void* m;             // n output sizes, int32 or int64
    const int64_t* w;          // n durations
    int64_t base_dur;          // sum of all w
    const int32_t* cap;        // n per-node caps, or nullptr
    const int32_t* seqs;
    const int32_t* lens;
    const int64_t* offs;       // B + 1 row offsets, or nullptr: the kernel finds the packed rows itself
    int64_t* out_peak;
    int64_t* out_dur;
    int32_t* out_status;
    int32_t single_len;        // profile: length of the one sequence at seqs[0..)
    int64_t* out_profile;      // ... usage per step, free step per step (may be null)
    int32_t* out_free;
    uint32_t word_bytes;       // 8 (n + 2) rounded to 32 (kAcc = 2: 4 (n + 2) rounded to 16), and 16 for the word of empty node slots
    uint32_t cnt_bytes;        // 2 (n + 2), rounded to 16
    uint32_t delta_bytes;      // the deltas, rounded to 16 (kChip: the graph follows them)
};

// Node record of `order`: word 0 = node | out-degree << 16 (a sink: 1, its successor the id n + 1), word 1 = index
// of its ninth successor in `succ`, words 4-7 = its first eight successor ids, 16 bits each.

__device__ __forceinline__ void sts_u64(uint32_t addr, uint64_t v) {
    asm volatile("st.shared.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ uint32_t atom_add_shared_u32(uint32_t addr, uint32_t v) {
    uint32_t old;
    asm volatile("atom.shared.add.u32 %0, [%1], %2;" : "=r"(old) : "r"(addr), "r"(v) : "memory");
    return old;
}

// Ascending sort of four 16-bit keys held as (k0, k1) in lo and (k2, k3) in hi: comparators (0,2)(1,3),
// (0,1)(2,3), (1,2), each on packed halves.
__device__ __forceinline__ void sort4_u16(uint32_t& lo, uint32_t& hi) {
    const uint32_t a = min_u16x2(lo, hi), b = max_u16x2(lo, hi);
    const uint32_t as = swap_halves(a), bs = swap_halves(b);
    const uint32_t a2 = __byte_perm(min_u16x2(a, as), max_u16x2(a, as), 0x7610);   // (min, max) of a
    const uint32_t b2 = __byte_perm(min_u16x2(b, bs), max_u16x2(b, bs), 0x7610);
    const uint32_t x = __byte_perm(a2, b2, 0x5432), y = swap_halves(x);            // (a2.hi, b2.lo) and swapped
    lo = __byte_perm(a2, min_u16x2(x, y), 0x5410);
    hi = __byte_perm(max_u16x2(x, y), b2, 0x7610);
}
__device__ __forceinline__ uint32_t max_halves(uint32_t v) { return max_u16x2(v, swap_halves(v)) & 0xFFFFu; }

__device__ __forceinline__ void quad_store(uint32_t addr, Amount<int32_t> a) { sts_u32(addr, (uint32_t)a.v); }
__device__ __forceinline__ void quad_store(uint32_t addr, Amount<int64_t> a) {
    asm volatile("st.shared.v2.u32 [%0], {%1,%2};" ::"r"(addr), "r"(a.lo), "r"(a.hi) : "memory");
}

// A node's word: four positions, or two where no node may have more (kAcc = 2).
template <int kAcc> struct QuadWord { uint2 v; };
template <> struct QuadWord<2> { uint32_t v; };
template <int kAcc>
__device__ __forceinline__ QuadWord<kAcc> quad_lds(uint32_t addr) {
    QuadWord<kAcc> r;
    if constexpr (kAcc == 2) r.v = lds_u32(addr);
    else r.v = lds_v2(addr);
    return r;
}

// The copies a_1 <= ... of one node and its running reductions over successor words.
template <int kAcc>
struct QuadNode {
    uint32_t base[kAcc], na[kAcc], G[kAcc];
    // own word after stage 1b
    __device__ __forceinline__ void open(QuadWord<kAcc> own) {
        uint32_t last;
        if constexpr (kAcc == 2) {
            const uint32_t x0 = own.v & 0xFFFFu, x1 = own.v >> 16;
            base[0] = min(x0, x1);
            base[1] = last = max(x0, x1);
        } else if constexpr (kAcc == 3) {          // the fourth quarter is a repetition
            const uint32_t x0 = own.v.x & 0xFFFFu, x1 = own.v.x >> 16, x2 = own.v.y & 0xFFFFu;
            const uint32_t lo = min(x0, x1), hi = max(x0, x1), mid = min(hi, x2);
            last = max(hi, x2);
            base[0] = min(lo, mid);
            base[1] = max(lo, mid);
            base[2] = last;
        } else {
            sort4_u16(own.v.x, own.v.y);
            base[0] = own.v.x & 0xFFFFu;
            base[1] = own.v.x >> 16;
            base[2] = own.v.y & 0xFFFFu;
            base[3] = last = own.v.y >> 16;
        }
#pragma unroll
        for (int j = 0; j < kAcc; ++j) na[j] = 0x00010000u - base[j] * 0x10001u;     // (-a, -a) mod 2^16
        G[0] = (last - base[0]) * 0x10001u;                                          // the last copy ends at itself at least
#pragma unroll
        for (int j = 1; j < kAcc; ++j) G[j] = ((base[j - 1] - base[j]) & 0xFFFFu) * 0x10001u;   // copy j ends at itself at least
    }
    __device__ __forceinline__ void visit(QuadWord<kAcc> r) {
#pragma unroll
        for (int j = 0; j < kAcc; ++j) {
            if constexpr (kAcc == 2) {
                G[j] = __viaddmax_u16x2(r.v, na[j], G[j]);
            } else {
                G[j] = __viaddmax_u16x2(r.v.x, na[j], G[j]);
                G[j] = __viaddmax_u16x2(r.v.y, na[j], G[j]);
            }
        }
    }
    // -m behind the end of every copy (and the ends themselves to `ends`, for a profile); returns a word whose bit 15
    // tells of a successor copy before a_1
    template <typename MemT, int kShift, bool kEnds>
    __device__ __forceinline__ uint32_t close(uint32_t da, Amount<MemT> m, int32_t* ends, bool real) {
        const uint32_t g0 = max_halves(G[0]), last = (base[0] + g0) & 0xFFFFu;
        red_sub_amount(da + (last << kShift), m);
        if (kEnds && real && !(g0 & 0x8000u)) ends[base[kAcc - 1] - 1] = (int32_t)last - 1;
#pragma unroll
        for (int j = 1; j < kAcc; ++j)
            if (base[j] != base[j - 1]) {                                       // copy j exists apart from copy j + 1
                const uint32_t end = (base[j] + max_halves(G[j])) & 0xFFFFu;
                red_sub_amount(da + (end << kShift), m);
                if (kEnds && real) ends[base[j - 1] - 1] = (int32_t)end - 1;
            }
        return g0;
    }
};

// Stage 1b for one node: c copies arrived in its word at `wv`; fills the empty places and writes +m at every copy.
template <typename MemT, int kAcc, int kShift>
__device__ __forceinline__ void quad_settle(uint32_t wv, uint32_t c, uint32_t dm1, Amount<MemT> mv) {
    if constexpr (kAcc == 2) {
        const uint32_t q = lds_u32(wv), x = c == 1 ? q * 0x10001u : q;
        if (c == 1) sts_u32(wv, x);
        quad_store(dm1 + ((x & 0xFFFFu) << kShift), mv);
        if (c > 1) quad_store(dm1 + ((x >> 16) << kShift), mv);
    } else {
        const uint2 q = lds_v2(wv);
        const uint32_t lo = c == 1 ? q.x * 0x10001u : q.x;
        const uint32_t hi = c < 3 ? lo : (c == 3 ? __byte_perm(q.y, q.x, 0x5410) : q.y);
        if (c < 4) sts_u64(wv, (uint64_t)lo | ((uint64_t)hi << 32));
        quad_store(dm1 + ((lo & 0xFFFFu) << kShift), mv);
        if (c > 1) quad_store(dm1 + ((lo >> 16) << kShift), mv);
        if (c > 2) quad_store(dm1 + ((hi & 0xFFFFu) << kShift), mv);
        if (kAcc > 3 && c > 3) quad_store(dm1 + ((hi >> 16) << kShift), mv);
    }
}
__device__ __forceinline__ uint32_t lds_u16(uint32_t addr) {
    uint32_t c;
    asm volatile("{\n\t.reg .u16 h;\n\tld.shared.u16 h, [%1];\n\tcvt.u32.u16 %0, h;\n\t}" : "=r"(c) : "r"(addr) : "memory");
    return c;
}

// kAcc: number of copies the node pass keeps apart (2, 3 or 4; C <= kAcc).
// kProfile: one sequence, whose usage per step and free steps are written out (moc_mem_profile).
// kMode: kQuadBlock  one sequence per block, the graph through L1
//        kQuadTeams  the block keeps a copy of the graph's tiles in shared memory; p.team warps share a sequence
//        kQuadWarps  the same with a warp per sequence
constexpr int kQuadBlock = 0, kQuadTeams = 1, kQuadWarps = 2;

template <typename MemT, int kAcc, bool kTiles, bool kProfile, int kMode>
__device__ __forceinline__ void quad_evaluate(const QuadParams& p) {
    constexpr bool kChip = kMode != kQuadBlock;
    static_assert(kTiles || !kChip, "only tiles are copied");
    extern __shared__ __align__(16) char smem[];
    __shared__ int64_t s_dur[32], s_top[32];
    __shared__ uint32_t s_lo[32], s_hi[32];
    constexpr int kShift = sizeof(MemT) == 4 ? 2 : 3;
    constexpr int kWord = kAcc == 2 ? 2 : 3;                // log2 of the bytes of a node's word
    constexpr uint32_t kFull = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31, block_warps = blockDim.x >> 5;
    const int block_warp = __shfl_sync(kFull, (int)threadIdx.x >> 5, 0);
    // sequences in flight per block, this warp's, and its place among the warps of that one
    const int n_warps = kMode == kQuadBlock ? block_warps : (kMode == kQuadTeams ? p.team : 1);
    const int group = kMode == kQuadBlock ? 0 : (kMode == kQuadTeams ? block_warp / n_warps : block_warp);
    const int groups = kMode == kQuadBlock ? 1 : (kMode == kQuadTeams ? block_warps / n_warps : block_warps);
    const int warp = kMode == kQuadWarps ? 0 : block_warp - group * n_warps, first_warp = group * n_warps;
    const int tid = 32 * warp + lane, nthr = 32 * n_warps;
    auto sync = [&]() {
        if constexpr (kMode == kQuadBlock) __syncthreads();
        else if constexpr (kMode == kQuadTeams) asm volatile("bar.sync %0, %1;" ::"r"(group), "r"(nthr) : "memory");
        else __syncwarp();
    };
    auto sync_or = [&](uint32_t x) -> bool {          // the same, and whether any thread of the sequence had x != 0
        if constexpr (kMode == kQuadBlock) return __syncthreads_or((int)x) != 0;
        else if constexpr (kMode == kQuadTeams) {
            uint32_t any;
            asm volatile("{\n\t.reg .pred a, b;\n\tsetp.ne.u32 a, %1, 0;\n\tbar.red.or.pred b, %2, %3, a;\n\tselp.u32 %0, 1, 0, b;\n\t}"
                         : "=r"(any) : "r"(x), "r"(group), "r"(nthr) : "memory");
            return any != 0;
        } else {
            const bool any = __any_sync(kFull, x != 0);
            __syncwarp();
            return any;
        }
    };
    int n = p.n;
    MOC_KEEP(n);
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem);
    // graph (kChip) | per sequence in flight: words | counters | delta[0..]
    const uint32_t recs = sbase, wsl = recs + p.rec_bytes, sells = wsl + p.w_bytes, rows = sells + p.sell_bytes;
    uint32_t wa = sbase + (kChip ? p.rec_bytes + p.w_bytes + p.sell_bytes + p.row_bytes : 0u) + (uint32_t)group * (p.word_bytes + p.cnt_bytes + p.delta_bytes);
    uint32_t ca = wa + p.word_bytes, da = ca + p.cnt_bytes;
    MOC_KEEP(wa);
    MOC_KEEP(ca);
    MOC_KEEP(da);
    const uint32_t dm1 = da - (uint32_t)sizeof(MemT);
    if constexpr (kChip) {
        // asynchronous copies: complete behind the search for the rows and, for one sequence, the arrival of its row
        auto copy = [&](uint32_t to, const void* from, uint32_t bytes) {
            for (uint32_t i = 16u * threadIdx.x; i < bytes; i += 16u * blockDim.x)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + i), "l"(reinterpret_cast<const char*>(from) + i) : "memory");
        };
        copy(recs, p.rec, p.rec_bytes);
        copy(wsl, p.wslot, p.w_bytes);
        copy(sells, p.sell, p.sell_bytes);
        copy(rows, p.tile_row, p.row_bytes);
    }
    auto amount = [&](int v) -> Amount<MemT> {       // m of node v in the form of the deltas
        Amount<MemT> a;
        if constexpr (sizeof(MemT) == 4) {
            a.v = __ldg(reinterpret_cast<const int32_t*>(p.m) + v);
        } else {
            const int64_t mv = __ldg(reinterpret_cast<const int64_t*>(p.m) + v);
            a.lo = (uint32_t)mv;
            a.hi = (uint32_t)(mv >> p.split);
        }
        return a;
    };
    // words and counters are zero when a sequence begins (stage 1b writes every delta that the prefix sum reads)
    auto clear = [&]() {
        const uint32_t nz = p.word_bytes + p.cnt_bytes;
        for (uint32_t i = 16u * (uint32_t)tid; i < nz; i += 16u * (uint32_t)nthr)
            asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(wa + i), "r"(0) : "memory");
    };

    // ---- rows: a block takes a contiguous range of the sequences, its teams in turn, or every grid-th one with the offsets given
    const bool self = !kProfile && p.offs == nullptr;
    int b = (int)blockIdx.x + (int)gridDim.x * group, b_end = p.B, b_step = (int)gridDim.x * groups;
    int64_t off = 0;
    // the lengths of b, b + 1 .. by lane (rows found by the kernel: what lies between this sequence and the team's next)
    int32_t T_next = 0, len_raw = 0, len_c0 = 0;
    uint32_t early[2] = {0u, 0u};        // kProfile: a thread's first elements of the row, requested before the state is clear
    auto lanes_sum = [&](int32_t raw, int lanes) -> int64_t {   // sum of max(raw, 0) over lanes < `lanes`
        const uint32_t v = (lane < lanes && raw > 0) ? (uint32_t)raw : 0u;
        const uint32_t lo = __reduce_add_sync(kFull, v & 0xFFFFu), hi = __reduce_add_sync(kFull, v >> 16);
        return (int64_t)lo + ((int64_t)hi << 16);
    };
    if (self) {
        const int c0 = (int)blockIdx.x * p.per_block + min((int)blockIdx.x, p.spare);
        b = c0 + group;
        b_end = c0 + p.per_block + ((int)blockIdx.x < p.spare ? 1 : 0);
        b_step = groups;
        if constexpr (kMode != kQuadBlock) {
            len_c0 = c0 + lane < p.B ? __ldg(p.lens + c0 + lane) : 0;
            len_raw = b + lane < p.B ? __ldg(p.lens + b + lane) : 0;
        } else {
            T_next = b < p.B ? __ldg(p.lens + b) : 0;
        }
        const uint64_t sum = lengths_before(p.lens, c0, threadIdx.x, blockDim.x);
        clear();
        const uint64_t part = warp_sum_u59(sum);
        if (lane == 0) s_dur[block_warp] = (int64_t)part;
        __syncthreads();
        off = (int64_t)warp_sum_u59(lane < block_warps ? (uint64_t)s_dur[lane] : 0);
        if constexpr (kMode != kQuadBlock) {
            off += lanes_sum(len_c0, group);
            T_next = __shfl_sync(kFull, len_raw, 0);
        }
    } else {
        T_next = kProfile ? p.single_len : (b < p.B ? __ldg(p.lens + b) : 0);      // one sequence ahead
        if constexpr (kProfile) {
#pragma unroll
            for (int k = 0; k < 2; ++k) early[k] = tid + k * nthr < T_next ? (uint32_t)__ldg(p.seqs + tid + k * nthr) : 0u;
        }
        clear();
        if (!kChip || kProfile) sync();
    }
    if constexpr (kChip && !kProfile) {          // (a profile waits for the graph behind the arrival of its row)
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
    }
    while (b < b_end) {
        const int32_t T = T_next;
        const int b_next = b + b_step;
        int64_t off_next = 0;
        if (kMode != kQuadBlock && self) {
            off_next = off + lanes_sum(len_raw, groups);
            if (b_next < b_end) len_raw = b_next + lane < p.B ? __ldg(p.lens + b_next + lane) : 0;
        } else if (!kProfile) {
            if (!self) off = __ldg(p.offs + b);
            if (b_next < b_end) T_next = __ldg(p.lens + b_next);
        }
        int64_t out_pk = -1, out_du = -1;
        int32_t out_st = -2;
        if (T >= n && T <= p.max_T) {      // uniform over the block
            // ---- stage 1a
            uint32_t flags = 0;
            {
                const int32_t* row = p.seqs + off;
                auto put = [&](uint32_t id, int t) {
                    if (id < (uint32_t)n) {
                        const uint32_t sh = (id & 1u) << 4;
                        const uint32_t k = (atom_add_shared_u32(ca + ((id >> 1) << 2), 1u << sh) >> sh) & 0xFFFFu;
                        if (k < (kAcc == 2 ? 2u : 4u)) sts_u16(wa + (id << kWord) + (k << 1), (uint32_t)t + 1u);
                    } else {
                        flags = 1;
                    }
                };
                int t = tid;
                if constexpr (kProfile) {
                    if (t < T) put(early[0], t);
                    if (t + nthr < T) put(early[1], t + nthr);
                    t += 2 * nthr;
                }
                for (; t + 3 * nthr < T; t += 4 * nthr) {      // four loads in flight per thread
                    const uint32_t i0 = (uint32_t)__ldg(row + t), i1 = (uint32_t)__ldg(row + t + nthr),
                                   i2 = (uint32_t)__ldg(row + t + 2 * nthr), i3 = (uint32_t)__ldg(row + t + 3 * nthr);
                    put(i0, t);
                    put(i1, t + nthr);
                    put(i2, t + 2 * nthr);
                    put(i3, t + 3 * nthr);
                }
                if (t < T) {                                   // up to three more
                    const bool h1 = t + nthr < T, h2 = t + 2 * nthr < T;
                    const uint32_t i0 = (uint32_t)__ldg(row + t), i1 = h1 ? (uint32_t)__ldg(row + t + nthr) : 0u,
                                   i2 = h2 ? (uint32_t)__ldg(row + t + 2 * nthr) : 0u;
                    put(i0, t);
                    if (h1) put(i1, t + nthr);
                    if (h2) put(i2, t + 2 * nthr);
                }
                if (tid == 0) {
                    // the made-up successor of sinks, and the word that empty node slots own
                    if constexpr (kAcc == 2) {
                        sts_u32(wa + ((uint32_t)(n + 1) << 2), (uint32_t)T * 0x10001u);
                        sts_u32(wa + p.word_bytes - 16u, 0x00010001u);
                    } else {
                        sts_u64(wa + ((uint32_t)(n + 1) << 3), (uint64_t)(uint32_t)T * 0x0001000100010001ull);
                        sts_u64(wa + p.word_bytes - 16u, 0x0001000100010001ull);
                    }
                }
            }
            if constexpr (kChip && kProfile) asm volatile("cp.async.wait_all;" ::: "memory");
            sync();
            // records and first successor row of a tile are requested while the tile before it (or stage 1b) is worked on
            uint4 r_next[2];
            const uint32_t* ps_next = nullptr;
            uint32_t ss_next = 0, e_first = 0;
            auto request = [&](int d) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int slot = (2 * d + h) * 32 + lane;
                    if constexpr (sizeof(MemT) == 4) {
                        const uint2 r = kChip ? lds_v2(recs + 8u * (uint32_t)slot) : __ldg(reinterpret_cast<const uint2*>(p.rec) + slot);
                        r_next[h].x = r.x;
                        r_next[h].z = r.y;
                    } else {
                        r_next[h] = kChip ? lds_v4(recs + 16u * (uint32_t)slot) : __ldg(reinterpret_cast<const uint4*>(p.rec) + slot);
                    }
                }
                if constexpr (kChip) {
                    ss_next = sells + 128u * lds_u32(rows + 4u * (uint32_t)d) + 4u * (uint32_t)lane;
                    e_first = lds_u32(ss_next);
                } else {
                    ps_next = p.sell + 32 * __ldg(p.tile_row + d) + lane;
                    e_first = __ldg(ps_next);
                }
            };
            if (kTiles && !kChip && warp < p.n_tiles) request(warp);
            // ---- stage 1b
            int64_t dur = 0;
            if constexpr (kChip) {
                const int n_halves = 2 * p.n_tiles;
                for (int hh = warp; hh < n_halves; hh += n_warps) {
                    const uint32_t slot = 32u * (uint32_t)hh + (uint32_t)lane;
                    uint32_t x;
                    Amount<MemT> mv;
                    if constexpr (sizeof(MemT) == 4) {
                        const uint2 r = lds_v2(recs + 8u * slot);
                        x = r.x & 0xFFFFu;
                        mv.v = (MemT)r.y;
                    } else {
                        const uint4 r = lds_v4(recs + 16u * slot);
                        x = r.x & 0xFFFFu;
                        mv.lo = r.z;
                        mv.hi = r.w;
                    }
                    const uint32_t wv = wa + (x << (kWord - 2));
                    if (wv == wa + p.word_bytes - 16u) continue;              // an empty slot
                    const uint32_t c = lds_u16(ca + (x >> 1));
                    uint32_t limit = (uint32_t)p.C;
                    if (p.cap != nullptr) limit = min(limit, (uint32_t)__ldg(p.cap + (x >> 2)));
                    if (c - 1u >= limit) {       // absent or overfull: its word holds no usable positions
                        flags |= 1;
                        continue;
                    }
                    if (c > 1) dur += (int64_t)(c - 1) * (int64_t)(lds_u64(wsl + 8u * slot) & kPairDurMask);
                    quad_settle<MemT, kAcc, kShift>(wv, c, dm1, mv);
                }
            } else {
                Amount<MemT> m_next = amount(min(tid, n - 1));          // one round ahead
                for (int v = tid; v < n; v += nthr) {
                    uint32_t limit = (uint32_t)p.C;
                    const uint32_t c = lds_u16(ca + 2u * (uint32_t)v);
                    if (p.cap != nullptr) limit = min(limit, (uint32_t)__ldg(p.cap + v));
                    const Amount<MemT> mv = m_next;
                    m_next = amount(min(v + nthr, n - 1));
                    if (c - 1u >= limit) {
                        flags |= 1;
                        continue;
                    }
                    if (c > 1) dur += (int64_t)(c - 1) * __ldg(p.w + v);
                    quad_settle<MemT, kAcc, kShift>(wa + ((uint32_t)v << kWord), c, dm1, mv);
                }
            }
            const bool malformed = sync_or(flags);
            bool dep = false;
            int64_t dw = 0;
            if (!malformed) {
                // ---- stage 2 and the scatter of stage 3
                uint32_t depw = 0;
                if constexpr (kTiles) {
                    if (kChip && warp < p.n_tiles) request(warp);
                    for (int d = warp; d < p.n_tiles; d += n_warps) {
                        QuadNode<kAcc> u[2];
                        Amount<MemT> m[2];
                        const uint32_t x0 = r_next[0].x, x1 = r_next[1].x;
                        const uint32_t* ps = ps_next;
                        uint32_t ss = ss_next, e_next = e_first;
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            if constexpr (sizeof(MemT) == 4) {
                                m[h].v = (MemT)r_next[h].z;
                            } else {
                                m[h].lo = r_next[h].z;
                                m[h].hi = r_next[h].w;
                            }
                            u[h].open(quad_lds<kAcc>(wa + ((r_next[h].x & 0xFFFFu) << (kWord - 2))));
                        }
                        if (d + n_warps < p.n_tiles) request(d + n_warps);
                        const int n_rows = __shfl_sync(kFull, (int)(x0 >> 16), 0);
                        for (int k = 0; k < n_rows; ++k) {
                            const uint32_t e = e_next;
                            ps += 32;
                            ss += 128u;
                            if (k + 1 < n_rows) e_next = kChip ? lds_u32(ss) : __ldg(ps);
                            const QuadWord<kAcc> r0 = quad_lds<kAcc>(wa + ((e & 0xFFFFu) << (kWord - 2))),
                                                 r1 = quad_lds<kAcc>(wa + ((e >> 16) << (kWord - 2)));
                            u[0].visit(r0);
                            u[1].visit(r1);
                        }
                        // an empty node slot owns the last word of the area: no step is its own
                        const uint32_t none = (p.word_bytes - 16u) >> (kWord - 2);
                        const bool real0 = !kProfile || (x0 & 0xFFFFu) != none, real1 = !kProfile || (x1 & 0xFFFFu) != none;
                        depw |= u[0].template close<MemT, kShift, kProfile>(da, m[0], p.out_free, real0 && p.out_free != nullptr);
                        depw |= u[1].template close<MemT, kShift, kProfile>(da, m[1], p.out_free, real1 && p.out_free != nullptr);
                    }
                } else {
                    const int n_round = (n + 31) & ~31;
                    for (int i = tid; i < n_round; i += nthr) {
                        uint32_t node = 0, deg = 0, e8 = 0;
                        uint4 inl = make_uint4(0, 0, 0, 0);
                        if (i < n) {
                            const uint4 r = __ldg(p.order + 2 * i);
                            inl = __ldg(p.order + 2 * i + 1);
                            node = r.x & 0xFFFFu;
                            deg = r.x >> 16;
                            e8 = r.y;
                        }
                        const int rounds = __reduce_max_sync(kFull, (int)deg);
                        QuadNode<kAcc> u;
                        u.open(quad_lds<kAcc>(wa + (node << kWord)));
                        const uint32_t in8[4] = {inl.x, inl.y, inl.z, inl.w};
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            if (k < rounds) {
                                if ((uint32_t)k < deg) u.visit(quad_lds<kAcc>(wa + (((k & 1) ? in8[k >> 1] >> 16 : in8[k >> 1] & 0xFFFFu) << kWord)));
                            }
                        }
                        for (int k = 8; k < rounds; ++k)
                            if ((uint32_t)k < deg) u.visit(quad_lds<kAcc>(wa + ((uint32_t)__ldg(p.succ + e8 + (k - 8)) << kWord)));
                        if (i < n) depw |= u.template close<MemT, kShift, kProfile>(da, amount((int)node), p.out_free, p.out_free != nullptr);
                    }
                }
                dep = sync_or(depw & 0x8000u);
                // per-warp sums of the durations, read behind the next barrier
                if constexpr (!kProfile) {
                    dw = p.small_w ? (int64_t)__reduce_add_sync(kFull, (uint32_t)dur) : warp_sum64(dur);
                    if (lane == 0) s_dur[first_warp + warp] = dw;
                }
            }
            if (b_next < b_end) clear();       // for the next sequence: nothing reads the words any more
            const int chunk = ((T + nthr - 1) / nthr) | 1;
            const int tb = min(tid * chunk, T), te = min(tb + chunk, T);
            uint32_t lo_in = 0, hi_in = 0;          // deltas of the warp's threads in front of this one
            MemT w_top = 0;
            if (!malformed && !dep) {
                // ---- stages 3 and 4: prefix sum, each thread a chunk of consecutive steps (odd length: no bank conflicts);
                // a warp's largest usage counts from the usage in front of the warp
                uint32_t ad = da + ((uint32_t)tb << kShift), lo = 0, hi = 0;
                MemT top = sizeof(MemT) == 8 ? (MemT)INT64_MIN : (MemT)INT32_MIN;
                for (int t = tb; t < te; ++t, ad += (uint32_t)sizeof(MemT)) {
                    MemT at;
                    if constexpr (sizeof(MemT) == 4) {
                        lo += lds_u32(ad);
                        at = (MemT)lo;
                    } else {
                        const uint2 q = lds_v2(ad);
                        lo += q.x;
                        hi += q.y;
                        at = split_value(lo, hi, p.split);
                    }
                    top = at > top ? at : top;
                }
                lo_in = warp_inclusive_sum(lo, lane);
                if constexpr (sizeof(MemT) == 8) hi_in = warp_inclusive_sum(hi, lane);
                if (lane == 31) {
                    s_lo[first_warp + warp] = lo_in;
                    s_hi[first_warp + warp] = hi_in;
                }
                lo_in -= lo;
                hi_in -= hi;
                if constexpr (!kProfile) {          // (a profile is asked for neither peak nor duration)
                    MemT before;
                    if constexpr (sizeof(MemT) == 4) before = (MemT)lo_in;
                    else before = split_value(lo_in, hi_in, p.split);
                    // a thread without steps counts nothing (the first step of the warp is one of the others', or the warp's usage in front)
                    w_top = warp_max_t(tb < te ? (MemT)(before + top) : (sizeof(MemT) == 8 ? (MemT)(INT64_MIN / 4) : (MemT)INT32_MIN));
                    if (lane == 0) s_top[first_warp + warp] = (int64_t)w_top;
                }
            }
            sync();
            if (kMode == kQuadWarps) {
                if (!malformed) {
                    out_du = p.base_dur + dw;
                    out_st = -1;
                    if (!dep) {
                        out_pk = (int64_t)w_top;
                        out_st = out_pk <= p.M ? 1 : 0;
                    }
                }
            } else if (!malformed) {
                if (!kProfile && warp == 0) out_du = p.base_dur + warp_sum64(lane < n_warps ? s_dur[first_warp + lane] : 0);
                out_st = -1;
                if (!dep) {
                    if (kProfile || warp == 0) {
                        // usage in front of every warp
                        uint32_t lo_w = lane < n_warps ? s_lo[first_warp + lane] : 0u, hi_w = lane < n_warps ? s_hi[first_warp + lane] : 0u;
                        const uint32_t lo_i = warp_inclusive_sum(lo_w, lane) - lo_w, hi_i = sizeof(MemT) == 8 ? warp_inclusive_sum(hi_w, lane) - hi_w : 0u;
                        if constexpr (kProfile) {
                            out_st = 1;
                        } else {
                            MemT in_front;
                            if constexpr (sizeof(MemT) == 4) in_front = (MemT)lo_i;
                            else in_front = split_value(lo_i, hi_i, p.split);
                            // a warp without steps holds the smallest value and stays below the others (which are usages, 0 or more)
                            const MemT pk = warp_max_t(lane < n_warps && s_top[first_warp + lane] > (sizeof(MemT) == 8 ? INT64_MIN / 4 : (int64_t)INT32_MIN)
                                                           ? (MemT)(in_front + (MemT)s_top[first_warp + lane]) : MemT(0));
                            out_pk = (int64_t)pk;
                            out_st = out_pk <= p.M ? 1 : 0;
                        }
                        if constexpr (kProfile) {
                            uint32_t lo = __shfl_sync(kFull, lo_i, warp) + lo_in, hi = __shfl_sync(kFull, hi_i, warp) + hi_in,
                                     ad = da + ((uint32_t)tb << kShift);
                            for (int t = tb; t < te; ++t, ad += (uint32_t)sizeof(MemT)) {
                                if constexpr (sizeof(MemT) == 4) {
                                    lo += lds_u32(ad);
                                    p.out_profile[t] = (int64_t)(MemT)lo;
                                } else {
                                    const uint2 q = lds_v2(ad);
                                    lo += q.x;
                                    hi += q.y;
                                    p.out_profile[t] = split_value(lo, hi, p.split);
                                }
                            }
                        }
                    }
                }
            }
        }
        if constexpr (kProfile) {
            if (tid == 0) p.out_status[0] = out_st;
            if (out_st < 0) {
                for (int t = tid; t < T; t += nthr) {
                    p.out_profile[t] = -1;
                    if (p.out_free) p.out_free[t] = -1;
                }
            }
            break;
        }
        if (tid == 0) {
            p.out_peak[b] = out_pk;
            p.out_dur[b] = out_du;
            p.out_status[b] = out_st;
        }
        if constexpr (kMode == kQuadBlock) {
            off += max(T, 0);
        } else if (self) {
            off = off_next;
            T_next = __shfl_sync(kFull, len_raw, 0);
        }
        b = b_next;
    }
    if constexpr (kChip && kProfile) asm volatile("cp.async.wait_all;" ::: "memory");      // nothing under way where no sequence was evaluated
}

// Blocks of up to 1024 threads leave 64 registers a thread.  Four copies kept apart need more: with 64-bit sums 52 bytes a
// thread are spilled for a block per sequence, 88 for teams and 116 for a warp per sequence (32-bit sums: 24 for teams; three
// copies, 64 bits: 12 to 24).
template <typename MemT, int kAcc, bool kTiles, bool kProfile, int kMode>
__global__ void __launch_bounds__(1024) eval_quad_kernel(const QuadParams p) {
    quad_evaluate<MemT, kAcc, kTiles, kProfile, kMode>(p);
}
// a warp per sequence: a module of its own
template <typename MemT, int kAcc>
__global__ void __launch_bounds__(1024) eval_quad_warp_kernel(const QuadParams p) {
    quad_evaluate<MemT, kAcc, true, false, kQuadWarps>(p);
}

}  // namespace moc
