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
// word offsets; read through L1, a block has no room for a copy) where the graph has them, else a record per node
// with bounds tests.  Rows are found from the lengths (each block sums those in front of its range), or through `offs`.
// The kernel is bound by instruction issue and by the barriers between its stages; the threads per sequence
// follow the batch (quad_shape).  n = 1000, C = 3, B = 4096: 60.5 -> 53.3 us (issue slots 61 % busy, shared-memory data
// pipe 47 %); n = 5000, C = 3, B = 1024: 93 -> 81 us; n = 442, C = 3, B = 64: 12.4 -> 8.3 us (before: rows through the
// offsets kernel, every word sorted, a fixed number of threads).
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
    int64_t M;
    int32_t n_tiles, split;    // as in PairParams
    const void* rec;
    const uint32_t* sell;
    const int32_t* tile_row;   // first row of every tile in `sell`
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
    uint32_t word_bytes;       // 8 (n + 2) rounded to 32, and 16 for the word of empty node slots
    uint32_t cnt_bytes;        // 2 (n + 2), rounded to 16
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

// The copies a_1 <= ... of one node and its running reductions over successor words.
template <int kAcc>
struct QuadNode {
    uint32_t base[kAcc], na[kAcc], G[kAcc];
    // own word after stage 1b
    __device__ __forceinline__ void open(uint2 own) {
        uint32_t last;
        if constexpr (kAcc == 3) {          // the fourth quarter is a repetition
            const uint32_t x0 = own.x & 0xFFFFu, x1 = own.x >> 16, x2 = own.y & 0xFFFFu;
            const uint32_t lo = min(x0, x1), hi = max(x0, x1), mid = min(hi, x2);
            last = max(hi, x2);
            base[0] = min(lo, mid);
            base[1] = max(lo, mid);
            base[2] = last;
        } else {
            sort4_u16(own.x, own.y);
            base[0] = own.x & 0xFFFFu;
            base[1] = own.x >> 16;
            base[2] = own.y & 0xFFFFu;
            base[3] = last = own.y >> 16;
        }
#pragma unroll
        for (int j = 0; j < kAcc; ++j) na[j] = 0x00010000u - base[j] * 0x10001u;     // (-a, -a) mod 2^16
        G[0] = (last - base[0]) * 0x10001u;                                          // the last copy ends at itself at least
#pragma unroll
        for (int j = 1; j < kAcc; ++j) G[j] = ((base[j - 1] - base[j]) & 0xFFFFu) * 0x10001u;   // copy j ends at itself at least
    }
    __device__ __forceinline__ void visit(uint2 r) {
#pragma unroll
        for (int j = 0; j < kAcc; ++j) {
            G[j] = __viaddmax_u16x2(r.x, na[j], G[j]);
            G[j] = __viaddmax_u16x2(r.y, na[j], G[j]);
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

// kAcc: number of copies the node pass keeps apart (3 or 4).
// kProfile: one sequence, whose usage per step and free steps are written out (moc_mem_profile).
template <typename MemT, int kAcc, bool kTiles, bool kProfile>
__global__ void __launch_bounds__(1024) eval_quad_kernel(const QuadParams p) {
    extern __shared__ __align__(16) char smem[];
    __shared__ int64_t s_dur[32];
    __shared__ uint32_t s_lo[32], s_hi[32];
    __shared__ int64_t s_top[32];
    __shared__ uint32_t s_flags;
    constexpr int kShift = sizeof(MemT) == 4 ? 2 : 3;
    constexpr uint32_t kFull = 0xFFFFFFFFu;
    const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, n_warps = nthr >> 5;
    const int warp = __shfl_sync(kFull, tid >> 5, 0);
    int n = p.n;
    MOC_KEEP(n);
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem);
    uint32_t wa = sbase, ca = sbase + p.word_bytes, da = ca + p.cnt_bytes;   // words | counters | delta[0..]
    MOC_KEEP(wa);
    MOC_KEEP(ca);
    MOC_KEEP(da);
    const uint32_t dm1 = da - (uint32_t)sizeof(MemT);
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

    // ---- rows: block c takes [c * B / grid, (c + 1) * B / grid), or every grid-th one with the offsets given
    const bool self = !kProfile && p.offs == nullptr;
    int b = self ? (int)((int64_t)blockIdx.x * p.B / gridDim.x) : (int)blockIdx.x, b_end = p.B, b_step = gridDim.x;
    int64_t off = 0;
    int32_t T_next = kProfile ? p.single_len : (b < p.B ? __ldg(p.lens + b) : 0);      // one sequence ahead
    if (self) {
        b_end = (int)(((int64_t)blockIdx.x + 1) * p.B / gridDim.x);
        b_step = 1;
        int64_t sum = 0;
        int i = tid;
        if ((reinterpret_cast<uintptr_t>(p.lens) & 15) == 0) {
            const int4* l4 = reinterpret_cast<const int4*>(p.lens);
            for (int k = tid; k < b >> 2; k += nthr) {
                const int4 x = __ldg(l4 + k);
                sum += (int64_t)max(x.x, 0) + max(x.y, 0) + max(x.z, 0) + max(x.w, 0);
            }
            i += b & ~3;
        }
        for (; i < b; i += nthr) sum += max(__ldg(p.lens + i), 0);
        sum = warp_sum64(sum);
        if (lane == 0) s_dur[warp] = sum;
        __syncthreads();
        for (int k = 0; k < n_warps; ++k) off += s_dur[k];
    }
    for (; b < b_end; b += b_step) {
        const int32_t T = T_next;
        if (!kProfile && b + b_step < b_end) T_next = __ldg(p.lens + b + b_step);
        if (!self && !kProfile) off = __ldg(p.offs + b);
        int64_t out_pk = -1, out_du = -1;
        int32_t out_st = -2;
        if (T >= n && T <= p.max_T) {      // uniform over the block
            // ---- clear words and counters (stage 1b writes every delta the prefix sum reads)
            {
                const int4 z = make_int4(0, 0, 0, 0);
                int4* s4 = reinterpret_cast<int4*>(smem);
                const int nz = (int)((p.word_bytes + p.cnt_bytes) >> 4);
                for (int i = tid; i < nz; i += nthr) s4[i] = z;
                if (tid == 0) s_flags = 0;
            }
            __syncthreads();
            Amount<MemT> m_next = amount(min(tid, n - 1));          // for stage 1b, one round ahead
            // ---- stage 1a
            uint32_t flags = 0;    // bit 0: malformed, bit 1: precedence violated
            {
                const int32_t* row = p.seqs + off;
                auto put = [&](uint32_t id, int t) {
                    if (id < (uint32_t)n) {
                        const uint32_t sh = (id & 1u) << 4;
                        const uint32_t k = (atom_add_shared_u32(ca + ((id >> 1) << 2), 1u << sh) >> sh) & 0xFFFFu;
                        if (k < 4) sts_u16(wa + (id << 3) + (k << 1), (uint32_t)t + 1u);
                    } else {
                        flags = 1;
                    }
                };
                int t = tid;
                for (; t + 3 * nthr < T; t += 4 * nthr) {      // four loads in flight per thread
                    const uint32_t i0 = (uint32_t)__ldg(row + t), i1 = (uint32_t)__ldg(row + t + nthr),
                                   i2 = (uint32_t)__ldg(row + t + 2 * nthr), i3 = (uint32_t)__ldg(row + t + 3 * nthr);
                    put(i0, t);
                    put(i1, t + nthr);
                    put(i2, t + 2 * nthr);
                    put(i3, t + 3 * nthr);
                }
                for (; t < T; t += nthr) put((uint32_t)__ldg(row + t), t);
                if (tid == 0) {
                    sts_u64(wa + ((uint32_t)(n + 1) << 3), (uint64_t)(uint32_t)T * 0x0001000100010001ull);
                    sts_u64(wa + p.word_bytes - 16u, 0x0001000100010001ull);      // owned by empty node slots
                }
            }
            __syncthreads();
            // records and first successor row of a tile are requested while the tile before it (or stage 1b) is worked on
            uint4 r_next[2];
            const uint32_t* ps_next = nullptr;
            uint32_t e_first = 0;
            auto request = [&](int d) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if constexpr (sizeof(MemT) == 4) {
                        const uint2 r = __ldg(reinterpret_cast<const uint2*>(p.rec) + (2 * d + h) * 32 + lane);
                        r_next[h].x = r.x;
                        r_next[h].z = r.y;
                    } else {
                        r_next[h] = __ldg(reinterpret_cast<const uint4*>(p.rec) + (2 * d + h) * 32 + lane);
                    }
                }
                ps_next = p.sell + 32 * __ldg(p.tile_row + d) + lane;
                e_first = __ldg(ps_next);
            };
            if (kTiles && warp < p.n_tiles) request(warp);
            // ---- stage 1b
            int64_t dur = 0;
            for (int v = tid; v < n; v += nthr) {
                uint32_t c, limit = (uint32_t)p.C;
                asm volatile("{\n\t.reg .u16 h;\n\tld.shared.u16 h, [%1];\n\tcvt.u32.u16 %0, h;\n\t}" : "=r"(c) : "r"(ca + 2u * (uint32_t)v) : "memory");
                if (p.cap != nullptr) limit = min(limit, (uint32_t)__ldg(p.cap + v));
                const uint2 q = lds_v2(wa + ((uint32_t)v << 3));
                const Amount<MemT> mv = m_next;
                m_next = amount(min(v + nthr, n - 1));
                if (c - 1u >= limit) {       // absent or overfull: its word holds no usable positions
                    flags |= 1;
                    continue;
                }
                if (c > 1) dur += (int64_t)(c - 1) * __ldg(p.w + v);
                const uint32_t lo = c == 1 ? q.x * 0x10001u : q.x;
                const uint32_t hi = c < 3 ? lo : (c == 3 ? __byte_perm(q.y, q.x, 0x5410) : q.y);
                if (c < 4) sts_u64(wa + ((uint32_t)v << 3), (uint64_t)lo | ((uint64_t)hi << 32));
                quad_store(dm1 + ((lo & 0xFFFFu) << kShift), mv);
                if (c > 1) quad_store(dm1 + ((lo >> 16) << kShift), mv);
                if (c > 2) quad_store(dm1 + ((hi & 0xFFFFu) << kShift), mv);
                if (kAcc > 3 && c > 3) quad_store(dm1 + ((hi >> 16) << kShift), mv);
            }
            flags = __reduce_or_sync(kFull, flags);
            dur = warp_sum64(dur);
            if (lane == 0) {
                if (flags) atomicOr(&s_flags, flags);
                s_dur[warp] = dur;
            }
            __syncthreads();
            const bool malformed = (s_flags & 1u) != 0;
            if (!malformed) {
                // ---- stage 2 and the scatter of stage 3
                uint32_t depw = 0;
                if constexpr (kTiles) {
                    for (int d = warp; d < p.n_tiles; d += n_warps) {
                        QuadNode<kAcc> u[2];
                        Amount<MemT> m[2];
                        const uint32_t x0 = r_next[0].x, x1 = r_next[1].x;
                        const uint32_t* ps = ps_next;
                        uint32_t e_next = e_first;
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            if constexpr (sizeof(MemT) == 4) {
                                m[h].v = (MemT)r_next[h].z;
                            } else {
                                m[h].lo = r_next[h].z;
                                m[h].hi = r_next[h].w;
                            }
                            u[h].open(lds_v2(wa + ((r_next[h].x & 0xFFFFu) << 1)));
                        }
                        if (d + n_warps < p.n_tiles) request(d + n_warps);
                        const int rows = __shfl_sync(kFull, (int)(x0 >> 16), 0);
                        for (int k = 0; k < rows; ++k) {
                            const uint32_t e = e_next;
                            ps += 32;
                            if (k + 1 < rows) e_next = __ldg(ps);
                            const uint2 r0 = lds_v2(wa + ((e & 0xFFFFu) << 1)), r1 = lds_v2(wa + ((e >> 16) << 1));
                            u[0].visit(r0);
                            u[1].visit(r1);
                        }
                        // an empty node slot owns the last word of the area: no step is its own
                        const bool real0 = !kProfile || (x0 & 0xFFFFu) << 1 != p.word_bytes - 16u, real1 = !kProfile || (x1 & 0xFFFFu) << 1 != p.word_bytes - 16u;
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
                        u.open(lds_v2(wa + (node << 3)));
                        const uint32_t in8[4] = {inl.x, inl.y, inl.z, inl.w};
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            if (k < rounds) {
                                if ((uint32_t)k < deg) u.visit(lds_v2(wa + (((k & 1) ? in8[k >> 1] >> 16 : in8[k >> 1] & 0xFFFFu) << 3)));
                            }
                        }
                        for (int k = 8; k < rounds; ++k)
                            if ((uint32_t)k < deg) u.visit(lds_v2(wa + ((uint32_t)__ldg(p.succ + e8 + (k - 8)) << 3)));
                        if (i < n) depw |= u.template close<MemT, kShift, kProfile>(da, amount((int)node), p.out_free, p.out_free != nullptr);
                    }
                }
                if (__any_sync(kFull, (depw & 0x8000u) != 0) && lane == 0) atomicOr(&s_flags, 2u);
            }
            __syncthreads();
            const uint32_t fl = s_flags;
            if (!(fl & 1u)) {
                out_du = p.base_dur;
                for (int k = 0; k < n_warps; ++k) out_du += s_dur[k];
                out_st = -1;
            }
            if (fl == 0) {
                // ---- stages 3 and 4: prefix sum, each thread a chunk of consecutive steps (odd length: no bank conflicts)
                const int chunk = ((T + nthr - 1) / nthr) | 1;
                const int tb = min(tid * chunk, T), te = min(tb + chunk, T);
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
                // chunk sums -> usage in front of every chunk; a thread without steps passes its prefix on
                uint32_t lo_in = warp_inclusive_sum(lo, lane), hi_in = 0;
                if constexpr (sizeof(MemT) == 8) hi_in = warp_inclusive_sum(hi, lane);
                if (lane == 31) {
                    s_lo[warp] = lo_in;
                    s_hi[warp] = hi_in;
                }
                __syncthreads();
                lo_in -= lo;
                hi_in -= hi;
                for (int k = 0; k < warp; ++k) {
                    lo_in += s_lo[k];
                    if constexpr (sizeof(MemT) == 8) hi_in += s_hi[k];
                }
                MemT before;
                if constexpr (sizeof(MemT) == 4) before = (MemT)lo_in;
                else before = split_value(lo_in, hi_in, p.split);
                MemT peak = tb < te ? before + top : MemT(0);
                if constexpr (kProfile) {
                    ad = da + ((uint32_t)tb << kShift);
                    lo = lo_in;
                    hi = hi_in;
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
                peak = warp_max_t(peak);
                if (lane == 0) s_top[warp] = (int64_t)peak;
                __syncthreads();
                if (tid == 0) {
                    out_pk = s_top[0];
                    for (int k = 1; k < n_warps; ++k) out_pk = s_top[k] > out_pk ? s_top[k] : out_pk;
                    out_st = out_pk <= p.M ? 1 : 0;
                }
            }
        }
        if constexpr (kProfile) {
            if (tid == 0) s_flags = (uint32_t)out_st;      // only thread 0 knows 0 or 1; nothing reads the flags any more
            __syncthreads();
            const int32_t st = (int32_t)s_flags;
            if (tid == 0) p.out_status[0] = st;
            if (st < 0) {
                for (int t = tid; t < T; t += nthr) {
                    p.out_profile[t] = -1;
                    if (p.out_free) p.out_free[t] = -1;
                }
            }
            return;
        }
        if (tid == 0) {
            p.out_peak[b] = out_pk;
            p.out_dur[b] = out_du;
            p.out_status[b] = out_st;
        }
        off += max(T, 0);
        __syncthreads();    // the state is reused by the next sequence
    }
}

}  // namespace moc
