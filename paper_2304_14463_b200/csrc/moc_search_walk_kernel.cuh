// The search (paper: Section 3, the two-phase local search), all generations of a call in one kernel.  The chains are independent, so a warp takes its chain through
// every generation of the launch with the chain's copy positions in shared memory; nothing is exchanged
// between warps.  C <= 2 and graphs of the warp-per-sequence layout (moc_pair_kernel.cuh).
//
// What a generation costs.  About four proposals of five are refused by a test on the edited node alone
// (copy count, Eq. 5 on the edges that touch the node).  A lane therefore draws and tests one proposal, 32 of
// one generation or of several generations at a time against the chain's present sequence, and the warp
// evaluates only the admissible ones, in order.  An accepted one changes the sequence: the generations
// behind it are tested again (a draw does not depend on the sequence, only its reading does).
// An admissible proposal is evaluated in full, but not from its sequence: the copy positions of the edited
// sequence are the parent's, shifted by at most one step, which is two packed instructions per word, so that
// the occurrence pass of the evaluation kernel (data-dependent exchanges) falls away.  A proposal that
// cannot be accepted whatever its peak (longer duration while the chain is within the budget) is not
// evaluated: the key of the chain decides already.
// With kFloor the test also works out the usage that the edited sequence has at the step where the chain reaches its peak.  The new
// peak is no lower, which refuses proposals and orders the others: the first of them that reaches its bound ends the generation.  Of 3.3 admissible proposals
// of 32 0.97 are evaluated (n = 442, over the budget; counted on the CPU), and nearly every one of those is accepted.
//
// The sequence itself stays in global memory (L2): the tests read one element per proposal, and an
// accepted edit shifts the elements between its two places by one.  It is kept there because 3.5 KB per warp
// less (n = 442) let 28 warps share an SM instead of 22.
//
// Chains without a valid sequence (status < 0) have no test to rely on: their proposals are evaluated from
// the written-out order, one generation at a time, until one is valid.
//
// Bound: instruction issue (76 % of the slots with 32 proposals a generation; a generation of new chains takes 3300 instructions, behind ten of them 2600) and, for small populations,
// the latency of its dependent shared-memory reads; 28 warps beat 24 and 20 with more registers each, and 30 with fewer.
// n = 442, state copied out: 4096 chains x 20 generations 436 -> 41.9 us against two kernels per generation that
// write every proposal out, 38.9 with the neighbours' lists on chip, 37.1 with the words of a sequence from eight loads in flight; 32768 chains x 32 proposals x 10 generations 2409 -> 1052 us
// against a cached evaluation per chain that is rebuilt after every acceptance, 1010 -> 951 with the lists, 870 -> 500 (another GPU 1004 -> 508) with the bound,
// 508 -> 472 with the draws kept between tests and their keys in the constant bank.
// Tried: the chain's deltas kept and corrected for the few intervals that an edit changes instead of stages 2 and 3 over all nodes (two more calls and
// serial chains per evaluation: 503 -> 578 us there, small graphs 20 to 40 % slower; n = 900 gained 20 %).
#pragma once
#include "moc_edit_kernels.cuh"
#include "moc_search_kernels.cuh"

namespace moc {

constexpr int kWalkThreads = 896;     // 28 warps, 72 registers per thread

struct WalkParams {
    SearchParams s;            // s.generation: number of the first generation
    int32_t n_gen;             // generations of this launch
    int32_t samples;           // E: proposals per chain and generation
    int32_t lanes_per_gen;     // E rounded up to a power of two, at most 32
    int32_t* peak_at;          // P: walk_eval's `at` of each chain's sequence, 0: not known
    uint32_t round_key[20];    // of the draws: operands from the constant bank instead of twenty additions
    int32_t n, C, n_tiles;
    int32_t split;             // 64-bit sums: as in PairParams
    const void* rec;           // node records and successor tiles of the warp-per-sequence layout
    const uint32_t* sell;
    const int32_t* succ_start;
    const int32_t* succ;
    const int32_t* pred_start;
    const int32_t* pred;
    const int64_t* w;
    const int64_t* m;
    const int32_t* cap;        // per-node caps or nullptr
    uint32_t rec_bytes, sell_bytes;      // graph, once per block
    int32_t n_edges;
    const uint32_t* lists;     // kLists: the neighbours' lists (walk_lists), behind the graph in shared memory
    uint32_t list_bytes;                 // of the lists, with m behind them where `sizes`
    int32_t sizes;
    uint32_t word_bytes;       // occurrence words (n + 2, padded) without the constant word behind them
    uint32_t delta_bytes;      // front pad + deltas for C * n steps
};

// Scalars of the warp's chain that are needed between evaluations only.  They are kept in shared memory: as
// registers they were spilled, and the local memory of 28 warps is far larger than the L1 that is left beside
// the chains' state.
constexpr uint32_t kWalkQd = 0, kWalkJi = 4, kWalkX = 8, kWalkWx = 12;           // the chosen proposal
constexpr uint32_t kWalkBestA = 16, kWalkBestD = 24, kWalkBestPk = 32;           // its key and peak (without one: the chain's key)
constexpr uint32_t kWalkBestAt = 40, kWalkAcc = 44, kWalkPk = 48, kWalkDu = 56;  // its `at`; the chain: accepted, peak, duration
constexpr uint32_t kWalkNoteBytes = 64;

// Bytes of one warp: two sets of words, each followed by the constant word, the scalars, and the deltas.
__host__ __device__ inline size_t walk_warp_bytes(uint32_t word_bytes, uint32_t delta_bytes) {
    return 2 * ((size_t)word_bytes + kPairWordTail) + kWalkNoteBytes + delta_bytes;
}

// [p > k] per 16-bit half (p, k < 2^15): max(min(p - k, 1), 0).
__device__ __forceinline__ uint32_t walk_above(uint32_t p, uint32_t k) {
    return __viaddmin_s16x2_relu(p, ((0x00010000u - k) & 0xFFFFu) * 0x10001u, 0x00010001u);
}

// Stages 2 to 4 of the evaluation (moc_pair_kernel.cuh) on the occurrence words at `wa`: the peak, whether a
// consumer lacks a producer copy, and `at`: a step at which the peak is reached (1-based) or, without kExact, minus the first step of a
// vector of deltas that has one.  The deltas are zero on entry and on return.
template <typename MemT, bool kExact>
__device__ __forceinline__ MemT walk_eval(uint32_t wa, uint32_t da, uint32_t rec0, uint32_t sell0, int n_tiles, int32_t T, int lane,
                                       int32_t split, bool& dep, int32_t& at) {
    constexpr uint32_t kRecB = sizeof(MemT) == 4 ? 8u : 16u, kFull = 0xFFFFFFFFu;
    constexpr int kPerVec = 16 / (int)sizeof(MemT), kShift = sizeof(MemT) == 4 ? 2 : 3;
    const uint32_t da1 = da - (uint32_t)sizeof(MemT);
    uint32_t depw = 0, prec = rec0, ps = sell0;
    for (int d = 0; d < n_tiles; ++d, prec += 64u * kRecB) {
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
            const uint32_t own = lds_u32(wa + (x & 0xFFFFu)), sw = swap_halves(own);
            const uint32_t mn = min_u16x2(own, sw), mx = max_u16x2(own, sw);
            ab[h] = __byte_perm(mn, mx, 0x7610);
            naa[h] = 0x00010000u - mn;
            nbb[h] = 0x00010000u - mx;
            Ga[h] = mx - mn;
            Gb[h] = 0x00010000u - Ga[h];
        }

#pragma unroll 2
        for (int k = 0; k < rows; ++k) {
            const uint32_t e = lds_u32(ps);
            ps += 128u;
            const uint32_t r0 = lds_u32(wa + (e & 0xFFFFu)), r1 = lds_u32(wa + (e >> 16));
            Ga[0] = __viaddmax_u16x2(r0, naa[0], Ga[0]);
            Ga[1] = __viaddmax_u16x2(r1, naa[1], Ga[1]);
            Gb[0] = __viaddmax_u16x2(r0, nbb[0], Gb[0]);
            Gb[1] = __viaddmax_u16x2(r1, nbb[1], Gb[1]);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            depw |= Ga[h];
            const uint32_t gg = max_u16x2(__byte_perm(Ga[h], Gb[h], 0x5410), __byte_perm(Ga[h], Gb[h], 0x7632));
            const uint32_t v = gg + ab[h], a16 = ab[h] & 0xFFFFu, b16 = ab[h] >> 16;
            red_add_amount(da1 + (b16 << kShift), m[h]);
            red_sub_amount(da + ((v & 0xFFFFu) << kShift), m[h]);
            if (a16 != b16) {
                red_add_amount(da1 + (a16 << kShift), m[h]);
                red_sub_amount(da + ((v >> 16) << kShift), m[h]);
            }
        }
    }
    dep = __any_sync(kFull, (depw & 0x80008000u) != 0);
    __syncwarp();
    // prefix sum and running maximum; lane owns V consecutive vectors
    const int nvec = (T + 2 + kPerVec - 1) / kPerVec, V = ((nvec + 31) >> 5) | 1;
    uint32_t ad = da + 16u * (uint32_t)(lane * V);
    MemT top = sizeof(MemT) == 8 ? (MemT)INT64_MIN : (MemT)INT32_MIN;
    int vec = 0;                       // the lane's vector that holds its maximum
    MemT run = 0;
    uint32_t lo = 0, hi = 0;           // 64-bit sums: the two parts of the running sum (moc_pair_kernel.cuh)
    for (int j = 0; j < V; ++j, ad += 16u) {
        const uint4 q = lds_v4(ad);
        if constexpr (!kExact) asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(ad), "r"(0) : "memory");
        MemT most;
        if constexpr (sizeof(MemT) == 4) {
            run += (MemT)q.x; most = run;
            run += (MemT)q.y; most = max(most, run);
            run += (MemT)q.z; most = max(most, run);
            run += (MemT)q.w; most = max(most, run);
        } else {
            lo += q.x; hi += q.y;
            most = split_value(lo, hi, split);
            lo += q.z; hi += q.w;
            const MemT u = split_value(lo, hi, split);
            most = u > most ? u : most;
        }
        if (most > top) { top = most; vec = j; }
    }
    if constexpr (sizeof(MemT) == 4) top += warp_inclusive_sum(run, lane) - run;
    else top += split_value(warp_inclusive_sum(lo, lane) - lo, warp_inclusive_sum(hi, lane) - hi, split);
    const MemT peak = warp_max_t(top);
    const int src = __ffs(__ballot_sync(kFull, top == peak)) - 1;
    vec = src * V + __shfl_sync(kFull, vec, src);
    at = kPerVec * vec + 1;
    if constexpr (kExact) {
        const uint4 q = lds_v4(da + 16u * (uint32_t)vec);       // the first of its steps with the largest sum of deltas
        if constexpr (sizeof(MemT) == 4) {
            const MemT s1 = (MemT)q.y, s2 = s1 + (MemT)q.z, s3 = s2 + (MemT)q.w, most = max(max(s1, s2), max(s3, (MemT)0));
            at += most == 0 ? 0 : most == s1 ? 1 : most == s2 ? 2 : 3;
        } else {
            at += split_value(q.z, q.w, split) > 0 ? 1 : 0;
        }
        __syncwarp();
        ad = da + 16u * (uint32_t)(lane * V);
        for (int j = 0; j < V; ++j, ad += 16u) asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(ad), "r"(0) : "memory");
    } else {
        at = -at;
    }
    __syncwarp();
    return peak;
}

// Element qd taken out of row[0..T) (none: kEditNone), then x put in front of index ji of what is left (none:
// kEditNone), in place: the elements between the two places move by one.  Not inlined: its eight loads in
// flight would cost the whole kernel registers.
static __device__ __noinline__ void walk_apply(int32_t* row, int32_t T, int32_t qd, int32_t ji, int32_t x, int lane) {
    const bool left = qd != kEditNone && (ji == kEditNone || ji >= qd);
    const int32_t a = left ? qd + 1 : ji, b = left ? (ji == kEditNone ? T : ji + 1) : (qd == kEditNone ? T : qd), dir = left ? -1 : 1;
    for (int32_t done = 0; done < b - a; done += 256) {
        int32_t v[8];
        // ascending pieces to the left, descending pieces to the right: no element is overwritten unread
        const int32_t base = (left ? a + done : b - done - 256) + lane;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (base + 32 * k >= a && base + 32 * k < b) v[k] = row[base + 32 * k];
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (base + 32 * k >= a && base + 32 * k < b) row[base + 32 * k + dir] = v[k];
        __syncwarp();
    }
    if (ji != kEditNone && lane == 0) row[ji] = x;
    __syncwarp();
}

// kLists: the test of a proposal reads the neighbours' lists from the block's shared memory (durations below 2^31, at most 65535 edges);
// through L1, of which the chains' state leaves little, a third of the kernel's stalls were waits for them.
template <typename MemT, bool kLists, bool kFloor>
__global__ void __launch_bounds__(kWalkThreads, 1) search_walk_kernel(const WalkParams p) {
    extern __shared__ __align__(16) char smem[];
    const SearchParams& s = p.s;
    constexpr uint32_t kRecB = sizeof(MemT) == 4 ? 8u : 16u, kFull = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
    const int warp = __shfl_sync(kFull, (int)(threadIdx.x >> 5), 0);
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem);
    uint32_t l_node = sbase + p.rec_bytes + p.sell_bytes;
    {
        // asynchronous copies: a block of a small population has few threads for them
        auto copy = [&](uint32_t to, const void* from, uint32_t bytes) {
            for (uint32_t i = 16u * threadIdx.x; i < bytes; i += 16u * blockDim.x)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + i), "l"(reinterpret_cast<const char*>(from) + i) : "memory");
        };
        copy(sbase, p.rec, p.rec_bytes);
        copy(sbase + p.rec_bytes, p.sell, p.sell_bytes);
        if constexpr (kLists) copy(l_node, p.lists, p.list_bytes);
    }
    const uint32_t word_set = p.word_bytes + kPairWordTail;
    auto duration = [&](int32_t v) -> int64_t { return kLists ? (int64_t)lds_u32_nv(l_node + 8u * (uint32_t)v + 4u) : __ldg(p.w + v); };
    auto neighbour = [&](uint32_t list, const int32_t* far, int32_t k) -> uint32_t {
        if constexpr (kLists) {
            uint32_t x;
            asm("{\n\t.reg .u16 h;\n\tld.shared.u16 h, [%1];\n\tcvt.u32.u16 %0, h;\n\t}" : "=r"(x) : "r"(list + 2u * (uint32_t)k));
            return x;
        } else {
            return (uint32_t)__ldg(far + k);
        }
    };
    const uint32_t mine = sbase + p.rec_bytes + p.sell_bytes + (kLists ? p.list_bytes : 0u) + (uint32_t)warp * (2u * word_set + kWalkNoteBytes + p.delta_bytes);
    const uint32_t note = mine + 2u * word_set;
    const uint32_t da = note + kWalkNoteBytes + kPairDeltaFront;     // &delta[0]
    const uint32_t rec0 = sbase + kRecB * (uint32_t)lane, sell0 = sbase + p.rec_bytes + 4u * (uint32_t)lane;
    const int n = p.n, n_tiles = p.n_tiles;
    if (lane < 2) sts_u32(mine + word_set * (uint32_t)lane + p.word_bytes, 0x00010001u);   // owned by empty node slots
    for (uint32_t o = 16u * (uint32_t)lane; o < p.delta_bytes; o += 512u)
        asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(da - kPairDeltaFront + o), "r"(0) : "memory");
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if constexpr (kLists) MOC_STAGED(l_node);
    const uint32_t l_succ = l_node + 8u * (uint32_t)(p.n + 1), l_pred = l_succ + 2u * (uint32_t)((p.n_edges + 3) & ~3), l_size = l_pred + 2u * (uint32_t)((p.n_edges + 3) & ~3);
    auto size_of = [&](int32_t v) -> MemT {
        if (kLists && sizeof(MemT) == 4 && p.sizes) return (MemT)lds_u32_nv(l_size + 4u * (uint32_t)v);
        return (MemT)__ldg(p.m + v);
    };
    auto successors = [&](int32_t v, int32_t& from, int32_t& to) {
        if constexpr (kLists) {
            from = (int32_t)(lds_u32_nv(l_node + 8u * (uint32_t)v) & 0xFFFFu);
            to = (int32_t)(lds_u32_nv(l_node + 8u * (uint32_t)v + 8u) & 0xFFFFu);
        } else {
            from = __ldg(p.succ_start + v);
            to = __ldg(p.succ_start + v + 1);
        }
    };

    for (int32_t c = blockIdx.x * wpb + warp; c < s.P; c += gridDim.x * wpb) {
        int32_t* row = s.rows + ((int64_t)s.cur[c] * s.P + c) * s.stride;
        int32_t T = s.lens[c], tp = p.peak_at[c];
        if constexpr (!kFloor) tp = abs(tp);            // a step of either kind
        bool valid = s.status[c] >= 0;
        bool over = valid && s.peak[c] > s.M;       // over the budget
        if (lane == 0) {
            sts_u64(note + kWalkPk, (uint64_t)s.peak[c]);
            sts_u64(note + kWalkDu, (uint64_t)s.dur[c]);
            sts_u32(note + kWalkAcc, 0u);
        }
        __syncwarp();
        uint32_t wa = mine, wb = mine + word_set;       // the chain's words, and those of a proposal
        // occurrence words of the edited row (qd = ji = kEditNone: the row itself) by exchanges, as in the
        // evaluation kernel; returns the summed durations of the lane's elements.  Invalid ids go to the spare word n.
        auto words_of = [&](uint32_t w0, int32_t Tc, int32_t qd, int32_t ji, int32_t x) -> int64_t {
            for (uint32_t o = 16u * (uint32_t)lane; o < p.word_bytes; o += 512u)
                asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(w0 + o), "r"(0) : "memory");
            __syncwarp();
            int64_t sum = 0;
            for (int32_t t = lane; t < Tc; t += 32) {
                int32_t v = x;
                if (t != ji) {
                    const int32_t k = t - (t > ji ? 1 : 0);
                    v = row[k + (k >= qd ? 1 : 0)];
                }
                if ((uint32_t)v < (uint32_t)n) sum += duration(v);
                const uint32_t addr = w0 + 4u * min((uint32_t)v, (uint32_t)n);
                const uint32_t old = exch_shared(addr, ((uint32_t)t + 1u) * 0x10001u);
                sts_u16_if_nonzero(old, addr + 2, old);
            }
            __syncwarp();
            if (lane == 0) sts_u32(w0 + 4u * (uint32_t)(n + 1), (uint32_t)Tc * 0x10001u);
            __syncwarp();
            return sum;
        };
        if (valid) {
            // the words of the chain's sequence, eight elements of the row in flight per lane
            for (uint32_t o = 16u * (uint32_t)lane; o < p.word_bytes; o += 512u)
                asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(wa + o), "r"(0) : "memory");
            __syncwarp();
            for (int32_t t0 = lane; t0 < T; t0 += 256) {
                int32_t v[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] = t0 + 32 * k < T ? row[t0 + 32 * k] : n;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    if (t0 + 32 * k >= T) break;
                    const uint32_t addr = wa + 4u * min((uint32_t)v[k], (uint32_t)n);
                    const uint32_t old = exch_shared(addr, (uint32_t)(t0 + 32 * k + 1) * 0x10001u);
                    sts_u16_if_nonzero(old, addr + 2, old);
                }
            }
            __syncwarp();
            if (lane == 0) sts_u32(wa + 4u * (uint32_t)(n + 1), (uint32_t)T * 0x10001u);
            __syncwarp();
        }
        if constexpr (kFloor) {
            // A place from the other variant is not exact.  One evaluation finds it; without it a chain that hardly accepts any more would stay without a bound.
            bool dep;
            if (valid && tp < 0) {
                walk_eval<MemT, true>(wa, da, rec0, sell0, n_tiles, T, lane, p.split, dep, tp);
                if (lane == 0) p.peak_at[c] = tp;       // once, whether or not the chain accepts in this launch
            }
            tp = max(tp, 0);
        }
        // out with step qd_s, in at index ji_s: the words of the edited sequence at w1, from the parent's at w0
        auto shift_words = [&](uint32_t w0, uint32_t w1, int32_t Tc_s, int32_t qd_s, int32_t ji_s, int32_t x_s, uint32_t wx_s) {
            const uint32_t kq = qd_s == kEditNone ? 0x7FFFu : (uint32_t)qd_s + 1u, kj = ji_s == kEditNone ? 0x7FFFu : (uint32_t)ji_s;
            for (uint32_t o = 16u * (uint32_t)lane; o < p.word_bytes; o += 512u) {
                uint4 v = lds_v4(w0 + o);
                v.x -= walk_above(v.x, kq); v.x += walk_above(v.x, kj);
                v.y -= walk_above(v.y, kq); v.y += walk_above(v.y, kj);
                v.z -= walk_above(v.z, kq); v.z += walk_above(v.z, kj);
                v.w -= walk_above(v.w, kq); v.w += walk_above(v.w, kj);
                asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(w1 + o), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
            }
            __syncwarp();
            if (lane == 0) {
                sts_u32(w1 + 4u * (uint32_t)x_s, wx_s);
                sts_u32(w1 + 4u * (uint32_t)(n + 1), (uint32_t)Tc_s * 0x10001u);
            }
            __syncwarp();
        };

        // The edit (qd, ji) of node x against the chain's valid sequence: can it be accepted, as far as the copies of x
        // and of its neighbours tell; the node's word after the edit, the new duration, and, with kFloor, what the new peak cannot be below: at
        // most the usage after the edit at the step where the chain reaches its peak (0: that step is not known, or is the one taken out).
        // An edit of x changes what is resident there for x and its predecessors only.  A node is resident at step tp when its last copy
        // up to tp is the step itself, or has a consumer at tp or behind it and in front of the node's next copy.
        auto test = [&](int32_t op, int32_t qd, int32_t ji, int32_t x, uint32_t& wx_new, int64_t& du_c, MemT& floor_c) -> bool {
            const uint32_t wx = lds_u32(wa + 4u * (uint32_t)x);
            const int32_t xa = (int32_t)min(wx & 0xFFFFu, wx >> 16) - 1, xb = (int32_t)max(wx & 0xFFFFu, wx >> 16) - 1;
            const int32_t cnt = xa == xb ? 1 : 2, cnt2 = cnt - (op >= 1 ? 1 : 0) + (op != 1 ? 1 : 0);
            if (!(cnt2 == 1 || (cnt2 == 2 && p.C >= 2 && (p.cap == nullptr || __ldg(p.cap + x) >= 2)))) return false;
            const int64_t more = duration(x) * (cnt2 - cnt);
            du_c = (int64_t)lds_u64(note + kWalkDu) + more;
            floor_c = 0;
            const bool longer = more > 0;
            if (longer && !over) return false;      // within the budget only the duration decides
            const bool known = tp > 0 && (!kFloor || tp != qd + 1);
            const int32_t tmax = kFloor ? tp : tp + 16 / (int32_t)sizeof(MemT) - 1;
            // Over the budget a longer sequence has to lower the peak.  A second copy of x lowers the usage at the
            // peak's step only when x is resident there for a later consumer, which the second copy can serve.
            // (Everything else an inserted copy does to the profile adds to it.)
            if (longer && known && !(xa + 1 < tmax && ji >= tp)) return false;
            auto map = [&](int32_t t) -> int32_t { const int32_t t1 = t - (t > qd ? 1 : 0); return t1 + (t1 >= ji ? 1 : 0); };
            // first child copy c0 (and c1), with the parent steps of other nodes' copies that lie in front of c0
            // (r < tb0) and behind it (r > ta0), 1-based, as in moc_edit_pass.cuh
            int32_t c0 = kEditNone, c1 = kEditNone, ta0 = 0, tb0 = 0;
            auto push = [&](int32_t cs, int32_t ta, int32_t tb) {
                if (c0 == kEditNone) { c0 = cs; ta0 = ta; tb0 = tb; }
                else if (cs < c0) { c1 = c0; c0 = cs; ta0 = ta; tb0 = tb; }
                else { c1 = cs; }
            };
            const int32_t thr = ji == kEditNone ? -1 : ji + (ji >= qd ? 1 : 0);     // steps in front of the inserted copy
            if (xa != qd) push(map(xa), xa + 1, xa + 1);
            if (cnt == 2 && xb != qd) push(map(xb), xb + 1, xb + 1);
            if (ji != kEditNone) push(ji, thr, thr + 1);
            wx_new = (uint32_t)(c0 + 1) | (uint32_t)((c1 == kEditNone ? c0 : c1) + 1) << 16;
            bool viol = false;
            int32_t p0, p1, s0, s1;
            successors(x, s0, s1);
            if constexpr (kLists) {
                p0 = (int32_t)(lds_u32_nv(l_node + 8u * (uint32_t)x) >> 16);
                p1 = (int32_t)(lds_u32_nv(l_node + 8u * (uint32_t)x + 8u) >> 16);
            } else {
                p0 = __ldg(p.pred_start + x);
                p1 = __ldg(p.pred_start + x + 1);
            }
            // without kFloor: a longer sequence needs a consumer of x that the second copy serves, and none from the peak to that copy
            const bool must_drop = !kFloor && longer && known;
            bool served = false;
            const uint32_t from_tp = ((0x00010000u - (uint32_t)tp) & 0xFFFFu) * 0x10001u;     // -tp in both halves
            uint32_t next = 0xFFFFFFFFu;            // first consumer of x at tp or behind it, counted from there
            // two reads of each kind in flight
#pragma unroll 1
            for (int32_t k = 0; k < max(p1 - p0, s1 - s0); k += 2) {
                uint32_t pw[2], sw[2];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    pw[i] = p0 + k + i < p1 ? lds_u32(wa + 4u * (int32_t)neighbour(l_pred, p.pred, p0 + k + i)) : 0u;
                    sw[i] = s0 + k + i < s1 ? lds_u32(wa + 4u * (int32_t)neighbour(l_succ, p.succ, s0 + k + i)) : 0xFFFFFFFFu;
                }
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int32_t ua = (int32_t)min(pw[i] & 0xFFFFu, pw[i] >> 16), r0 = (int32_t)min(sw[i] & 0xFFFFu, sw[i] >> 16);
                    viol |= ua > ta0 || r0 < tb0;
                    if constexpr (kFloor) {
                        next = __viaddmin_u16x2(sw[i], from_tp, next);
                    } else if (s0 + k + i < s1) {
                        const int32_t r1 = (int32_t)max(sw[i] & 0xFFFFu, sw[i] >> 16);
                        viol |= must_drop && ((r0 >= tmax && r0 <= ji) || (r1 >= tmax && r1 <= ji));
                        served |= r1 > ji;
                    }
                }
            }
            if (viol) return false;
            if (!kFloor) return !must_drop || served || s0 == s1;
            if (!known) return true;
            // copies of x at tp or in front of it, before and after; the last step in front of the next one
            bool had = xa < tp, has = thr >= 0 && thr < tp;
            int32_t lim_old = had && xb >= tp ? xb : 0x7FFF, lim_new = thr >= tp ? thr : 0x7FFF;
            if (xa != qd) {
                has |= xa < tp;
                if (xa >= tp) lim_new = min(lim_new, xa);
            }
            if (xb != qd) {
                has |= xb < tp;
                if (xb >= tp) lim_new = min(lim_new, xb);
            }
            const int64_t pk = (int64_t)lds_u64(note + kWalkPk);
            MemT change = 0;
            if (xa + 1 != tp && xb + 1 != tp) {
                const int32_t first = s0 == s1 ? 0x7FFF : (int32_t)min(next & 0xFFFFu, next >> 16) + tp;    // a sink is kept to the end
                const bool now = has && first <= lim_new, then = had && first <= lim_old;
                if (now != then) change = now ? size_of(x) : -size_of(x);
            }
            // A predecessor that loses a consumer: qd lies behind tp in the range of its copy, ji does not, and no other consumer does.
            // What one gains is left out (0.97 instead of 0.95 evaluations a generation, for less than half of the lists to go through).
            if (qd >= tp && qd != kEditNone) {
                const int32_t j_won = thr >= tp ? thr : 0x8000;
                uint32_t rest = 0xFFFFFFFFu;            // the copies of x that stay
                if (xa != qd) rest = (uint32_t)(xa + 1) * 0x10001u;
                if (xb != qd) rest = xa != qd ? (rest & 0xFFFFu) | (uint32_t)(xb + 1) << 16 : (uint32_t)(xb + 1) * 0x10001u;
#pragma unroll 1
                for (int32_t k = p0; k < p1; ++k) {
                    const int32_t u = (int32_t)neighbour(l_pred, p.pred, k);
                    const uint32_t pw = lds_u32(wa + 4u * (uint32_t)u);
                    const int32_t ua = (int32_t)min(pw & 0xFFFFu, pw >> 16), ub = (int32_t)max(pw & 0xFFFFu, pw >> 16), end = ub > tp ? ub : 0x7FFF;
                    if (qd + 1 >= end || end > j_won || ua >= tp || ub == tp) continue;
                    int32_t t0, t1;
                    successors(u, t0, t1);
                    uint32_t near = 0xFFFFFFFFu;        // another consumer
#pragma unroll 1
                    for (int32_t i = t0; i < t1; i += 2) {
                        const int32_t v0 = (int32_t)neighbour(l_succ, p.succ, i), v1 = (int32_t)neighbour(l_succ, p.succ, min(i + 1, t1 - 1));
                        const uint32_t w0 = lds_u32(wa + 4u * (uint32_t)v0), w1 = lds_u32(wa + 4u * (uint32_t)v1);
                        near = __viaddmin_u16x2(v0 == x ? rest : w0, from_tp, near);
                        near = __viaddmin_u16x2(v1 == x ? rest : w1, from_tp, near);
                    }
                    if ((int32_t)min(near & 0xFFFFu, near >> 16) + tp >= end) change -= size_of(u);
                }
            }
            floor_c = (MemT)pk + change;
            const int64_t a_c = (int64_t)floor_c > s.M ? (int64_t)floor_c : s.M, a_p = over ? pk : s.M;
            return a_c < a_p || (a_c == a_p && more <= 0);
        };
        // smallest of the lanes' values >= 0
        auto min64 = [&](int64_t v, bool in) -> int64_t {
            const uint32_t hi = in ? (uint32_t)((uint64_t)v >> 32) : kFull, hmin = __reduce_min_sync(kFull, hi);
            const uint32_t lo = (in && hi == hmin) ? (uint32_t)v : kFull, lmin = __reduce_min_sync(kFull, lo);
            return (int64_t)((uint64_t)hmin << 32 | lmin);
        };

        // A batch is `span` generations of E proposals with a lane each, or, for E > 32, 32 proposals of one
        // generation; the best proposal of the generation is then carried from batch to batch.
        const int64_t m_cap = sizeof(MemT) == 4 ? (int64_t)INT32_MAX : INT64_MAX;
        const MemT m_low = (MemT)min(max(s.M, (int64_t)0), m_cap);
        const int32_t E = p.samples, per = p.lanes_per_gen, span = 32 / per, my_gen = lane / per, my_e = lane % per;
        bool b_has = false, b_here = false;         // a proposal is chosen; its words are at wb
        int32_t b_e = 0;                            // its number (with E <= 32 its lane: generations are settled one at a time)
        auto fresh = [&]() {                        // a chain without a valid sequence takes any valid proposal
            b_has = false;
            if (lane == 0) {
                sts_u64(note + kWalkBestA, !valid ? (uint64_t)INT64_MAX : over ? lds_u64(note + kWalkPk) : (uint64_t)s.M);
                sts_u64(note + kWalkBestD, lds_u64(note + kWalkDu));
            }
            __syncwarp();
        };
        // the chosen proposal replaces the chain's sequence
        auto settle = [&]() {
            const int32_t qd_s = (int32_t)lds_u32(note + kWalkQd), ji_s = (int32_t)lds_u32(note + kWalkJi), x_s = (int32_t)lds_u32(note + kWalkX);
            const int32_t Tc_s = T + (qd_s == kEditNone ? 1 : 0) - (ji_s == kEditNone ? 1 : 0);
            if (!b_here) shift_words(wa, wb, Tc_s, qd_s, ji_s, x_s, lds_u32(note + kWalkWx));
            walk_apply(row, T, qd_s, ji_s, x_s, lane);
            const uint32_t sw = wa;
            wa = wb;
            wb = sw;
            T = Tc_s;
            tp = abs((int32_t)lds_u32(note + kWalkBestAt));
            valid = true;
            over = (int64_t)lds_u64(note + kWalkBestPk) > s.M;
            if (lane == 0) {
                sts_u64(note + kWalkPk, lds_u64(note + kWalkBestPk));
                sts_u64(note + kWalkDu, lds_u64(note + kWalkBestD));
                sts_u32(note + kWalkAcc, lds_u32(note + kWalkAcc) + 1u);
            }
            __syncwarp();
        };
        for (int32_t g0 = 0; g0 < p.n_gen && T > 0; g0 += span) {
            fresh();
            for (int32_t e0 = 0; e0 < E; e0 += 32) {
                const uint32_t drawn = __ballot_sync(kFull, g0 + my_gen < p.n_gen && e0 + my_e < E);
                // The lane's draw {r1, r2, kind of the edit}, kept for the tests after an acceptance (drawn again each time: n = 30, 32768 chains x 20
                // 158 -> 150 us, n = 442, 4096 x 20 32.8 -> 31.0).  In the lane's own memory (volatile: not in registers over the evaluations): 384 bytes
                // of shared memory a warp take as long at n = 442, but cost others a warp, that is a round of chains, or the lists (32 proposals x 10: n = 790,
                // 64-bit sums, 1600 chains 250 -> 176 us, n = 620, 8000 395 -> 360; one proposal 79 -> 57 and 110 -> 102).  With 64-bit sums, the lists read
                // through L1 and most proposals refused at once, the draws' lines cost more there than they save: one proposal x 10, 12288 chains, n = 900
                // 379 us drawn again, 393 kept, n = 600 221 and 227; with the bound on the new peak (8 proposals, n = 900) 1330 and 1285.
                constexpr bool kKeep = kLists || kFloor || sizeof(MemT) == 4;
                auto draw = [&]() -> uint3 {
                    const uint4 r = philox4x32_10_by(make_uint4(s.generation + (uint32_t)(g0 + my_gen), s.chain0 + (uint32_t)c, (uint32_t)(e0 + my_e), 0u),
                                                     [&](int k) { return make_uint2(p.round_key[2 * k], p.round_key[2 * k + 1]); });
                    return make_uint3(r.y, r.z, search_pick_kind(s.kinds, r.x));
                };
                volatile uint32_t kept[3];
                if constexpr (kKeep) {
                    const uint3 r = draw();
                    kept[0] = r.x;
                    kept[1] = r.y;
                    kept[2] = r.z;
                }
                uint32_t pending = drawn;
                while (pending && T > 0) {
                    // ---- the pending proposals against the present sequence, a lane each
                    const uint3 r = kKeep ? make_uint3(kept[0], kept[1], kept[2]) : draw();
                    const int32_t op = (int32_t)r.z;
                    const int32_t q = (int32_t)(r.x % (uint32_t)T), j = (int32_t)(r.y % ((uint32_t)T + (op == 0 ? 1u : 0u)));
                    const int32_t qd = op >= 1 ? q : kEditNone, ji = op != 1 ? j : kEditNone;
                    const int32_t Tc = T + (op == 0 ? 1 : 0) - (op == 1 ? 1 : 0);
                    const int32_t x = row[q];
                    bool adm = (pending >> lane & 1u) != 0 && Tc >= n && Tc <= s.max_T;
                    uint32_t wx_new = 0;
                    int64_t du_c = 0;
                    MemT floor_c = 0;
                    if (adm && valid) adm = test(op, qd, ji, x, wx_new, du_c, floor_c);
                    const MemT a_low = kFloor && floor_c > m_low ? floor_c : m_low;       // the least the key's first part can be
                    const uint32_t places = (uint32_t)q | (uint32_t)j << 15 | (uint32_t)op << 30;     // T < 2^15
                    uint32_t todo = __ballot_sync(kFull, adm);
                    pending = 0;
                    while (todo) {
                        // ---- the earliest generation that has proposals left: in order of the least their key can be, then number
                        const int gen = (__ffs(todo) - 1) / per;
                        const uint32_t group = (per == 32 ? kFull : (1u << per) - 1u) << (gen * per);
                        uint32_t cand = todo & group;
                        todo &= ~group;
                        while (cand) {
                            int sl = __ffs(cand) - 1;
                            if (cand & (cand - 1u)) {
                                bool in = (cand >> lane & 1u) != 0;
                                if constexpr (kFloor) {
                                    MemT a_min;             // by all lanes, whether or not theirs is left
                                    if constexpr (sizeof(MemT) == 4) a_min = __reduce_min_sync(kFull, in ? a_low : (MemT)INT32_MAX);
                                    else a_min = min64(a_low, in);
                                    in = in && a_low == a_min;
                                }
                                const int64_t d_min = min64(du_c, in);
                                sl = __ffs(__ballot_sync(kFull, in && du_c == d_min)) - 1;
                            }
                            cand &= ~(1u << sl);
                            const uint32_t at_s = __shfl_sync(kFull, places, sl), wx_s = __shfl_sync(kFull, wx_new, sl);
                            const int32_t op_s = (int32_t)(at_s >> 30), x_s = __shfl_sync(kFull, x, sl);
                            const int32_t qd_s = op_s >= 1 ? (int32_t)(at_s & 0x7FFFu) : kEditNone, ji_s = op_s != 1 ? (int32_t)(at_s >> 15 & 0x7FFFu) : kEditNone;
                            const int32_t Tc_s = T + (op_s == 0 ? 1 : 0) - (op_s == 1 ? 1 : 0);
                            int64_t du_s = __shfl_sync(kFull, du_c, sl);
                            // nothing behind the chosen proposal in this order can be better
                            if constexpr (kFloor) {
                                if (b_has) {
                                    const MemT l_s = __shfl_sync(kFull, a_low, sl);
                                    const int64_t a_s = (int64_t)l_s > s.M ? (int64_t)l_s : s.M, b_a = (int64_t)lds_u64(note + kWalkBestA), b_d = (int64_t)lds_u64(note + kWalkBestD);
                                    if (a_s > b_a || (a_s == b_a && (du_s > b_d || (du_s == b_d && e0 + sl > b_e)))) break;
                                }
                            } else {
                                if (b_has && (int64_t)lds_u64(note + kWalkBestA) == s.M && du_s >= (int64_t)lds_u64(note + kWalkBestD)) break;
                            }
                            b_here = false;
                            if (valid) {
                                shift_words(wa, wb, Tc_s, qd_s, ji_s, x_s, wx_s);
                            } else {
                                // from scratch: every node present, as many second copies as steps beyond n, caps
                                du_s = warp_sum64(words_of(wb, Tc_s, qd_s, ji_s, x_s));
                                uint32_t two = 0;
                                bool bad = false;
                                for (int32_t v = lane; v < n; v += 32) {
                                    const uint32_t wv = lds_u32(wb + 4u * (uint32_t)v);
                                    const bool t2 = (wv & 0xFFFFu) != wv >> 16;
                                    two += t2 ? 1u : 0u;
                                    bad |= wv == 0 || (t2 && (p.C < 2 || (p.cap != nullptr && __ldg(p.cap + v) < 2)));
                                }
                                two = __reduce_add_sync(kFull, two);
                                if (__any_sync(kFull, bad) || (int32_t)two != Tc_s - n) continue;
                            }
                            bool dep;
                            int32_t at;
                            const int64_t pk_s = (int64_t)walk_eval<MemT, kFloor>(wb, da, rec0, sell0, n_tiles, Tc_s, lane, p.split, dep, at);
                            const int64_t a_s = pk_s > s.M ? pk_s : s.M, b_a = (int64_t)lds_u64(note + kWalkBestA), b_d = (int64_t)lds_u64(note + kWalkBestD);
                            if (dep || a_s > b_a || (a_s == b_a && (du_s > b_d || (du_s == b_d && b_has && (!kFloor || e0 + sl > b_e))))) continue;
                            b_has = b_here = true;
                            b_e = e0 + sl;
                            __syncwarp();
                            if (lane == 0) {
                                sts_u64(note + kWalkBestA, (uint64_t)a_s);
                                sts_u64(note + kWalkBestD, (uint64_t)du_s);
                                sts_u64(note + kWalkBestPk, (uint64_t)pk_s);
                                sts_u32(note + kWalkBestAt, (uint32_t)at);
                                sts_u32(note + kWalkQd, (uint32_t)qd_s);
                                sts_u32(note + kWalkJi, (uint32_t)ji_s);
                                sts_u32(note + kWalkX, (uint32_t)x_s);
                                sts_u32(note + kWalkWx, wx_s);
                            }
                            __syncwarp();
                        }
                        if (b_has && E <= 32) {
                            settle();
                            fresh();
                            // the generations behind this one see the new sequence
                            pending = gen == span - 1 ? 0u : (kFull << ((gen + 1) * per)) & drawn;
                            break;
                        }
                    }
                }
            }
            if (b_has) settle();
        }
        __syncwarp();
        const uint32_t n_acc = lds_u32(note + kWalkAcc);
        if (lane == 0 && n_acc) {
            const int64_t pk = (int64_t)lds_u64(note + kWalkPk);
            s.lens[c] = T;
            s.peak[c] = pk;
            s.dur[c] = (int64_t)lds_u64(note + kWalkDu);
            s.status[c] = pk <= s.M ? 1 : 0;
            s.n_acc[c] += (int32_t)n_acc;
            p.peak_at[c] = kFloor ? tp : -tp;
        }
        __syncwarp();
    }
}

}  // namespace moc
