// Device code of the interval-form checker: a batch of solutions in the paper's own variables
// (starts s, ends e, activity flags a of the retention intervals; Section 2, Eqs. 1-8, and the staged
// event domain of "Complexity Reduction by Enforcing an Initial Topological Ordering") is checked
// constraint by constraint, with the duration (Eq. 1) and the peak of the usage of Eq. 4.
//
// One warp per solution at a time, warp-synchronous, a block being a few warps that share nothing but the launch;
// or, where an SM would have few warps at work (bitmaps of a large domain, small batches), a block of up to 16 warps per
// solution.  The event domain can be far larger than the number of intervals
// (n(n+1)/2 staged events for n*C intervals), so usage is not accumulated per event.  It can only
// rise at the start of an active interval, hence the peak is the largest usage over those start
// events.  A bitmap over the domain marks them, a prefix count over its words turns an event t into
// rank(t) = number of marked events <= t, and every active interval [s, e] with s <= e adds m to the
// marked events rank(s) .. rank(e): a difference array over at most n*C ranks and one prefix sum.
// The same ranks order the active intervals into the execution sequence the solution stands for.
//
// Bound: latency at the few warps whose bitmaps fit an SM (staged domain, n = 442: 97903 events, 12 KB a warp).  The rank
// bases therefore take 16 bits per four bitmap words, and the staged rule a 32-bit float root: staged, 16384 solutions,
// n = 442: 1355 -> 529 us (6 -> 9 warps per SM), n = 900, 2000 solutions: 900 -> 559 us, n = 100: 66.7 -> 58.8 us.  Blocks per solution:
// n = 442, 6000 solutions 222 -> 101 us, 148 39 -> 11; n = 932, 1500 solutions 433 -> 68.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace moc {

constexpr int kIvMaxWarps = 8;   // warps (solutions in flight) per block, fewer when shared memory is short
constexpr int kIvMaxTeam = 16;   // warps per solution, where few solutions are in flight
constexpr int32_t kIvEq2 = 1, kIvEq3 = 2, kIvEq4 = 4, kIvEq5 = 8, kIvEq6 = 16, kIvEq7 = 32, kIvEq8 = 64, kIvStage = 128;
constexpr int kIvMaxC = 8;       // slots per node held in registers

struct IntervalParams {
    int32_t n, C;
    const int32_t* succ_start;   // n+1, successor lists (CSR)
    const int32_t* succ;
    const int64_t* w;            // n durations
    const int64_t* m;            // n output sizes
    const int32_t* s;            // B * n * C each, [B][n][C]
    const int32_t* e;
    const int32_t* a;
    int32_t B;
    int32_t D;                   // events are 1..D
    const int32_t* topo_index;   // n (1-based index in the input topological order): staged model; nullptr: plain
    int64_t M;
    int64_t* out_peak;
    int64_t* out_dur;
    int32_t* out_mask;
    int32_t* out_seqs;           // B rows of n*C ints, or nullptr
    int32_t* out_lens;           // B, or nullptr
    uint32_t words;              // bitmap words: (D + 32) / 32, rounded up to a multiple of 4  (bit t of the bitmap = event t, bit 0 unused)
    uint32_t warp_bytes;         // shared memory of one warp
    int32_t team;                // a block per solution (else a warp)
    int32_t byte_marks;          // plain model, and two bytes per event fit the space of the difference array
};

// Shared memory of one warp, in this order: bitmap of active starts [words], bitmap of all starts
// [words] (plain model only, else absent; words a multiple of 4), rank base per four words (16 bits each: there are
// fewer than 65536 intervals on chip), difference array [n*C + 2]
// (MemT), then -- when it fits -- the solution: start of every active slot (0 = inactive) and end of
// every slot, [n*C] int32 each, written while the solution is read from HBM for the only time.
__host__ __device__ inline size_t interval_bitmap_bytes(uint32_t words, bool plain) {
    return ((size_t)words * 4 * (plain ? 2 : 1) + (size_t)words / 4 * 2 + 15) & ~size_t(15);
}
__host__ __device__ inline size_t interval_clear_bytes(uint32_t words, int64_t K, bool plain, size_t mem_sz) {
    return interval_bitmap_bytes(words, plain) + (((size_t)(K + 2) * mem_sz + 15) & ~size_t(15));
}
__host__ __device__ inline size_t interval_stage_bytes(int64_t K, size_t pos_sz) { return ((size_t)K * 2 * pos_sz + 15) & ~size_t(15); }

// exact test "x = j(j-1)/2 for an integer j >= jmin"; 0 <= x < 2^30
__device__ __forceinline__ bool is_triangular_from(uint32_t x, uint32_t jmin) {
    // j = (1 + sqrt(1 + 8x)) / 2 up to rounding (j < 46342, an error below 1), corrected to the integer root
    uint32_t j = max((uint32_t)((1.0f + sqrtf(1.0f + 8.0f * (float)x)) * 0.5f), 1u);
    while (j * (j - 1) / 2 > x) --j;
    while ((j + 1) * j / 2 <= x) ++j;
    return j * (j - 1) / 2 == x && j >= jmin;
}

__device__ __forceinline__ void iv_add(int32_t* p, int32_t v) { atomicAdd(p, v); }
__device__ __forceinline__ void iv_add(int64_t* p, int64_t v) {
    atomicAdd(reinterpret_cast<unsigned long long*>(p), (unsigned long long)v);
}

// kPlain: plain model (Eq. 6) or staged model; CP: slots per node held in registers (>= C); MemT: type
// of the usage sums (int32 when C * sum(m) < 2^31); kStage: the solution is kept in shared memory
// after the first pass (otherwise the second pass reads it again through L1/L2), as PosT (uint16 when
// D < 65536).
// kTeams: p.team may ask for a block per solution (without, a warp has each: eight registers less, which small graphs need to
// fill an SM: n = 60, 16384 solutions 37.0 us, 39.5 with).
template <bool kPlain, int CP, typename MemT, bool kStage, typename PosT, bool kTeams>
__global__ void __launch_bounds__(32 * (kTeams ? kIvMaxTeam : kIvMaxWarps)) check_intervals_kernel(const IntervalParams p) {
    extern __shared__ __align__(16) char smem[];
    // what the warps of a solution tell one another (p.team)
    __shared__ int64_t s_dur[kIvMaxTeam], s_sum[kIvMaxTeam], s_top[kIvMaxTeam];
    __shared__ int32_t s_act[kIvMaxTeam], s_distinct[kIvMaxTeam], s_bits[kIvMaxTeam], s_marks[kIvMaxTeam], s_mask[kIvMaxTeam];
    const int lane = threadIdx.x & 31;
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0);
    const int wpb = blockDim.x >> 5;
    // a solution has this warp or, with p.team, the block
    const bool team = kTeams && p.team != 0;
    const int tid = team ? (int)threadIdx.x : lane, tn = team ? (int)blockDim.x : 32;
    auto sync = [&]() {
        if (team) __syncthreads();
        else __syncwarp();
    };
    // sum of the warps' values, which have been written to `part` in front of the last barrier
    auto warps_sum = [&](const int32_t* part) -> int32_t { return (int32_t)__reduce_add_sync(0xFFFFFFFFu, lane < wpb ? (uint32_t)part[lane] : 0u); };
    const int32_t n = p.n, C = p.C, K = n * C;
    char* ws = smem + (team ? (size_t)0 : (size_t)warp * p.warp_bytes);
    uint32_t* bm_act = reinterpret_cast<uint32_t*>(ws);
    uint32_t* bm_all = bm_act + p.words;                               // plain model only
    uint16_t* rbase = reinterpret_cast<uint16_t*>(bm_act + p.words * (kPlain ? 2u : 1u));
    MemT* delta = reinterpret_cast<MemT*>(ws + interval_bitmap_bytes(p.words, kPlain));
    PosT* sS = reinterpret_cast<PosT*>(ws + interval_clear_bytes(p.words, K, kPlain, sizeof(MemT)));
    PosT* sE = sS + K;
    // plain model: two bytes per event during pass 1 (active start, any start), in the space of the difference
    // array when it is large enough (byte_marks)
    const uint32_t by_stride = ((uint32_t)p.D + 1u + 15u) & ~15u;
    uint8_t* by_act = reinterpret_cast<uint8_t*>(delta);
    constexpr uint32_t kFull = 0xFFFFFFFFu;
    const int nz = (int)(interval_clear_bytes(p.words, K, kPlain, sizeof(MemT)) >> 4);

    for (int32_t b = team ? blockIdx.x : blockIdx.x * wpb + warp; b < p.B; b += team ? gridDim.x : gridDim.x * wpb) {
        const int32_t* __restrict__ gs = p.s + (int64_t)b * K;
        const int32_t* __restrict__ ge = p.e + (int64_t)b * K;
        const int32_t* __restrict__ ga = p.a + (int64_t)b * K;
        {
            int4* z4 = reinterpret_cast<int4*>(ws);
            for (int i = tid; i < nz; i += tn) z4[i] = make_int4(0, 0, 0, 0);
        }
        sync();
        // C = 2 and the three rows of this solution start on 8 bytes: slots are read in pairs
        const bool pairs = C == 2 && ((reinterpret_cast<uintptr_t>(gs) | reinterpret_cast<uintptr_t>(ge) | reinterpret_cast<uintptr_t>(ga)) & 7) == 0;

        // ---- pass 1, per node: read the C slots; Eq. 8; Eqs. 1, 2, 3, 7; mark the starts in the bitmaps
        // (Eq. 6 / staged rule).  A start outside the domain marks nothing; the marks are used only when
        // Eq. 8 holds everywhere.
        int32_t mask = 0, n_act = 0, n_distinct = 0;
        int64_t dur = 0;
        for (int32_t v = tid; v < n; v += tn) {
            int32_t sv[CP], ev[CP], av[CP];
            if (CP == 2 && pairs) {                         // two slots per node: one 8-byte load per array
                const int2 s2 = __ldg(reinterpret_cast<const int2*>(gs) + v), e2 = __ldg(reinterpret_cast<const int2*>(ge) + v),
                           a2 = __ldg(reinterpret_cast<const int2*>(ga) + v);
                sv[0] = s2.x; sv[1] = s2.y;
                ev[0] = e2.x; ev[1] = e2.y;
                av[0] = a2.x; av[1] = a2.y;
            } else {
#pragma unroll
                for (int i = 0; i < CP; ++i) {
                    const bool in = i < C;
                    sv[i] = in ? __ldg(gs + v * C + i) : 0;
                    ev[i] = in ? __ldg(ge + v * C + i) : 0;
                    av[i] = in ? __ldg(ga + v * C + i) : 0;
                }
            }
            const int64_t wv = __ldg(&p.w[v]);
            int64_t k = 0;
            if (!kPlain) {
                k = (int64_t)__ldg(&p.topo_index[v]);
                if ((int64_t)sv[0] != k * (k + 1) / 2) mask |= kIvStage;
            }
            if (av[0] != 1) mask |= kIvEq7;
            if (kStage && CP == 2 && sizeof(PosT) == 2 && C == 2) {       // both slots in one 32-bit store per array
                reinterpret_cast<uint32_t*>(sS)[v] = (uint32_t)(uint16_t)(av[0] == 1 ? sv[0] : 0) | (uint32_t)(uint16_t)(av[1] == 1 ? sv[1] : 0) << 16;
                reinterpret_cast<uint32_t*>(sE)[v] = (uint32_t)(uint16_t)ev[0] | (uint32_t)(uint16_t)ev[1] << 16;
            }
#pragma unroll
            for (int i = 0; i < CP; ++i) {
                if (i < C) {
                    const bool in_dom = sv[i] >= 1 && sv[i] <= p.D;
                    if (!in_dom || ev[i] < 1 || ev[i] > p.D || (av[i] != 0 && av[i] != 1)) mask |= kIvEq8;
                    if (sv[i] > ev[i]) mask |= kIvEq2;
                    if (i + 1 < CP && i + 1 < C && ev[i] > sv[i + 1]) mask |= kIvEq3;
                    const bool act = av[i] == 1;
                    if (act) { dur += wv; ++n_act; }
                    if (kStage && !(CP == 2 && sizeof(PosT) == 2 && C == 2)) {
                        sS[v * C + i] = (PosT)(act ? sv[i] : 0);
                        sE[v * C + i] = (PosT)ev[i];
                    }
                    if (in_dom) {
                        // Each node marks its distinct starts; Eq. 6 holds iff no two nodes marked the same event,
                        // i.e. iff as many events end up marked as marks were made.  With byte marks (plain
                        // stores: marks of neighbouring events share a word without colliding) the two bitmaps
                        // are made from the bytes below; otherwise the marks go straight into them.
                        const uint32_t bit = 1u << (sv[i] & 31);
                        if (act) {
                            if (kPlain && p.byte_marks) by_act[2 * sv[i]] = 1;
                            else atomicOr(&bm_act[sv[i] >> 5], bit);
                            if (!kPlain && !((int64_t)sv[i] >= k && is_triangular_from((uint32_t)((int64_t)sv[i] - k), (uint32_t)k))) mask |= kIvStage;
                        }
                        if (kPlain) {
                            bool seen = false;
#pragma unroll
                            for (int i2 = 0; i2 < i; ++i2) seen |= sv[i2] == sv[i];
                            if (!seen) {
                                if (p.byte_marks) by_act[2 * sv[i] + 1] = 1;
                                else atomicOr(&bm_all[sv[i] >> 5], bit);
                                ++n_distinct;
                            }
                        }
                    }
                }
            }
        }
        int32_t total_act = (int32_t)__reduce_add_sync(kFull, (uint32_t)n_act), distinct = kPlain ? (int32_t)__reduce_add_sync(kFull, (uint32_t)n_distinct) : 0;
        if (team && lane == 0) {
            s_act[warp] = total_act;
            s_distinct[warp] = distinct;
        }
        if (team ? __syncthreads_or(mask & kIvEq8) != 0 : __any_sync(kFull, mask & kIvEq8) != 0) {     // nothing else is evaluated
            if (tid == 0) {
                p.out_mask[b] = kIvEq8;
                p.out_peak[b] = -1;
                p.out_dur[b] = -1;
                if (p.out_lens) p.out_lens[b] = -1;
            }
            __syncwarp();
            continue;
        }
        __syncwarp();
        if (team) {
            total_act = warps_sum(s_act);
            distinct = warps_sum(s_distinct);
        }
        if (kPlain && p.byte_marks) {
            // bytes -> bitmaps: the warp reads the byte pairs of 32 consecutive events, the two ballots are their
            // bitmap words, kept by lane (word mod 32) and stored 32 words at a time; then the bytes, which
            // borrowed the difference array, are cleared again
            const uint16_t* by2 = reinterpret_cast<const uint16_t*>(by_act);
            for (uint32_t w0 = team ? 32u * (uint32_t)warp : 0u; w0 < p.words; w0 += (uint32_t)tn) {
                uint32_t keep_a = 0, keep_l = 0;
                const uint32_t w1 = min(p.words, w0 + 32u);
                for (uint32_t wd = w0; wd < w1; ++wd) {
                    const int32_t t = (int32_t)(wd * 32u) + lane;
                    const uint32_t pr = t <= p.D ? (uint32_t)by2[t] : 0u;
                    const uint32_t ba = __ballot_sync(kFull, (pr & 0xFFu) != 0), bl = __ballot_sync(kFull, (pr >> 8) != 0);
                    if (lane == (int)(wd - w0)) {
                        keep_a = ba;
                        keep_l = bl;
                    }
                }
                if (w0 + lane < w1) {
                    bm_act[w0 + lane] = keep_a;
                    bm_all[w0 + lane] = keep_l;
                }
            }
            sync();
            int4* z4 = reinterpret_cast<int4*>(by_act);
            for (uint32_t i = tid; i < (2u * by_stride + 15u) / 16u; i += tn) z4[i] = make_int4(0, 0, 0, 0);
            sync();
        }

        // ---- rank base of every four bitmap words: exclusive prefix sum of the popcounts
        int32_t R;
        {
            const uint32_t groups = p.words / 4, per = ((groups + (uint32_t)tn - 1u) / (uint32_t)tn) | 1u;      // odd: the lanes' vectors fall into different banks
            const uint32_t g0 = min(groups, (uint32_t)tid * per), g1 = min(groups, g0 + per);
            const uint4* v4 = reinterpret_cast<const uint4*>(bm_act);
            uint32_t cnt = 0;
            for (uint32_t i = g0; i < g1; ++i) {
                const uint4 v = v4[i];
                cnt += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
            }
            uint32_t incl = cnt;
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t o = __shfl_up_sync(kFull, incl, d);
                if (lane >= d) incl += o;
            }
            uint32_t run = incl - cnt;
            R = (int32_t)__shfl_sync(kFull, incl, 31);       // number of distinct active starts
            if (team) {
                if (lane == 0) s_marks[warp] = R;
                __syncthreads();
                run += __reduce_add_sync(kFull, lane < warp ? (uint32_t)s_marks[lane] : 0u);
                R = warps_sum(s_marks);
            }
            for (uint32_t i = g0; i < g1; ++i) {
                rbase[i] = (uint16_t)run;
                const uint4 v = v4[i];
                run += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
            }
        }
        int32_t bits = 0;
        if (kPlain) {
            for (uint32_t i = tid; i < p.words; i += tn) bits += __popc(bm_all[i]);
            bits = __reduce_add_sync(kFull, bits);
        }
        const bool has_seq = R == total_act;
        int32_t* row = (p.out_seqs != nullptr && has_seq) ? p.out_seqs + (int64_t)b * K : nullptr;
        sync();
        auto rank = [&](int32_t t) -> int32_t {   // marked events <= t
            const uint4 v = reinterpret_cast<const uint4*>(bm_act)[t >> 7];
            const int32_t w = t >> 5 & 3;
            const uint32_t upto = 0xFFFFFFFFu >> (31 - (t & 31));       // of word w; the words in front of it count whole
            return (int32_t)rbase[t >> 7] + __popc(w == 0 ? v.x & upto : v.x) + (w < 1 ? 0 : __popc(w == 1 ? v.y & upto : v.y)) +
                   (w < 2 ? 0 : __popc(w == 2 ? v.z & upto : v.z)) + (w < 3 ? 0 : __popc(v.w & upto));
        };
        // start (0 = inactive) and end of slot i of node v
        // both slots of node v at once (C = 2, positions staged in 16 bits)
        constexpr bool kPairStage = kStage && CP == 2 && sizeof(PosT) == 2;
        auto start_pair = [&](int32_t v) -> uint32_t { return reinterpret_cast<const uint32_t*>(sS)[v]; };
        auto end_pair = [&](int32_t v) -> uint32_t { return reinterpret_cast<const uint32_t*>(sE)[v]; };
        auto slot = [&](int32_t v, int32_t i, int32_t& s_out, int32_t& e_out) {
            if (kStage) {
                s_out = (int32_t)sS[v * C + i];
                e_out = (int32_t)sE[v * C + i];
            } else {
                s_out = __ldg(ga + v * C + i) == 1 ? __ldg(gs + v * C + i) : 0;
                e_out = __ldg(ge + v * C + i);
            }
        };

        // ---- pass 2, per node u: Eq. 4 (its active intervals with s <= e cover the marked events
        // rank(s)..rank(e)), the sequence, and Eq. 5 for its successors
        for (int32_t u = tid; u < n; u += tn) {
            int32_t us[CP], ue[CP];
            const MemT mv = (MemT)__ldg(&p.m[u]);
            if (kPairStage && C == 2) {
                const uint32_t sp = start_pair(u), ep = end_pair(u);
                us[0] = (int32_t)(sp & 0xFFFFu); us[1] = (int32_t)(sp >> 16);
                ue[0] = (int32_t)(ep & 0xFFFFu); ue[1] = (int32_t)(ep >> 16);
            } else {
#pragma unroll
                for (int j = 0; j < CP; ++j) {
                    us[j] = 0;
                    ue[j] = 0;
                    if (j < C) slot(u, j, us[j], ue[j]);
                }
            }
#pragma unroll
            for (int j = 0; j < CP; ++j) {
                if (us[j] != 0) {
                    const int32_t r = rank(us[j]);
                    if (us[j] <= ue[j]) {
                        iv_add(&delta[r], mv);
                        iv_add(&delta[rank(ue[j]) + 1], (MemT)(-mv));
                    }
                    if (row) row[r - 1] = u;
                } else {
                    us[j] = INT32_MAX - 1;      // an inactive slot serves nobody
                    ue[j] = 0;
                }
            }
            // Eq. 5: every active start t of a successor lies in (us, ue] of one slot of u, tested as
            // (t - lo) <= len in unsigned arithmetic with lo = us + 1, len = ue - lo; a slot that serves nobody
            // (inactive, or ue <= us) gets lo = 2^32 - 1, len = 0, which no t >= 1 satisfies
            uint32_t lo5[CP], len5[CP];
#pragma unroll
            for (int j = 0; j < CP; ++j) {
                const bool serves = ue[j] > us[j];
                lo5[j] = serves ? (uint32_t)us[j] + 1u : 0xFFFFFFFFu;
                len5[j] = serves ? (uint32_t)(ue[j] - us[j] - 1) : 0u;
            }
            const int32_t e0 = __ldg(&p.succ_start[u]), e1 = __ldg(&p.succ_start[u + 1]);
            for (int32_t q = e0; q < e1; ++q) {
                const int32_t v = __ldg(&p.succ[q]);
                uint32_t tp = 0;
                if (kPairStage && C == 2) tp = start_pair(v);
#pragma unroll
                for (int i = 0; i < CP; ++i) {
                    if (i < C) {
                        int32_t t, te = 0;
                        if (kPairStage && C == 2) t = (int32_t)(i == 0 ? tp & 0xFFFFu : tp >> 16);
                        else slot(v, i, t, te);
                        bool found = t == 0;                    // an inactive slot of the successor asks for nothing
#pragma unroll
                        for (int j = 0; j < CP; ++j) found |= (uint32_t)t - lo5[j] <= len5[j];
                        if (!found) mask |= kIvEq5;
                    }
                }
            }
        }
        sync();

        // ---- prefix sum over the ranks 1..R and its maximum: a thread owns a run of consecutive ranks
        int64_t peak, carry;
        {
            const int32_t per = (R + tn - 1) / tn;
            const int32_t r0 = min(R, tid * per) + 1, r1 = min(R, tid * per + per) + 1;   // ranks [r0, r1)
            int64_t sum = 0, top = INT64_MIN;
            for (int32_t r = r0; r < r1; ++r) {
                sum += (int64_t)delta[r];
                top = sum > top ? sum : top;
            }
            int64_t incl = sum;
            for (int d = 1; d < 32; d <<= 1) {
                const int64_t o = __shfl_up_sync(kFull, incl, d);
                if (lane >= d) incl += o;
            }
            // largest usage in the warp's runs, from the usage in front of the warp on
            peak = r1 > r0 ? incl - sum + top : (team ? INT64_MIN : 0);
            for (int d = 16; d > 0; d >>= 1) {
                const int64_t o = __shfl_xor_sync(kFull, peak, d);
                peak = o > peak ? o : peak;
            }
            carry = __shfl_sync(kFull, incl, 31);
        }
        // ---- duration, flags, outputs
        for (int d = 16; d > 0; d >>= 1) dur += __shfl_xor_sync(kFull, dur, d);
        mask = __reduce_or_sync(kFull, mask);
        if (team) {
            if (lane == 0) {
                s_sum[warp] = carry;
                s_top[warp] = peak;
                s_dur[warp] = dur;
                s_mask[warp] = mask;
                s_bits[warp] = bits;
            }
            __syncthreads();
            if (warp != 0) continue;
            const bool in = lane < wpb;
            const int64_t part = in ? s_sum[lane] : 0, most = in ? s_top[lane] : INT64_MIN;
            int64_t incl = part;
            for (int d = 1; d < 32; d <<= 1) {
                const int64_t o = __shfl_up_sync(kFull, incl, d);
                if (lane >= d) incl += o;
            }
            peak = most == INT64_MIN ? 0 : incl - part + most;         // usages are 0 or more
            dur = in ? s_dur[lane] : 0;
            for (int d = 16; d > 0; d >>= 1) {
                const int64_t o = __shfl_xor_sync(kFull, peak, d);
                peak = o > peak ? o : peak;
                dur += __shfl_xor_sync(kFull, dur, d);
            }
            mask = __reduce_or_sync(kFull, in ? s_mask[lane] : 0);
            bits = warps_sum(s_bits);
        }
        if (kPlain && bits != distinct) mask |= kIvEq6;
        if (peak > p.M) mask |= kIvEq4;
        if (tid == 0) {
            p.out_mask[b] = mask;
            p.out_peak[b] = peak;
            p.out_dur[b] = dur;
            if (p.out_lens) p.out_lens[b] = has_seq ? R : -1;
        }
        __syncwarp();
    }
}

}  // namespace moc
