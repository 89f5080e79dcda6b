// Interval-form checker for the plain event domain with two slots per node (C = 2, D <= 32766: the setting of
// Section 4.3 with D = C n of Section 2).  Same quantities as check_intervals_kernel (moc_interval_kernels.cuh),
// which serves every other case; a warp per solution, the graph staged once per block.
//
// What differs.  The domain is about as large as the number of slots, so nothing is compressed to ranks: the usage
// of Eq. 4 is a difference array over the events themselves, and the execution sequence is read off an array
// that holds, per event, the node whose active interval starts there (plain 16-bit stores), 32 events at a time
// with ballots, so that the row is written in order with full sectors (scattered 4-byte stores before) and
// the entries behind it in the same pass.  Eq. 5 walks the successor tiles of the evaluation kernel (two nodes per lane,
// uniform trip counts) with both starts of a successor tested at once: with lo = s + 1 and len = e - lo per slot,
//     max(t - lo, len) = len  iff  t in (s, e]            (one packed 16-bit operation per slot, modulo 2^16)
// and a start is served iff one of the two differences vanishes.
//
// An inactive slot's start is replaced by that of the other slot (it then asks for nothing new); a solution in which
// some node has no active slot at all takes a plain loop over the edges instead.
//
// Bound: instruction issue (58 % of the slots), the shared-memory data pipe (52 %) and the latency of the solution's loads.
// n = 442, D = 884, 16384 solutions with their sequences: 179.8 -> 90.5 us, where the 207 MB of DRAM traffic alone
// take 32; 91.9 -> 88.5 with both slots of a node in one packed word (36 operations for 55 in a half of a tile) and the walk over the
// events ended at the last active start.  Taken back: the next solution fetched into L2 (+5 us and 60 MB of traffic), two nodes'
// loads ahead instead of four at a time (+3.5), one mark for active and inactive starts (+2.7, with a third fewer stores).
#pragma once
#include "moc_interval_kernels.cuh"
#include "moc_pair_kernel.cuh"

namespace moc {

constexpr int kIvPlainThreads = 896;

struct IntervalPlainParams {
    IntervalParams q;
    int32_t n_tiles, split;      // as in PairParams
    const void* rec;             // node records of the warp-per-sequence layout
    const uint32_t* sell;        // its successor tiles; a used-up list repeats a successor, a sink reads its own word
    uint32_t rec_bytes, sell_bytes;     // graph, once per block
    uint32_t word_bytes;         // start words (4 (n + 2), rounded to 16) without the word of empty slots behind them
    uint32_t event_bytes;        // marks, later the difference array
    bool fill;                   // write -1 behind the sequences (and to the rows without one)
};

// Bytes of the event area of one warp: marks (2 + 1 bytes per event), or deltas in a whole odd number of 16-byte
// vectors per lane.
__host__ __device__ inline size_t interval_plain_event_bytes(int32_t D, size_t mem_sz) {
    const size_t vec = ((size_t)D + 2 + 16 / mem_sz - 1) / (16 / mem_sz), marks = (3 * ((size_t)D + 64) + 15) / 16;
    return 32 * 16 * ((((vec > marks ? vec : marks) + 31) / 32) | 1);
}

// 0xFFFF in each half whose bit 15 is set, else 0 (prmt's sign mode, which __byte_perm masks out)
__device__ __forceinline__ uint32_t iv_half_signs(uint32_t x) {
    uint32_t r;
    asm("prmt.b32 %0, %1, %1, 0xBB99;" : "=r"(r) : "r"(x));
    return r;
}

template <typename MemT>
__global__ void __launch_bounds__(kIvPlainThreads, 1) check_plain_kernel(const IntervalPlainParams pp) {
    extern __shared__ __align__(16) char smem[];
    const IntervalParams& p = pp.q;
    constexpr uint32_t kRecB = sizeof(MemT) == 4 ? 8u : 16u, kFull = 0xFFFFFFFFu;
    constexpr int kShift = sizeof(MemT) == 4 ? 2 : 3;
    const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
    const int warp = __shfl_sync(kFull, (int)(threadIdx.x >> 5), 0);
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem);
    {
        // asynchronous copies: the graph is first read in pass 2
        auto copy = [&](uint32_t to, const void* from, uint32_t bytes) {
            for (uint32_t i = 16u * threadIdx.x; i < bytes; i += 16u * blockDim.x)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + i), "l"(reinterpret_cast<const char*>(from) + i) : "memory");
        };
        copy(sbase, pp.rec, pp.rec_bytes);
        copy(sbase + pp.rec_bytes, pp.sell, pp.sell_bytes);
    }
    const int32_t n = p.n, K = 2 * n, D = p.D;
    const uint32_t word_set = pp.word_bytes + kPairWordTail;
    const uint32_t sa = sbase + pp.rec_bytes + pp.sell_bytes + (uint32_t)warp * (2u * word_set + pp.event_bytes);   // start words
    const uint32_t ea = sa + word_set;                               // end words: e | active << 15 per slot
    const uint32_t da = ea + word_set;                               // events
    const uint32_t all = da + 2u * (uint32_t)((D + 64) & ~31);       // byte marks of all starts, behind the owners (16 bits)
    const uint32_t rec0 = sbase + kRecB * (uint32_t)lane, sell0 = sbase + pp.rec_bytes + 4u * (uint32_t)lane;
    if (lane == 0) {
        sts_u32(sa + pp.word_bytes, 0u);          // empty node slots: inactive
        sts_u32(ea + pp.word_bytes, 0u);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    auto clear_events = [&]() {
        for (uint32_t o = 16u * (uint32_t)lane; o < pp.event_bytes; o += 512u)
            asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(da + o), "r"(0) : "memory");
        __syncwarp();
    };

    const int32_t step = gridDim.x * wpb;
    for (int32_t b = blockIdx.x * wpb + warp; b < p.B; b += step) {
        const int2* gs = reinterpret_cast<const int2*>(p.s + (int64_t)b * K);
        const int2* ge = reinterpret_cast<const int2*>(p.e + (int64_t)b * K);
        const int2* ga = reinterpret_cast<const int2*>(p.a + (int64_t)b * K);
        clear_events();
        // ---- pass 1, per node: Eqs. 1, 2, 3, 7, 8; marks of the starts; the solution on chip.  The tests gather as running
        // extremes that are looked at once: a value outside its domain makes the rest meaningless, but harmless.
        uint32_t far = 0, flag = 0, first = 1, none = 1, n_act = 0, n_same = 0, dur_hi = 0;
        int32_t late = INT32_MIN, lap = INT32_MIN;
        uint64_t dur_lo = 0;
        auto node = [&](uint32_t v4, const int2 s2, const int2 e2, const int2 a2, const uint2 w2) {
            far = __viaddmax_u32((uint32_t)s2.x, 0xFFFFFFFFu, far);           // Eq. 8: largest s - 1, e - 1 and a
            far = __viaddmax_u32((uint32_t)s2.y, 0xFFFFFFFFu, far);
            far = __viaddmax_u32((uint32_t)e2.x, 0xFFFFFFFFu, far);
            far = __viaddmax_u32((uint32_t)e2.y, 0xFFFFFFFFu, far);
            const uint32_t a0 = (uint32_t)a2.x, a1 = (uint32_t)a2.y;
            flag = max(flag, a0 | a1);
            late = max(late, max(s2.x - e2.x, s2.y - e2.y));                  // Eq. 2: s > e
            lap = max(lap, e2.x - s2.y);                                      // Eq. 3: e > next s
            first = min(first, a0);                                           // Eq. 7
            none = min(none, a0 | a1);
            n_act += a0 + a1;
            dur_lo += (uint64_t)w2.x * (a0 + a1);
            dur_hi += w2.y * (a0 + a1);
            n_same += s2.x == s2.y ? 1u : 0u;
            const int32_t t0 = a0 ? s2.x : (a1 ? s2.y : 0), t1 = a1 ? s2.y : t0;
            sts_u32(sa + v4, __byte_perm((uint32_t)t0, (uint32_t)t1, 0x5410));
            sts_u32(ea + v4, __byte_perm((uint32_t)e2.x, (uint32_t)e2.y, 0x5410) | a0 << 15 | a1 << 31);
            const uint32_t m0 = min((uint32_t)s2.x, (uint32_t)D), m1 = min((uint32_t)s2.y, (uint32_t)D);
            asm volatile("st.shared.u8 [%0], %1;" ::"r"(all + m0), "r"(1) : "memory");
            asm volatile("st.shared.u8 [%0], %1;" ::"r"(all + m1), "r"(1) : "memory");
            if (a0) sts_u16(da + 2u * m0, (v4 >> 2) + 1u);
            if (a1) sts_u16(da + 2u * m1, (v4 >> 2) + 1u);
        };
        const uint2* gw = reinterpret_cast<const uint2*>(p.w);
        for (int32_t v = lane; v < n; v += 128) {             // four nodes' loads in flight
            int2 s4[4], e4[4], a4[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int32_t u = min(v + 32 * k, n - 1);
                s4[k] = __ldg(gs + u);
                e4[k] = __ldg(ge + u);
                a4[k] = __ldg(ga + u);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (v + 32 * k < n) node(4u * (uint32_t)(v + 32 * k), s4[k], e4[k], a4[k], __ldg(gw + v + 32 * k));
        }
        int32_t* row = p.out_seqs ? p.out_seqs + (int64_t)b * K : nullptr;
        if (__any_sync(kFull, far >= (uint32_t)D || flag > 1u)) {     // Eq. 8: nothing else is evaluated
            if (lane == 0) {
                p.out_mask[b] = kIvEq8;
                p.out_peak[b] = -1;
                p.out_dur[b] = -1;
                if (p.out_lens) p.out_lens[b] = -1;
            }
            if (pp.fill && row)
                for (int32_t i = lane; i < K; i += 32) row[i] = -1;
            __syncwarp();
            continue;
        }
        int32_t mask = (late > 0 ? kIvEq2 : 0) | (lap > 0 ? kIvEq3 : 0) | (first != 1u ? kIvEq7 : 0);
        const bool idle = none == 0;              // some node has no active slot
        __syncwarp();
        // ---- events: distinct starts (Eq. 6: as many as the nodes marked), distinct active starts, and the sequence
        const int32_t total = (int32_t)__reduce_add_sync(kFull, n_act), n_ev = (D + 32) & ~31;
        {
            uint32_t marked = 0;
            for (uint32_t o = 4u * (uint32_t)lane; o < (uint32_t)n_ev; o += 128u) marked = __dp4a(lds_u32(all + o), 0x01010101u, marked);
            if ((int32_t)__reduce_add_sync(kFull, marked) != 2 * n - (int32_t)__reduce_add_sync(kFull, n_same)) mask |= kIvEq6;
        }
        auto owner_of = [&](int32_t t) -> uint32_t {
            uint32_t owner;
            asm volatile("{\n\t.reg .u16 h;\n\tld.shared.u16 h, [%1];\n\tcvt.u32.u16 %0, h;\n\t}" : "=r"(owner) : "r"(da + 2u * (uint32_t)t) : "memory");
            return owner;
        };
        // The row is written while its length is counted when it may be repaired afterwards (two active intervals with
        // one start leave no sequence), else after the count.
        int32_t R = 0;
        for (int pass = (pp.fill && row) ? 1 : 0; pass < 2; ++pass) {
            if (pass == 1 && (!row || (!pp.fill && R != total))) break;
            int32_t at = 0;
            for (int32_t t = lane; t < n_ev; t += 32) {
                const uint32_t owner = owner_of(t), here = __ballot_sync(kFull, owner != 0);
                if (pass == 1 && owner != 0) row[at + __popc(here & ((1u << lane) - 1u))] = (int32_t)owner - 1;
                at += __popc(here);
                if (at == total) break;          // there are no more active starts than that
            }
            R = at;
        }
        const bool has_seq = R == total;
        if (pp.fill && row)
            for (int32_t i = (has_seq ? R : 0) + lane; i < K; i += 32) row[i] = -1;
        __syncwarp();
        clear_events();
        // ---- pass 2, per node slot: Eq. 4 and Eq. 5
        uint32_t viol = 0, prec = rec0, ps = sell0;
        for (int d = 0; d < pp.n_tiles; ++d, prec += 64u * kRecB) {
            uint32_t nlo[2][2], len[2][2];        // [slot][half]: -(s + 1) and e - s - 1 of the half's node, in both 16-bit halves
            uint32_t rows_x = 0;
            const uint32_t e_first = lds_u32(ps);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t x;
                Amount<MemT> m;
                if constexpr (sizeof(MemT) == 4) {
                    const uint2 r = lds_v2(prec + 32u * kRecB * h);
                    x = r.x;
                    m.v = (MemT)r.y;
                } else {
                    const uint4 r = lds_v4(prec + 32u * kRecB * h);
                    x = r.x;
                    m.lo = r.z;
                    m.hi = r.w;
                }
                if (h == 0) rows_x = x;
                const uint32_t off = x & 0xFFFFu, sp = lds_u32(sa + off), ep = lds_u32(ea + off);
                const bool sink = (h == 0 ? e_first & 0xFFFFu : e_first >> 16) == off;       // no successor: everything is served
                // both slots at once, 16 bits each: 2^15 + e - s (bit 15: e >= s), and with 1 taken off (bit 15: e > s); bit 15 of
                // ep tells that the slot is active
                const uint32_t d = (ep | 0x80008000u) - sp, gap = d - 0x00010001u, held = d & ep;
                const uint32_t serves = iv_half_signs(gap & ep);       // 0xFFFF where the slot is active and e > s
                if (held & 0x8000u) {
                    red_add_amount(da + ((sp & 0xFFFFu) << kShift), m);
                    red_sub_amount(da + (((ep & 0x7FFFu) + 1u) << kShift), m);
                }
                if (held & 0x80000000u) {
                    red_add_amount(da + ((sp >> 16) << kShift), m);
                    red_sub_amount(da + (((ep >> 16 & 0x7FFFu) + 1u) << kShift), m);
                }
                // lo = s + 1 and len = e - lo where the slot serves, else 2^16 - 1 and 0
                const uint32_t ln = sink ? 0xFFFFFFFFu : gap & 0x7FFF7FFFu & serves, nl = sink ? 0u : (serves & ~sp) | (~serves & 0x00010001u);
                nlo[0][h] = __byte_perm(nl, 0u, 0x1010u);
                nlo[1][h] = __byte_perm(nl, 0u, 0x3232u);
                len[0][h] = __byte_perm(ln, 0u, 0x1010u);
                len[1][h] = __byte_perm(ln, 0u, 0x3232u);
            }
            const int rows = __shfl_sync(kFull, (int)(rows_x >> 16), 0);
            uint32_t e = e_first;
            for (int k = 0; k < rows; ++k) {
                ps += 128u;
                const uint32_t r0 = lds_u32(sa + (e & 0xFFFFu)), r1 = lds_u32(sa + (e >> 16));
                if (k + 1 < rows) e = lds_u32(ps);
                viol |= min_u16x2(__viaddmax_u16x2(r0, nlo[0][0], len[0][0]) - len[0][0], __viaddmax_u16x2(r0, nlo[1][0], len[1][0]) - len[1][0]);
                viol |= min_u16x2(__viaddmax_u16x2(r1, nlo[0][1], len[0][1]) - len[0][1], __viaddmax_u16x2(r1, nlo[1][1], len[1][1]) - len[1][1]);
            }
        }
        if (__any_sync(kFull, idle)) {
            // a successor without an active slot asks for nothing: Eq. 5 edge by edge
            viol = 0;
            for (int32_t u = lane; u < n; u += 32) {
                const uint32_t sp = lds_u32(sa + 4u * (uint32_t)u), ep = lds_u32(ea + 4u * (uint32_t)u);
                const uint32_t s0 = sp & 0xFFFFu, s1 = sp >> 16, e0 = (ep & 0x8000u) ? ep & 0x7FFFu : 0u, e1 = ep >> 31 ? ep >> 16 & 0x7FFFu : 0u;
                for (int32_t k = __ldg(p.succ_start + u); k < __ldg(p.succ_start + u + 1); ++k) {
                    const uint32_t r = lds_u32(sa + 4u * (uint32_t)__ldg(p.succ + k));
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const uint32_t t = i == 0 ? r & 0xFFFFu : r >> 16;
                        if (t != 0 && !((t > s0 && t <= e0) || (t > s1 && t <= e1))) viol = 1;
                    }
                }
            }
        }
        if (viol != 0) mask |= kIvEq5;
        __syncwarp();
        // ---- usage per event and its maximum: lane owns V consecutive vectors
        int64_t peak;
        {
            const int V = (int)(pp.event_bytes / 512u);
            uint32_t ad = da + 16u * (uint32_t)(lane * V), lo = 0, hi = 0;
            MemT top = sizeof(MemT) == 8 ? (MemT)INT64_MIN : (MemT)INT32_MIN;
            for (int j = 0; j < V; ++j, ad += 16u) {
                const uint4 q = lds_v4(ad);
                if constexpr (sizeof(MemT) == 4) {
                    lo += q.x; top = max(top, (MemT)lo);
                    lo += q.y; top = max(top, (MemT)lo);
                    lo += q.z; top = max(top, (MemT)lo);
                    lo += q.w; top = max(top, (MemT)lo);
                } else {
                    lo += q.x; hi += q.y;
                    MemT at = split_value(lo, hi, pp.split);
                    top = at > top ? at : top;
                    lo += q.z; hi += q.w;
                    at = split_value(lo, hi, pp.split);
                    top = at > top ? at : top;
                }
            }
            if constexpr (sizeof(MemT) == 4) top += (MemT)(warp_inclusive_sum(lo, lane) - lo);
            else top += split_value(warp_inclusive_sum(lo, lane) - lo, warp_inclusive_sum(hi, lane) - hi, pp.split);
            peak = (int64_t)warp_max_t(top);
        }
        if (peak > p.M) mask |= kIvEq4;
        const int64_t dur = warp_sum64((int64_t)(dur_lo + ((uint64_t)dur_hi << 32)));
        mask = __reduce_or_sync(kFull, mask);
        if (lane == 0) {
            p.out_mask[b] = mask;
            p.out_peak[b] = peak;
            p.out_dur[b] = dur;
            if (p.out_lens) p.out_lens[b] = has_seq ? R : -1;
        }
        __syncwarp();
    }
}

}  // namespace moc
