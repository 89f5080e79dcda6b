// Host side of libmoc_b200.so: graph handle, validation, launch planning and the C ABI declared in
// include/moc.h.  Every step of the evaluation itself runs in the kernels of moc_kernels.cuh.
#include <cuda.h>

#include <algorithm>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <memory>
#include <new>
#include <vector>

#include "moc_host.cuh"

using namespace moc_host;

namespace {
thread_local char g_err[512] = "";
thread_local int g_launches_tl = 0;
}  // namespace
#define g_launches (moc_host::launch_counter())

namespace moc_host {
int fail(int code, const char* fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
    return code;
}
void clear_error() { g_err[0] = 0; }
int& launch_counter() { return g_launches_tl; }
}  // namespace moc_host

namespace {

size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

int live_words(int n) { return n <= 32 ? 1 : (n <= 64 ? 2 : 4); }

// Raises a kernel's dynamic shared-memory limit to all the device offers beside its static part.
cudaError_t raise_smem_limit(const void* fn, size_t smem_optin) {
    cudaFuncAttributes a{};
    cudaError_t e = cudaFuncGetAttributes(&a, fn);
    if (e != cudaSuccess) return e;
    const size_t room = smem_optin > a.sharedSizeBytes ? smem_optin - a.sharedSizeBytes : 0;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)room);
}

int pow2_ceil(int x) {
    int p = 1;
    while (p < x) p <<= 1;
    return p;
}

// Plan of the sequence-per-lane path: the largest group whose state fits beside the graph, with as
// many warps per SM as fit.  Returns nullptr on success, else the reason it cannot serve the graph.
const char* plan_lane(const moc_graph* g, size_t smem_cap, Plan* out) {
    Plan pl = *out;
    const int64_t n = g->n, C = g->C, t_max = C * n;
    if (C > 2) return "C > 2";
    if ((__int128)C * g->sum_w >= ((__int128)1 << 40)) return "C * sum(w) reaches 2^40";
    const bool forced = g->want_kind == MOC_KERNEL_LANE;
    const size_t msz = pl.wide ? 8 : 4;
    for (int li = 0; li < 3; ++li) {
        const int lg = 5 - li, gsz = 1 << lg, S = 32 >> lg;
        const LaneLayout& L = g->lane[li];
        if (!L.ok) continue;
        if (forced && g->want_a && g->want_a != gsz) continue;
        const size_t rec_b = 32 * (size_t)S * L.n_bundles, succ_b = align16(4 * (size_t)L.succ_len),
                     part_b = 2 * align16(32 * msz * ((size_t)gsz + 1)),
                     word_b = moc::lane_special(gsz) + align16((size_t)moc::lane_word_row(gsz) * (n + 1)),
                     delta_b = align16(msz * gsz * (size_t)(t_max + 3));
        const size_t sm = rec_b + succ_b + part_b + word_b + delta_b;
        if (sm > smem_cap) continue;
        int best_w = 0, best_nb = 0, best_kp = 0;
        for (int w = 32; w >= gsz; w -= gsz) {    // a whole number of warps per row of the group
            if (forced && g->want_b && g->want_b != w) continue;
            // pieces of 128 steps fetched ahead per warp: enough for typical rows of about 1.3 n steps
            const int64_t pieces = ((n * 13 / 10 + 6) / 4 + 31) / 32;
            int kp = (int)((pieces * gsz + w - 1) / w);
            kp = std::min(8, std::max(2, (kp + 1) & ~1));
            LaneFn fn = lane_fn(pl.wide, lg, kp);
            if (raise_smem_limit((const void*)fn, g->smem_optin) != cudaSuccess) { cudaGetLastError(); continue; }
            int nb = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, (const void*)fn, w * 32, sm) != cudaSuccess) { cudaGetLastError(); continue; }
            if (nb < 1) continue;
            // as many warps per SM as fit, up to 64; among equals the shape with more blocks
            const int warps = std::min(nb * w, 64), best = std::min(best_nb * best_w, 64);
            if (warps > best || (warps == best && nb > best_nb && w >= 8)) { best_w = w; best_nb = nb; best_kp = kp; }
        }
        if (best_w == 0) continue;
        pl.lane = true;
        pl.lane_fn = lane_fn(pl.wide, lg, best_kp);
        pl.lane_lg = lg;
        pl.G = 32 * best_w / gsz;
        pl.gpc = gsz;
        pl.block = 32 * best_w;
        pl.smem = sm;
        pl.grid = g->sm_count * best_nb;
        pl.sm_count = g->sm_count;
        pl.lane_rec_b = (uint32_t)rec_b; pl.lane_succ_b = (uint32_t)succ_b;
        pl.lane_word_b = (uint32_t)word_b; pl.lane_delta_b = (uint32_t)delta_b;
        pl.valid = true;
        *out = pl;
        return nullptr;
    }
    return "the state of a group of sequences exceeds shared memory in the requested shape, n >= 4096, or a degree above 255";
}

// Shared memory of the block-per-sequence kernel: the state of a sequence and, behind it, the block's copy of the tiles.
struct QuadBytes {
    size_t word, cnt, delta, rec, w, sell, row;
    size_t state() const { return word + cnt + delta; }
    size_t graph() const { return rec + w + sell + row; }
};
QuadBytes quad_bytes(const moc_graph* g, bool wide, bool profile) {
    const size_t n = (size_t)g->n, t_max = (size_t)g->C * n, msz = wide ? 8 : 4;
    QuadBytes z;
    z.word = (g->C <= 2 && !profile ? 1 : 2) * align16(4 * (n + 2)) + 16;
    z.cnt = align16(2 * (n + 2));
    z.delta = align16(msz * (t_max + 4));
    z.rec = (wide ? 16 : 8) * 64 * (size_t)g->n_tiles;
    z.w = 8 * 64 * (size_t)g->n_tiles;
    z.sell = align16(4 * (size_t)g->sell_len);
    z.row = align16(4 * (size_t)g->n_tiles);
    return z;
}

// How the block-per-sequence kernel's code takes a batch: `team` warps on a sequence, `groups` sequences in flight per
// block, one block per SM, with the graph in shared memory.  team = 0: a block per sequence, the graph through L1.
struct QuadShape {
    int team = 0, groups = 0, grid = 0;
};
// Time in microseconds of a batch with u = n / 64 and s sequences per SM, in `rounds` rounds of what an SM holds at a time (fits to 354 batches
// with every team size: n = 24 to 5000, C = 3, 4, B = 1 to 18944; mean error 5 % with 32-bit sums):
//     a warp per sequence         4.3 + rounds (1.5 + (0.19 + 0.31 C) u) + s (0.07 + 0.009 C u)
//     t warps per sequence        5.0 + rounds (1.0 + (0.15 + 0.28 C) u / t) + s (0.09 + 0.054 t + 0.012 C u)
//     a block of 64 w threads     5.3 + rounds (1.3 + (0.40 + 0.15 C) u / w + 0.046 w) + s (0.10 + 0.040 w + 0.010 C u)
// The smallest of them costs on the mean, against always taking the fastest, 0.3 % at C = 3 and 1.7 % at C = 4 (108 batches), with 64-bit sums
// 0.5 and 1.4 % (330 batches), 2 and 7 % or less in nine of ten, 22 % at worst.  64-bit sums take 4 to 20 % longer than the lines, much the
// same on all three, so that a factor on one line only costs and lines of their own gain 0.3 %.  Against the version with a block per sequence for
// every batch they are faster by 1.20 (C = 3) and 1.16 (C = 4) on the mean of 112 batches; n = 1500, C = 4, B = 1776 (53 -> 58 us) and n = 700, C = 4,
// B = 592 (13.3 -> 14.3) lose.  Before / now (C = 3): n = 153,
// B = 18944 68 -> 39 us, n = 24 45 -> 21, n = 442, B = 4736 33 -> 27, n = 1000, B = 1776 26.9 -> 24.8.
double quad_block_cost(int64_t n, int32_t C, int64_t per_sm, int blocks, int w) {
    const double u = (double)n / 64.0, rounds = (double)((per_sm + blocks - 1) / blocks);
    return 5.3 + rounds * (1.27 + (0.40 + 0.15 * C) * u / w + 0.046 * w) + (double)per_sm * (0.10 + 0.040 * w + 0.010 * C * u);
}
QuadShape quad_shape(const moc_graph* g, int32_t B, bool profile) {
    QuadShape best;
    const bool wide = g->sum_m > (int64_t)INT32_MAX / g->C;
    if (!g->n_tiles || g->C > 4 || g->sum_w >= (int64_t)1 << moc::kPairCntShift || (wide && !g->split_ok)) return best;
    if (g->want_kind == MOC_KERNEL_BLOCK && g->want_a && !profile) return best;
    const QuadBytes z = quad_bytes(g, wide, profile);
    if (z.graph() + z.state() + 2048 > g->smem_optin) return best;
    const int64_t per_sm = ((int64_t)B + g->sm_count - 1) / g->sm_count, fit = (int64_t)((g->smem_optin - 2048 - z.graph()) / z.state());
    const double u = (double)g->n / 64.0;
    const int32_t C = g->C;
    double least = 0;
    auto offer = [&](double cost, int team, int64_t groups) {
        if (least != 0 && cost >= least) return;
        least = cost;
        best.team = team;
        best.groups = (int)groups;
    };
    for (int w = 1; w <= 16; w <<= 1) {         // registers: 64 a thread
        const int64_t blocks = std::min<int64_t>((int64_t)((g->smem_optin + 1024) / (z.state() + 2048)), 16 / w);
        if (blocks > 0) offer(quad_block_cost(g->n, C, per_sm, (int)blocks, w), 0, 0);
    }
    for (int team = 1; team <= 32; team <<= 1) {
        if (team == 1 && C < 3) continue;
        const int64_t most = std::min<int64_t>(fit, std::min(32 / team, team > 1 ? 16 : 32)), rounds = (per_sm + most - 1) / most;
        offer(team == 1 ? 4.3 + (double)rounds * (1.5 + (0.19 + 0.31 * C) * u) + (double)per_sm * (0.07 + 0.009 * C * u)
                        : 5.0 + (double)rounds * (1.0 + (0.15 + 0.28 * C) * u / team) + (double)per_sm * (0.09 + 0.054 * team + 0.012 * C * u),
              team, (per_sm + rounds - 1) / rounds);
    }
    best.grid = std::min(g->sm_count, B);
    return best;
}

// Plan of the block-per-sequence path with packed words (C <= 4).  Returns nullptr on success.
const char* plan_quad(const moc_graph* g, size_t smem_cap, bool profile, int mode, Plan* out) {
    Plan pl = *out;
    const int64_t n = g->n, C = g->C, t_max = C * n;
    if (C > 4) return "C > 4";
    if (!g->d_rec32 && !g->d_order) return "n above 32000 or a degree above 65535";
    if (t_max > 32766) return "sequences of more than 32766 steps";
    if (pl.wide && !g->split_ok) return "sum(m) too large for two-part sums";
    const QuadBytes z = quad_bytes(g, pl.wide, profile);
    const size_t sm = z.state() + (mode ? z.graph() : 0);
    if (sm > smem_cap) return "the state of a sequence exceeds shared memory";
    QuadFn fn = mode == moc::kQuadWarps ? quad_warp_fn(pl.wide, (int)C) : quad_fn(pl.wide, (int)C, g->d_rec32 != nullptr, mode == moc::kQuadTeams, profile);
    if (raise_smem_limit((const void*)fn, g->smem_optin) != cudaSuccess) { cudaGetLastError(); return "cudaFuncSetAttribute failed"; }
    const int forced = !profile && g->want_kind == MOC_KERNEL_BLOCK ? g->want_a : 0;
    bool any = mode != moc::kQuadBlock;
    for (int k = 0; k < 5 && mode == moc::kQuadBlock; ++k) {
        const int thr = forced ? forced : 64 << k;
        int nb = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, (const void*)fn, thr, sm) != cudaSuccess) { cudaGetLastError(); nb = 0; }
        pl.quad_nb[k] = nb;
        any = any || nb > 0;
    }
    if (!any) return "kernel does not fit on an SM";
    pl.quad = true;
    pl.quad_mode = mode;
    pl.quad_fn = fn;
    pl.quad_forced = forced;
    pl.gpc = 1;
    pl.smem = sm;
    pl.sm_count = g->sm_count;
    pl.grid = g->sm_count * std::max(1, pl.quad_nb[1]);
    pl.quad_word_b = (uint32_t)z.word;
    pl.quad_cnt_b = (uint32_t)z.cnt;
    pl.quad_delta_b = (uint32_t)z.delta;
    pl.rec_bytes = (uint32_t)z.rec;
    pl.w_bytes = (uint32_t)z.w;
    pl.sell_bytes = (uint32_t)z.sell;
    pl.quad_row_b = (uint32_t)z.row;
    pl.valid = true;
    *out = pl;
    return nullptr;
}

// Threads per sequence (64 << k) and blocks per SM of the block-per-sequence kernel proper.  With the blocks
// per SM that the state and the registers allow, a batch takes ceil(sequences per SM / blocks) rounds; as few
// blocks as that number of rounds needs keeps them even.  The line for the time (quad_block_cost) is a fit to 2175 timed shapes (n = 40 to 5000,
// C = 2, 3, 4, 32- and 64-bit sums, B = 1 to 8192, every thread count); the choice costs 0.5 % on the mean against the best of the five
// thread counts, 0.3 % or less in nine of ten, and 38 % at worst (n = 1500, C = 4, B = 148: 14.5 against 10.6 us).
void quad_threads(const Plan& pl, int64_t n, int32_t C, int32_t B, int* threads, int* blocks) {
    const int64_t per_sm = ((int64_t)B + pl.sm_count - 1) / pl.sm_count;
    double best = 0;
    *threads = 0;
    for (int k = 0; k < 5; ++k) {
        const int nb = pl.quad_nb[k];
        if (nb < 1) continue;
        const int64_t rounds = (per_sm + nb - 1) / nb;
        const double cost = quad_block_cost(n, C, per_sm, nb, 1 << k);
        if (*threads == 0 || cost < best) {
            best = cost;
            *threads = pl.quad_forced ? pl.quad_forced : 64 << k;
            *blocks = (int)((per_sm + rounds - 1) / rounds);
        }
    }
}

// Backward walk with a lane per sequence: n <= 128, C <= 4.  Used for the batches live_serves() names.
void plan_live(const moc_graph* g, Plan* pl) {
    pl->valid = true;
    const bool wide = g->sum_m > (int64_t)INT32_MAX / g->C || g->sum_w > (int64_t)INT32_MAX / g->C;
    pl->live_image = wide ? g->d_live64 : g->d_live32;
    LiveFn fn = live_fn(wide, live_words(g->n), g->C);
    if (raise_smem_limit((const void*)fn, g->smem_optin) != cudaSuccess) { cudaGetLastError(); return; }
    pl->live_fn = fn;
}

// Whether the warp-per-sequence kernel can serve the graph, as far as the host can tell.
bool warp_serves(const moc_graph* g) {
    const bool wide = g->sum_m > (int64_t)INT32_MAX / g->C;
    return g->C <= 2 && g->d_rec32 != nullptr && (!wide || g->split_ok) && (__int128)g->C * g->sum_w < ((__int128)1 << 48);
}

// Shared memory of the warp-per-sequence kernel: the graph once per block, the state of every sequence in flight.
void pair_bytes(const moc_graph* g, Plan* pl) {
    const size_t n = (size_t)g->n, msz = pl->wide ? 8 : 4, per_vec = 16 / msz;
    const size_t nvec_d = (g->C * n + 2 + per_vec - 1) / per_vec, v_max = ((nvec_d + 31) / 32) | 1;
    pl->rec_bytes = (uint32_t)((pl->wide ? 16 : 8) * 64 * (size_t)g->n_tiles);
    pl->w_bytes = (uint32_t)(8 * 64 * (size_t)g->n_tiles);
    pl->sell_bytes = (uint32_t)align16(4 * (size_t)g->sell_len);
    pl->word_bytes = (uint32_t)align16(4 * (n + 2));
    pl->delta_bytes = (uint32_t)(moc::kPairDeltaFront + 32 * v_max * 16);
    pl->pair_graph_b = (size_t)pl->rec_bytes + pl->w_bytes + pl->sell_bytes;
    pl->pair_warp_b = (size_t)pl->word_bytes + moc::kPairWordTail + pl->delta_bytes;
}

// Warps that share a sequence in the warp-per-sequence kernel, for batches that leave most of an SM's warps without
// a sequence of their own (1: none do), and the shape of the launch: one block per SM, up to 16 warps.  Sharing divides the
// latency of a sequence and costs barriers; with more than eight sequences on an SM the warps have enough to do (n = 1000, 12 per SM:
// 15.7 us without, 14.6 with two; n = 250, 64-bit sums 9.0 and 10.4).  Measured with 1 / 2 / 4 / 8 warps on a sequence (us; 32-bit sums): n = 153, B = 296
// 7.2 (before) / 6.1 / 6.0; n = 353, B = 592 8.3 / 6.4 / 6.4; n = 600, B = 148 10.4 / 8.3 / 6.3 / 6.0; n = 1000, B = 592 12.5 / 10.4 / 8.4; B = 1184 14.5 / 12.4;
// with 8 / 16: n = 1000, B = 148 6.2 / 6.2, n = 1400 6.9 / 6.6, n = 5000 12.0 / 10.4.  The block-per-sequence kernel's teams are nowhere faster at
// one sequence per SM (block / team, 56 batches, n = 400 to 598): n = 442, B = 1 5.9 / 5.9, B = 148 6.2 / 6.2; 64-bit sums n = 560, B = 148 8.2 / 7.2.
struct TeamShape {
    int team = 1, groups = 0, grid = 0;
};
TeamShape team_shape(const moc_graph* g, int32_t B) {
    TeamShape s;
    if (!warp_serves(g) || g->want_gpc || g->want_G || (g->want_kind != MOC_KERNEL_AUTO && g->want_kind != MOC_KERNEL_WARP)) return s;
    Plan pl;
    pl.wide = g->sum_m > (int64_t)INT32_MAX / g->C;
    pair_bytes(g, &pl);
    const int64_t per_sm = ((int64_t)B + g->sm_count - 1) / g->sm_count;
    for (int team = 16; team > 1; team >>= 1) {
        if (per_sm * team > 16 || team > g->n_tiles || g->n < (team == 16 ? 1400 : team == 8 ? 600 : 0)) continue;
        if (pl.pair_graph_b + per_sm * pl.pair_warp_b + 2048 > g->smem_optin) return s;
        s.team = team;
        s.groups = (int)per_sm;
        s.grid = std::min(B, g->sm_count);
        return s;
    }
    return s;
}

// Chooses kernel variant, group size and grid for the handle's current n and C.  The dynamic
// shared-memory limit of a kernel is a property of the kernel, not of the handle: it is always
// raised to the device maximum, so that handles with different needs can share one kernel.
int make_plan(const moc_graph* g, bool profile, Plan* out) {
    Plan pl;
    const int64_t n = g->n, C = g->C;
    pl.CP = C <= 2 ? 2 : (C <= 4 ? 4 : 8);
    pl.wide = g->sum_m > (int64_t)INT32_MAX / C;  // C*sum(m) bounds every partial sum of deltas
    const int64_t t_max = C * n;
    const size_t mem_sz = pl.wide ? 8 : 4;
    const size_t sh_cnt = align16(4 * n), sh_occ = align16(2 * n * pl.CP),
                 sh_delta = align16((t_max + 1) * mem_sz);
    const size_t sh_group = sh_cnt + sh_occ + sh_delta + align16(moc::kRedBytes);
    const size_t smem_cap = g->smem_optin > 1024 ? g->smem_optin - 1024 : 0;  // 1 KB per block is reserved
    const int kind = profile ? MOC_KERNEL_GROUP : g->want_kind;
    const bool shape_given = g->want_G != 0 || g->want_gpc != 0;       // moc_graph_set_launch
    if (profile && !plan_quad(g, smem_cap, true, quad_shape(g, 1, true).team ? moc::kQuadTeams : moc::kQuadBlock, &pl)) {
        *out = pl;
        return MOC_OK;
    }
    // Order of preference when nothing is forced: warp per sequence, then sequence per lane (it also
    // serves graphs whose degrees are too uneven for the warp kernel's padded successor tiles), then
    // the thread-group kernel, which serves everything.
    const bool warp_ok = warp_serves(g);
    if (kind == MOC_KERNEL_LANE || (kind == MOC_KERNEL_AUTO && !shape_given && !warp_ok)) {
        const char* why = plan_lane(g, smem_cap, &pl);
        if (!why) {
            *out = pl;
            return MOC_OK;
        }
        if (kind == MOC_KERNEL_LANE) return fail(MOC_ERR_ARG, "the sequence-per-lane kernel cannot serve this graph: %s", why);
    }
    if (kind == MOC_KERNEL_BLOCK || (kind == MOC_KERNEL_AUTO && !shape_given && !profile && C >= 3)) {
        const char* why = plan_quad(g, smem_cap, profile, moc::kQuadBlock, &pl);
        if (!why) {
            *out = pl;
            return MOC_OK;
        }
        if (kind == MOC_KERNEL_BLOCK) return fail(MOC_ERR_ARG, "the block-per-sequence kernel cannot serve this graph: %s", why);
    }
    if (kind == MOC_KERNEL_WARP && !warp_ok)
        return fail(MOC_ERR_ARG, "the warp-per-sequence kernel cannot serve this graph (C > 2, degrees too uneven, C * sum(w) >= 2^48 or sum(m) too large)");
    if (!profile && g->want_G == 0 && kind != MOC_KERNEL_GROUP && warp_ok) {
        // warp-per-sequence fast path
        pair_bytes(g, &pl);
        const size_t graph_b = pl.pair_graph_b, warp_b = pl.pair_warp_b;
        // vectors of the next row fetched ahead per lane: enough for a typical row of about 1.3 n steps
        const int pre = n < 256 ? 0 : (int)std::min<int64_t>(5, (n * 13 / 10 + 96) / 128);
        PairFn fn = pair_fn(pl.wide, pre);
        int best_wpb = 0, best_warps = 0, best_nb = 0;
        cudaError_t e = raise_smem_limit((const void*)fn, g->smem_optin);
        if (e != cudaSuccess) return fail(MOC_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
        for (int wpb = moc::pair_max_warps(pre, false); wpb >= 4; --wpb) {    // every variant is compiled for two blocks of so many on an SM
            if (g->want_gpc && wpb != std::min(g->want_gpc, 16)) continue;
            const size_t sm = graph_b + wpb * warp_b;
            if (sm > smem_cap) continue;
            int nb = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, (const void*)fn, wpb * 32, sm) != cudaSuccess) { cudaGetLastError(); continue; }
            if (pre == 0) nb = std::min(nb, 2);          // more and smaller blocks only stage the graph more often
            pl.pair_nb[wpb] = nb;
            if (nb * wpb > best_warps) { best_warps = nb * wpb; best_wpb = wpb; best_nb = nb; }
        }
        pl.sm_count = g->sm_count;
        if (best_warps >= 10) {
            pl.pair = true;
            pl.pair_fn = fn;
            pl.G = 32;
            pl.gpc = best_wpb;
            pl.block = 32 * best_wpb;
            pl.smem = graph_b + best_wpb * warp_b;
            pl.grid = g->sm_count * best_nb;
            pl.valid = true;
            *out = pl;
            return MOC_OK;
        }
    }
    // Sequences too long for ten warps of the warp-per-sequence kernel on an SM: warp / block with 16 warps 18.6 / 24.7 us (n = 1000, 32-bit
    // sums, B = 2368), with 14 37.0 / 39.1 (700, 64 bits, 4736), with 11 45.1 / 51.2 (1432, 32 bits, 3919), with 9 43.8 / 42.4 (1000, 64 bits,
    // 3552), with 6 61.8 / 30.9 (1400, 64 bits, 1776)
    if (kind == MOC_KERNEL_AUTO && !shape_given && !profile && C <= 2 && !plan_quad(g, smem_cap, profile, moc::kQuadBlock, &pl)) {
        *out = pl;
        return MOC_OK;
    }
    if (t_max <= 65534 && sh_group <= smem_cap) {
        pl.global_state = false;
        pl.cnt_bytes = (uint32_t)sh_cnt;
        pl.occ_bytes = (uint32_t)sh_occ;
        pl.delta_bytes = (uint32_t)sh_delta;
        pl.group_bytes = (uint32_t)sh_group;
        int G = 1024, gpc = 1;
        if (!profile) {
            const int per_sm = (int)std::max<size_t>(1, g->smem_optin / sh_group);  // groups resident per SM
            G = g->want_G ? g->want_G : std::min(1024, std::max(32, pow2_ceil(32 * 48 / std::min(per_sm, 48))));
            gpc = g->want_gpc ? g->want_gpc : std::max(1, 256 / G);
            gpc = std::min(gpc, G == 32 ? 32 : 15);          // named barriers 1..15
            gpc = std::min(gpc, 1024 / G);
            while (gpc > 1 && (size_t)gpc * sh_group > smem_cap) --gpc;
        }
        pl.G = G;
        pl.gpc = gpc;
        pl.block = G * gpc;
        pl.smem = (size_t)gpc * sh_group;
        pl.fn = shared_fn(pl.wide, G, pl.CP, profile);
        if (!pl.fn) return fail(MOC_ERR_ARG, "unsupported launch shape");
        cudaError_t e = raise_smem_limit((const void*)pl.fn, g->smem_optin);
        if (e != cudaSuccess) return fail(MOC_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
        int nb = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, (const void*)pl.fn, pl.block, pl.smem);
        if (e != cudaSuccess) return fail(MOC_ERR_CUDA, "occupancy query: %s", cudaGetErrorString(e));
        if (nb < 1) return fail(MOC_ERR_CUDA, "kernel does not fit on an SM (block %d, smem %zu)", pl.block, pl.smem);
        pl.grid = profile ? 1 : g->sm_count * nb;
    } else {
        // state in global memory: int32 positions, int64 sums
        pl.global_state = true;
        pl.wide = true;
        pl.cnt_bytes = (uint32_t)align16(4 * n);
        const size_t occ = align16(4 * n * pl.CP), del = align16((t_max + 1) * 8);
        const size_t grp = pl.cnt_bytes + occ + del + align16(moc::kRedBytes);
        if (grp > 0xFFFFFFFFull) return fail(MOC_ERR_ARG, "graph too large: per-sequence state of %zu bytes", grp);
        pl.occ_bytes = (uint32_t)occ;
        pl.delta_bytes = (uint32_t)del;
        pl.group_bytes = (uint32_t)grp;
        pl.G = 1024;
        pl.gpc = 1;
        pl.block = 1024;
        pl.smem = 0;
        pl.fn = global_fn(pl.CP, profile);
        int nb = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, (const void*)pl.fn, pl.block, 0);
        if (e != cudaSuccess) return fail(MOC_ERR_CUDA, "occupancy query: %s", cudaGetErrorString(e));
        if (nb < 1) nb = 1;
        pl.grid = profile ? 1 : g->sm_count * nb;
    }
    pl.valid = true;
    *out = pl;
    return MOC_OK;
}

int ensure(void** ptr, size_t* cap, size_t need) {
    if (need <= *cap) return MOC_OK;
    if (*ptr) {
        MOC_CUDA(cudaFree(*ptr));
        *ptr = nullptr;
        *cap = 0;
    }
    size_t want = std::max(need, *cap * 2);
    MOC_CUDA(cudaMalloc(ptr, want));
    *cap = want;
    return MOC_OK;
}


// The arrays of a handle, gathered for one allocation and, unless they are large, one copy, so that a further table
// costs a new handle its bytes and no calls.  Creating a handle of n = 20, 100, 442, 1000: 540, 600, 690 and 900 us
// with an allocation and a copy per array (23 of them at n = 442), 390, 395, 540 and 745 so; freeing it 340 and 275.
class Tables {
  public:
    // A device array for *dst, filled from `src` (alive until upload) or, without one, not at all.
    template <typename T>
    void add(T** dst, const void* src, size_t bytes) {
        parts_.push_back({(void**)dst, src, size_, bytes});
        size_ += (std::max<size_t>(bytes, 16) + 255) & ~size_t(255);
    }
    template <typename T, typename V>
    void add(T** dst, std::vector<V>&& v) {
        auto kept = std::make_shared<std::vector<V>>(std::move(v));
        keep_.push_back(kept);
        add(dst, kept->data(), kept->size() * sizeof(V));
    }
    cudaError_t upload(char** block) {
        cudaError_t e = cudaMalloc((void**)block, size_);
        if (e != cudaSuccess) return e;
        for (const Part& p : parts_) *p.dst = *block + p.at;
        if (size_ <= kTogether) {
            std::vector<char> all(size_);
            for (const Part& p : parts_)
                if (p.src) memcpy(all.data() + p.at, p.src, p.bytes);
            return cudaMemcpy(*block, all.data(), size_, cudaMemcpyHostToDevice);
        }
        for (const Part& p : parts_)
            if (p.src && p.bytes && e == cudaSuccess) e = cudaMemcpy(*p.dst, p.src, p.bytes, cudaMemcpyHostToDevice);
        return e;
    }

  private:
    static constexpr size_t kTogether = 1 << 20;       // up to here a second copy on the host costs less than the calls
    struct Part {
        void** dst;
        const void* src;
        size_t at, bytes;
    };
    std::vector<Part> parts_;
    std::vector<std::shared_ptr<void>> keep_;
    size_t size_ = 0;
};

// Words 4-5 of the node records of the sequence-per-lane layouts: w | 1 << 40 (counts the node when
// it has two copies) | 1 << 52 when the node's cap C_v is 1.
void set_lane_caps(moc_graph* g) {
    for (int li = 0; li < 3; ++li) {
        LaneLayout& L = g->lane[li];
        for (size_t r = 0; r < L.h_node.size(); ++r) {
            const int32_t v = L.h_node[r];
            uint64_t x = 0;
            if (v >= 0) {
                x = (uint64_t)g->h_w[v] | (uint64_t(1) << moc::kLaneCntShift);
                if (!g->h_cap.empty() && g->h_cap[v] == 1) x |= uint64_t(1) << moc::kLaneCapShift;
            }
            L.h_rec32[8 * r + 4] = L.h_rec64[8 * r + 4] = (uint32_t)(x & 0xFFFFFFFFu);
            L.h_rec32[8 * r + 5] = L.h_rec64[8 * r + 5] = (uint32_t)(x >> 32);
        }
    }
}

// Durations by slot of the warp-per-sequence layout: w | 1 << 48 (counts the node when it has two copies) | 1 << 63
// for nodes whose cap C_v is 1.
std::vector<uint64_t> slot_durations(const moc_graph* g) {
    std::vector<uint64_t> wslot(g->h_slot.size());
    for (size_t r = 0; r < wslot.size(); ++r) {
        const int32_t v = g->h_slot[r];
        uint64_t x = 0;
        if (v >= 0) {
            x = (uint64_t)g->h_w[v] | (uint64_t(1) << moc::kPairCntShift);
            if (!g->h_cap.empty() && g->h_cap[v] == 1) x |= uint64_t(1) << 63;
        }
        wslot[r] = x;
    }
    return wslot;
}

// Layouts for the sequence-per-lane kernel, one per group size g = 32, 16, 8 (S = 1, 2, 4 sub-lanes).
// Nodes in order of falling out-degree (a sink counts one: its made-up successor), S consecutive
// nodes form a bundle and share a row count; entry (k, h) of a bundle is the byte offset of the
// word row of the k-th successor of its h-th node, the node's own row once its list is used up.
void build_lane_layouts(moc_graph* g, const std::vector<int32_t>& succ_start, const std::vector<int32_t>& succ,
                        const int64_t* m, const std::vector<int32_t>& m32, Tables* tables) {
    const int32_t n = g->n;
    if (n >= 4096) return;                              // the count of two-copy nodes has 12 bits
    auto deg = [&](int32_t v) { return std::max(1, succ_start[v + 1] - succ_start[v]); };
    std::vector<int32_t> order((size_t)n);
    for (int32_t v = 0; v < n; ++v) order[v] = v;
    std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) { return deg(x) > deg(y); });
    if (deg(order[0]) > 255) return;
    for (int li = 0; li < 3; ++li) {
        const int lg = 5 - li, gsz = 1 << lg, S = 32 >> lg;
        LaneLayout& L = g->lane[li];
        const int32_t nb = (n + S - 1) / S;
        std::vector<int32_t> node((size_t)nb * S, -1);
        for (int32_t i = 0; i < n; ++i) node[i] = order[i];
        std::vector<uint32_t> rec32(node.size() * 8, 0u), rec64(node.size() * 8, 0u);
        std::vector<uint32_t> se;
        const uint32_t row_b = moc::lane_word_row(gsz);
        const uint32_t t_row = 0u - moc::lane_special(gsz), one_row = t_row + row_b;   // relative to the first node row
        for (int32_t bd = 0; bd < nb; ++bd) {
            int rows = 0;
            for (int h = 0; h < S; ++h)
                if (node[(size_t)bd * S + h] >= 0) rows = std::max(rows, deg(node[(size_t)bd * S + h]));
            const uint32_t first = (uint32_t)se.size();
            for (int k = 0; k < rows; ++k)
                for (int h = 0; h < S; ++h) {
                    const int32_t v = node[(size_t)bd * S + h];
                    uint32_t off;
                    if (v < 0) off = one_row;
                    else if (k < succ_start[v + 1] - succ_start[v]) off = (uint32_t)succ[succ_start[v] + k] * row_b;
                    else if (k == 0) off = t_row;                    // a sink: the word that holds T
                    else off = (uint32_t)v * row_b;
                    se.push_back(off);
                }
            for (int h = 0; h < S; ++h) {
                const size_t r = (size_t)bd * S + h;
                const int32_t v = node[r];
                const uint64_t mv = v >= 0 ? (uint64_t)m[v] : 0;
                rec32[8 * r + 0] = rec64[8 * r + 0] = v >= 0 ? (uint32_t)v * row_b : one_row;
                rec32[8 * r + 1] = rec64[8 * r + 1] = (4u * (first + (uint32_t)h)) | ((uint32_t)rows << 24);
                rec32[8 * r + 2] = v >= 0 ? (uint32_t)m32[v] : 0u;
                rec32[8 * r + 3] = 0u - rec32[8 * r + 2];
                rec64[8 * r + 2] = (uint32_t)(mv & 0xFFFFFFFFu);
                rec64[8 * r + 3] = (uint32_t)(mv >> 32);
                rec64[8 * r + 6] = (uint32_t)((0 - mv) & 0xFFFFFFFFu);
                rec64[8 * r + 7] = (uint32_t)((0 - mv) >> 32);
            }
        }
        while (se.size() % 4) se.push_back(one_row);
        if (se.empty()) se.assign(4, one_row);
        if (se.size() * 4 + 64 >= (size_t(1) << 24)) continue;
        L.n_bundles = nb;
        L.succ_len = (int64_t)se.size();
        L.h_node = std::move(node);
        L.h_rec32 = std::move(rec32);
        L.h_rec64 = std::move(rec64);
        L.ok = true;
        tables->add(&L.d_rec32, L.h_rec32.data(), L.h_rec32.size() * 4);       // the handle's copies: complete before they are sent
        tables->add(&L.d_rec64, L.h_rec64.data(), L.h_rec64.size() * 4);
        tables->add(&L.d_succ, std::move(se));
    }
    set_lane_caps(g);
}

// Layout for the block-per-sequence kernel on graphs without successor tiles: the nodes in order of falling
// out-degree (a sink counts one: its made-up successor n + 1) with the place of their successor lists, and the
// lists as 16-bit ids.
void build_quad_layout(moc_graph* g, const std::vector<int32_t>& succ_start, const std::vector<int32_t>& succ, Tables* tables) {
    const int32_t n = g->n;
    if (g->n_tiles || n > 32000) return;
    auto deg = [&](int32_t v) { return std::max(1, succ_start[v + 1] - succ_start[v]); };
    std::vector<int32_t> order((size_t)n);
    for (int32_t v = 0; v < n; ++v) order[v] = v;
    std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) { return deg(x) > deg(y); });
    if (deg(order[0]) > 65535) return;
    std::vector<uint32_t> rec((size_t)n * 8, 0u);
    std::vector<uint16_t> rest;
    for (int32_t i = 0; i < n; ++i) {
        const int32_t v = order[i];
        std::vector<uint16_t> ids;
        if (succ_start[v + 1] == succ_start[v]) ids.push_back((uint16_t)(n + 1));
        for (int32_t e = succ_start[v]; e < succ_start[v + 1]; ++e) ids.push_back((uint16_t)succ[e]);
        uint32_t* r = &rec[(size_t)i * 8];
        r[0] = (uint32_t)v | ((uint32_t)ids.size() << 16);
        r[1] = (uint32_t)rest.size();
        for (size_t k = 0; k < ids.size(); ++k) {
            if (k < 8) r[4 + k / 2] |= (uint32_t)ids[k] << (16 * (k & 1));
            else rest.push_back(ids[k]);
        }
    }
    tables->add(&g->d_order, std::move(rec));
    tables->add(&g->d_succ16, std::move(rest));
}

// The arrays that the kernels read of a graph: `keys` are its edges (u << 32 | v) in order, grouped by u in succ_start and succ;
// m32 is m cut to 32 bits.  What is not moved into `tables` outlives the upload.
void build_tables(moc_graph* g, const std::vector<uint64_t>& keys, const std::vector<int32_t>& succ_start, const std::vector<int32_t>& succ,
                  const int64_t* w, const int64_t* m, const std::vector<int32_t>& m32, Tables* tables) {
    const int32_t n = g->n;
    const int64_t ne = g->n_edges;
    tables->add(&g->d_succ_start, succ_start.data(), ((size_t)n + 1) * 4);
    tables->add(&g->d_succ, succ.data(), (size_t)ne * 4);
    {
        // predecessor lists (grouped by consumer) and the total output size of the sinks
        std::vector<int32_t> pred_start((size_t)n + 1, 0), pred((size_t)ne);
        for (int64_t k = 0; k < ne; ++k) pred_start[(keys[k] & 0xFFFFFFFFu) + 1]++;
        for (int32_t v = 0; v < n; ++v) g->max_indeg = std::max(g->max_indeg, pred_start[v + 1]);
        for (int32_t v = 0; v < n; ++v) pred_start[v + 1] += pred_start[v];
        std::vector<int32_t> fill(pred_start.begin(), pred_start.end() - 1);
        for (int64_t k = 0; k < ne; ++k) pred[fill[keys[k] & 0xFFFFFFFFu]++] = (int32_t)(keys[k] >> 32);
        for (int32_t v = 0; v < n; ++v)
            if (succ_start[v + 1] == succ_start[v]) g->sink_m += m[v];
        // (for the search; 1 to 2 % of creating a handle: n = 442 490 us, n = 5000 1790 -> 1815)
        if (ne <= 65535 && g->sum_w < ((int64_t)1 << 31) && g->n <= 16000) {
            const size_t list = ((size_t)ne + 3) & ~size_t(3);
            std::vector<uint32_t> near((2 * ((size_t)n + 1) + list + (size_t)n + 3) & ~size_t(3), 0u);
            uint16_t* lists = reinterpret_cast<uint16_t*>(near.data() + 2 * ((size_t)n + 1));
            for (int32_t v = 0; v <= n; ++v) {
                near[2 * (size_t)v] = (uint32_t)succ_start[v] | (uint32_t)pred_start[v] << 16;
                near[2 * (size_t)v + 1] = v < n ? (uint32_t)w[v] : 0u;
            }
            for (int64_t k = 0; k < ne; ++k) {
                lists[k] = (uint16_t)succ[k];
                lists[list + k] = (uint16_t)pred[k];
            }
            for (int32_t v = 0; v < n; ++v) near[2 * ((size_t)n + 1) + list + (size_t)v] = (uint32_t)m32[v];
            g->near_bytes = (4 * (2 * ((size_t)n + 1) + list) + 15) & ~size_t(15);
            g->near_size_bytes = near.size() * 4;
            tables->add(&g->d_near, std::move(near));
        }
        tables->add(&g->d_pred_start, std::move(pred_start));
        tables->add(&g->d_pred, std::move(pred));
    }
    if (n <= moc::kLiveMaxN) {
        // The nodes are dealt to the mask words so that the predecessors of a node lie in different words where
        // possible (moc_live_kernel.cuh): each node, most consumers first, goes to the word with the fewest other
        // predecessors of its consumers.
        const int words = live_words(n);
        std::vector<uint32_t> preds((size_t)n * words, 0u);
        std::vector<int32_t> order((size_t)n), clash((size_t)n * words, 0), fill((size_t)words, 0);
        for (int32_t v = 0; v < n; ++v) order[v] = v;
        std::stable_sort(order.begin(), order.end(),
                         [&](int32_t x, int32_t y) { return succ_start[x + 1] - succ_start[x] > succ_start[y + 1] - succ_start[y]; });
        g->h_live_place.assign((size_t)n, 0);
        for (int32_t u : order) {
            int best = -1, best_clash = 0;
            for (int k = 0; k < words; ++k) {
                int c = 0;
                for (int32_t e = succ_start[u]; e < succ_start[u + 1]; ++e) c += clash[(size_t)succ[e] * words + k];
                c += clash[(size_t)u * words + k];          // the node counts among its predecessors
                if (fill[k] < 32 && (best < 0 || c < best_clash || (c == best_clash && fill[k] < fill[best]))) { best = k; best_clash = c; }
            }
            for (int32_t e = succ_start[u]; e < succ_start[u + 1]; ++e) {
                ++clash[(size_t)succ[e] * words + best];
                preds[(size_t)succ[e] * words + best] |= 1u << fill[best];
            }
            ++clash[(size_t)u * words + best];
            if (succ_start[u + 1] == succ_start[u]) g->live_sinks[best] |= 1u << fill[best];
            g->h_live_place[u] = best << 5 | fill[best]++;
        }
        // tables for both widths, or the one that every C <= MOC_MAX_COPIES selects
        const bool narrow = g->sum_m <= INT32_MAX / MOC_MAX_COPIES && g->sum_w <= INT32_MAX / MOC_MAX_COPIES;
        for (int wide = 0; wide < (narrow ? 1 : 2); ++wide)
            tables->add(wide ? &g->d_live64 : &g->d_live32, moc::live_image(n, words, wide != 0, g->h_live_place, preds, m, w));
    }
    tables->add(&g->d_w, w, (size_t)n * 8);
    tables->add(&g->d_m64, m, (size_t)n * 8);
    tables->add(&g->d_m32, m32.data(), (size_t)n * 4);
    {
        // 64-bit sums: parts of m that 32-bit atomics can add (moc_pair_kernel.cuh), where sum(m) permits; with room for
        // two amounts per node at a time (the interval checker adds up intervals that may overlap)
        int k = 30;
        while (k > 0 && ((int64_t)1 << (30 - k)) < n) --k;
        g->split_ok = (g->sum_m >> k) < ((int64_t)1 << 30);
        g->split = g->split_ok ? k : 32;
    }
    if (n <= 16000) {
        // Layout for the warp-per-sequence kernel.  Lane l serves the nodes with id = l (mod 32);
        // each residue class is sorted by out-degree (descending, ties by id); half j holds the
        // j-th node of every class, a tile is two halves.  A tile stores, row by row, the word
        // offsets (4 * id) of its nodes' successors, two halves packed per 32-bit entry, padded with
        // the offset of a dummy word (4 * n).  Within a half the order of each node's successors
        // is chosen greedily so that the 32 words a row touches fall in different banks where
        // possible.  Skipped when padding would more than double the storage (a few very high
        // degrees): such graphs use the general kernel.
        auto deg = [&](int32_t v) { return succ_start[v + 1] - succ_start[v]; };
        const int32_t n_halves = 2 * ((n + 63) / 64), n_tiles = n_halves / 2;
        std::vector<int32_t> slot((size_t)n_halves * 32, -1);  // node at (half, lane) or -1
        for (int32_t l = 0; l < 32; ++l) {
            std::vector<int32_t> cls;
            for (int32_t v = l; v < n; v += 32) cls.push_back(v);
            std::stable_sort(cls.begin(), cls.end(), [&](int32_t x, int32_t y) { return deg(x) > deg(y); });
            for (size_t j = 0; j < cls.size(); ++j) slot[j * 32 + l] = cls[j];
        }
        std::vector<int32_t> rows((size_t)n_tiles, 0);
        int64_t sell_len = 0;
        for (int32_t d = 0; d < n_tiles; ++d) {
            for (int32_t s = 0; s < 64; ++s)
                if (slot[(size_t)d * 64 + s] >= 0)
                    rows[d] = std::max(rows[d], std::max(1, deg(slot[(size_t)d * 64 + s])));  // a sink gets one entry
            sell_len += 32 * (int64_t)rows[d];
        }
        int32_t max_rows = 0;
        for (int32_t d = 0; d < n_tiles; ++d) max_rows = std::max(max_rows, rows[d]);
        if (sell_len <= 2 * ne + 4096 && sell_len < (1 << 20) && max_rows < (1 << 12) && 4 * ((int64_t)n + 3) < 65536) {
            const uint32_t word_b = (uint32_t)align16(4 * ((size_t)n + 2));   // the constant word (1, 1) sits right after the words
            std::vector<uint32_t> rec32((size_t)n_halves * 32 * 2), rec64((size_t)n_halves * 32 * 4, 0u);
            // entry (row k, lane l) of a tile: word of the k-th successor of the node in half 0 | same for half 1 << 16;
            // a list that is used up continues with the node's own word
            std::vector<uint32_t> sell((size_t)std::max<int64_t>(sell_len, 1), word_b | (word_b << 16));
            auto own_word = [&](int32_t v) { return v >= 0 ? 4u * (uint32_t)v : word_b; };
            std::vector<int32_t> tile_row((size_t)n_tiles, 0);
            for (int32_t d = 1; d < n_tiles; ++d) tile_row[d] = tile_row[d - 1] + rows[d - 1];
            for (size_t r = 0; r < slot.size(); ++r) {
                const int32_t v = slot[r];
                const uint32_t x = own_word(v) | ((uint32_t)((r & 32) ? tile_row[r / 64] : rows[r / 64]) << 16);
                const uint64_t mv = v >= 0 ? (uint64_t)m[v] : 0;
                rec32[2 * r + 0] = x;
                rec32[2 * r + 1] = v >= 0 ? (uint32_t)m32[v] : 0u;
                rec64[4 * r + 0] = x;
                rec64[4 * r + 2] = (uint32_t)(mv & 0xFFFFFFFFu);
                rec64[4 * r + 3] = (uint32_t)(mv >> g->split);
            }
            uint32_t pos = 0;
            std::vector<std::vector<int32_t>> rem(32);
            for (int32_t d = 0; d < n_tiles; ++d) {
                for (int32_t h = 0; h < 2; ++h) {
                    std::vector<int32_t> lanes;
                    for (int32_t l = 0; l < 32; ++l) {
                        const int32_t v = slot[((size_t)2 * d + h) * 32 + l];
                        rem[l].clear();
                        if (v >= 0) rem[l].assign(succ.begin() + succ_start[v], succ.begin() + succ_start[v + 1]);
                        if (v >= 0 && rem[l].empty()) rem[l].push_back(n + 1);  // sink: the word that holds T
                        lanes.push_back(l);
                        for (int32_t k = 0; k < rows[d]; ++k) {
                            uint32_t& e = sell[(size_t)pos + 32 * (size_t)k + l];
                            e = h == 0 ? ((e & 0xFFFF0000u) | own_word(v)) : ((e & 0x0000FFFFu) | (own_word(v) << 16));
                        }
                    }
                    for (int32_t k = 0; k < rows[d]; ++k) {
                        int used[32] = {0};
                        for (int32_t l = 0; l < 32; ++l)
                            if (rem[l].empty()) used[l]++;   // reads its own word, which lies in bank l
                        std::stable_sort(lanes.begin(), lanes.end(),
                                         [&](int32_t x, int32_t y) { return rem[x].size() > rem[y].size(); });
                        for (int32_t l : lanes) {
                            if (rem[l].empty()) continue;  // stays the own word
                            const bool forced = (int32_t)rem[l].size() >= rows[d] - k;
                            int pick = -1;
                            for (size_t c = 0; c < rem[l].size(); ++c)
                                if (!used[rem[l][c] & 31]) { pick = (int)c; break; }
                            if (pick < 0 && !forced) continue;  // wait for a row where its bank is free
                            if (pick < 0) pick = 0;
                            used[rem[l][pick] & 31]++;
                            uint32_t& e = sell[(size_t)pos + 32 * (size_t)k + l];
                            const uint32_t off = 4u * (uint32_t)rem[l][pick];
                            e = h == 0 ? ((e & 0xFFFF0000u) | off) : ((e & 0x0000FFFFu) | (off << 16));
                            rem[l].erase(rem[l].begin() + pick);
                        }
                    }
                }
                pos += 32 * (uint32_t)rows[d];
            }
            // the same tiles for the interval checker: its padding repeats a successor, a sink reads its own word
            std::vector<uint32_t> sell_iv(sell);
            for (size_t r = 0; r < slot.size(); ++r) {
                const int32_t v = slot[r];
                const uint32_t own = own_word(v), pad = v >= 0 && deg(v) > 0 ? 4u * (uint32_t)succ[succ_start[v]] : own;
                const int sh = (r & 32) ? 16 : 0;
                for (int32_t k = 0; k < rows[r / 64]; ++k) {
                    uint32_t& e = sell_iv[32 * (size_t)(tile_row[r / 64] + k) + (r & 31)];
                    const uint32_t off = e >> sh & 0xFFFFu;
                    if (off == own || off == 4u * ((uint32_t)n + 1)) e = (e & ~(0xFFFFu << sh)) | pad << sh;
                }
            }
            tables->add(&g->d_sell_iv, std::move(sell_iv));
            tables->add(&g->d_tile_row, std::move(tile_row));
            g->sell_len = (int32_t)sell_len;
            g->h_slot = std::move(slot);
            g->n_tiles = n_tiles;
            tables->add(&g->d_rec32, std::move(rec32));
            tables->add(&g->d_rec64, std::move(rec64));
            tables->add(&g->d_wslot, slot_durations(g));
            tables->add(&g->d_sell, std::move(sell));
        }
    }
    build_lane_layouts(g, succ_start, succ, m, m32, tables);
    build_quad_layout(g, succ_start, succ, tables);
}

moc::EvalParams base_params(const moc_graph* g, const Plan& pl) {
    moc::EvalParams p{};
    p.g.n = g->n;
    p.g.C = g->C;
    p.g.succ_start = g->d_succ_start;
    p.g.succ = g->d_succ;
    p.g.w = g->d_w;
    p.g.m = pl.wide ? (const void*)g->d_m64 : (const void*)g->d_m32;
    p.g.cap = g->d_cap;
    p.cnt_bytes = pl.cnt_bytes;
    p.occ_bytes = pl.occ_bytes;
    p.delta_bytes = pl.delta_bytes;
    p.group_bytes = pl.group_bytes;
    return p;
}

moc::QuadParams quad_params(const moc_graph* g, const Plan& pl) {
    moc::QuadParams q{};
    q.n = g->n;
    q.C = g->C;
    q.max_T = g->C * g->n;
    q.n_tiles = g->n_tiles;
    q.split = g->split;
    q.rec = pl.wide ? g->d_rec64 : g->d_rec32;
    q.sell = g->d_sell;
    q.tile_row = g->d_tile_row;
    q.order = g->d_order;
    q.succ = g->d_succ16;
    q.base_dur = g->sum_w;
    q.m = pl.wide ? (const void*)g->d_m64 : (const void*)g->d_m32;
    q.w = g->d_w;
    q.cap = g->d_cap;
    q.word_bytes = pl.quad_word_b;
    q.cnt_bytes = pl.quad_cnt_b;
    q.delta_bytes = pl.quad_delta_b;
    q.wslot = (const uint64_t*)g->d_wslot;
    q.rec_bytes = pl.rec_bytes;
    q.w_bytes = pl.w_bytes;
    q.sell_bytes = pl.sell_bytes;
    q.row_bytes = pl.quad_row_b;
    q.small_w = (__int128)g->C * g->sum_w < ((int64_t)1 << 32) ? 1 : 0;
    return q;
}

// Batches the backward walk serves.  Its time is a sequence's latency until every SM has 16 warps (about 6 us + 0.17 us
// per node), the other kernels' grows with the batch: the warp-per-sequence kernel (C <= 2) by the successor tiles of
// 64 nodes that a sequence has, more with 64-bit sums, the block-per-sequence kernel (C >= 3) by the nodes.  Crossings
// measured on layered and training graphs, sequences (C = 2 | C = 2, 64-bit sums | C = 3, 4):
//     n =  20: 5000 | 4000 | 2300       n =  64: 12000 | 10500 | 4800       n = 100: 17000 | 12500 | 8000
//     n =  40: 9500 | 6000 | 3200       n =  65: 11500 |  7500 | 5500       n = 128: 24000 | 16000 | 8800
// Over batches of 700 to 26000 and n = 12 to 128 the lines below cost 0.1 to 0.3 % on the mean against always taking
// the faster kernel, next to a crossing at most a fifth.
bool live_serves(const moc_graph* g, int32_t B) {
    if (!g->d_live32 || g->C > moc::kLivePlanes || g->want_kind != MOC_KERNEL_AUTO || g->want_G || g->want_gpc) return false;
    const bool wide = g->sum_m > (int64_t)INT32_MAX / g->C;
    const int32_t n = g->n;
    if (g->C > 2) return B >= 900 + 76 * n;
    if (wide) return B >= (n <= 64 ? 300 + 160 * n : 120 * n);
    return B >= (n <= 64 ? 1500 + 170 * n : 185 * n - 800);
}

int enqueue_live(const moc_graph* g, const Plan& pl, const int64_t* offs, const int32_t* seqs, const int32_t* lens, int32_t B, int64_t M,
                 int64_t* out_peak, int64_t* out_dur, int32_t* out_feasible, cudaStream_t st) {
    moc::LiveParams q{};
    q.n = g->n;
    q.C = g->C;
    q.B = B;
    q.M = M;
    q.image = (const uint4*)pl.live_image;
    q.sink_m = g->sink_m;
    for (int k = 0; k < moc::kLiveMaxN / 32; ++k) q.sinks[k] = g->live_sinks[k];
    for (int c = 2; c <= moc::kLivePlanes; ++c)
        for (int32_t v = 0; v < g->n; ++v)
            if (c <= (g->h_cap.empty() ? g->C : g->h_cap[v])) q.allow[c - 2][g->h_live_place[v] >> 5] |= 1u << (g->h_live_place[v] & 31);
    q.seqs = seqs;
    q.lens = lens;
    q.offs = offs;
    q.out_peak = out_peak;
    q.out_dur = out_dur;
    q.out_status = out_feasible;
    // groups of 32 sequences; one block per SM, as many warps as it takes to have every group at once (at most 16)
    const int64_t groups = ((int64_t)B + 31) / 32, per_sm = (groups + g->sm_count - 1) / g->sm_count, rounds = (per_sm + 15) / 16;
    const int wpb = (int)std::max<int64_t>((per_sm + rounds - 1) / rounds, 1);
    const int grid = (int)std::min<int64_t>(g->sm_count, (groups + wpb - 1) / wpb);
    q.per_block = (int32_t)(groups / grid);
    q.spare = (int32_t)(groups % grid);
    if (g->ev_before) MOC_CUDA(cudaEventRecord(g->ev_before, st));
    pl.live_fn<<<grid, 32 * wpb, moc::live_smem_bytes(g->n, live_words(g->n)), st>>>(q);
    ++g_launches;
    MOC_CUDA(cudaGetLastError());
    if (g->ev_after) MOC_CUDA(cudaEventRecord(g->ev_after, st));
    return MOC_OK;
}

// Enqueues the evaluation of plan `pl`.  With `offs` the evaluation kernel reads the row offsets
// from that array, which the offsets kernel fills first from the lengths when `fill_offs` is set
// (packed rows) and which the caller has filled otherwise; with offs == nullptr (only the
// warp-per-sequence kernel can do that) the evaluation kernel finds the packed rows itself.
int enqueue_eval(const moc_graph* g, const Plan& pl, int64_t* offs, bool fill_offs, const int32_t* seqs, const int32_t* lens,
                 int32_t B, int64_t M, int64_t* out_peak, int64_t* out_dur, int32_t* out_feasible,
                 cudaStream_t st) {
    int grid = (int)std::min<int64_t>(pl.grid, ((int64_t)B + pl.gpc - 1) / pl.gpc);   // lane path: gpc = sequences per group
    int block = pl.block;
    size_t smem = pl.smem;
    const TeamShape team = pl.pair_team ? team_shape(g, B) : TeamShape();
    if (pl.pair_team) {
        grid = team.grid;
        block = 32 * team.team * team.groups;
        smem = pl.pair_graph_b + (size_t)team.groups * pl.pair_warp_b;
    } else if (pl.pair) {
        // Shape of this launch.  A warp works through its sequences one after the other, so a launch
        // takes ceil(sequences per block / warps per block) rounds, and a round costs about as much as
        // the SM has warps (the kernel is bound by on-chip throughput) but never less than a round of a
        // half-empty SM.  Pick the warps per block and blocks per SM with the least rounds x warps.
        int64_t best_cost = INT64_MAX;
        int best_w = pl.gpc, best_nb = std::max(1, pl.grid / std::max(1, pl.sm_count));
        for (int wpb = 4; wpb <= 19; ++wpb) {
            const int nb = pl.pair_nb[wpb];
            if (nb < 1) continue;
            const int64_t blocks = (int64_t)pl.sm_count * nb;
            const int64_t per_block = (B + blocks - 1) / blocks;
            const int64_t rounds = (per_block + wpb - 1) / wpb;
            const int64_t cost = rounds * std::max(wpb * nb, 16);
            // equal cost: fewer, larger blocks (every block stages the graph in its shared memory)
            if (cost < best_cost || (cost == best_cost && nb <= best_nb)) {
                best_cost = cost;
                best_w = wpb;
                best_nb = nb;
            }
        }
        grid = (int)std::min<int64_t>((int64_t)pl.sm_count * best_nb, ((int64_t)B + best_w - 1) / best_w);
        // A batch that one round of 16 warps per SM holds is bound by the latency of a sequence: spread it over all
        // SMs, with at least eight warps per block to stage the graph (n = 353, 64-bit sums, B = 1501: 11 warps on
        // 148 SMs instead of 16 on 94).
        const int spread = (int)std::max<int64_t>(8, ((int64_t)B + pl.sm_count - 1) / pl.sm_count);
        if (spread <= 16 && pl.pair_nb[spread] >= 1 && (g->want_kind != MOC_KERNEL_WARP || g->want_b == 0)) {
            best_w = spread;
            grid = std::min(B, pl.sm_count);
        }
        block = 32 * best_w;
        smem = pl.pair_graph_b + (size_t)best_w * pl.pair_warp_b;
    }
    QuadShape teams;
    if (pl.quad && pl.quad_mode != moc::kQuadBlock) {
        teams = quad_shape(g, B, false);
        grid = teams.grid;
        block = 32 * teams.team * teams.groups;
        const QuadBytes z = quad_bytes(g, pl.wide, false);
        smem = z.graph() + (size_t)teams.groups * z.state();
    } else if (pl.quad) {
        int nb = 1;
        quad_threads(pl, g->n, g->C, B, &block, &nb);
        grid = (int)std::min<int64_t>((int64_t)pl.sm_count * nb, B);
    }
    if (offs && fill_offs) {
        moc::offsets_kernel<<<(B + moc::kOffsTile - 1) / moc::kOffsTile, moc::kOffsThreads, 0, st>>>(lens, B, offs);
        ++g_launches;
    }
    if (g->ev_before) MOC_CUDA(cudaEventRecord(g->ev_before, st));
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    if (pl.quad) {
        moc::QuadParams q = quad_params(g, pl);
        q.B = B;
        q.per_block = B / grid;
        q.spare = B % grid;
        q.team = teams.team;
        q.M = M;
        q.seqs = seqs;
        q.lens = lens;
        q.offs = offs;
        q.out_peak = out_peak;
        q.out_dur = out_dur;
        q.out_status = out_feasible;
        MOC_CUDA(cudaLaunchKernelEx(&cfg, pl.quad_fn, q));
    } else if (pl.lane) {
        const LaneLayout& L = g->lane[5 - pl.lane_lg];
        moc::LaneParams q{};
        q.n = g->n;
        q.max_T = g->C * g->n;
        q.B = B;
        q.n_bundles = L.n_bundles;
        q.M = M;
        q.base_dur = g->sum_w;
        q.rec = (const uint4*)(pl.wide ? L.d_rec64 : L.d_rec32);
        q.succ = L.d_succ;
        q.seqs = seqs;
        q.lens = lens;
        q.offs = offs;
        q.out_peak = out_peak;
        q.out_dur = out_dur;
        q.out_status = out_feasible;
        q.rec_bytes = pl.lane_rec_b; q.succ_bytes = pl.lane_succ_b;
        q.word_bytes = pl.lane_word_b; q.delta_bytes = pl.lane_delta_b;
        MOC_CUDA(cudaLaunchKernelEx(&cfg, pl.lane_fn, q));
    } else if (pl.pair) {
        moc::PairParams q{};
        q.n = g->n;
        q.n_tiles = g->n_tiles;
        q.max_T = g->C * g->n;
        q.rec = pl.wide ? g->d_rec64 : g->d_rec32;
        q.wslot = (const uint64_t*)g->d_wslot;
        q.sell = g->d_sell;
        q.base_dur = g->sum_w;
        q.seqs = seqs;
        q.lens = lens;
        q.offs = offs;
        q.B = B;
        q.M = M;
        q.out_peak = out_peak;
        q.out_dur = out_dur;
        q.out_status = out_feasible;
        q.rec_bytes = pl.rec_bytes; q.w_bytes = pl.w_bytes; q.sell_bytes = pl.sell_bytes;
        q.word_bytes = pl.word_bytes; q.delta_bytes = pl.delta_bytes;
        q.split = g->split;
        q.small_w = g->sum_w < ((int64_t)1 << 32) ? 1 : 0;
        q.per_block = B / grid;
        q.spare = B % grid;
        q.team = team.team;
        MOC_CUDA(cudaLaunchKernelEx(&cfg, pl.pair_fn, q));
    } else {
        moc::EvalParams p = base_params(g, pl);
        p.seqs = seqs;
        p.lens = lens;
        p.offs = offs;
        p.B = B;
        p.M = M;
        p.out_peak = out_peak;
        p.out_dur = out_dur;
        p.out_status = out_feasible;
        p.gstate = g->d_state;
        MOC_CUDA(cudaLaunchKernelEx(&cfg, pl.fn, p));
    }
    ++g_launches;
    MOC_CUDA(cudaGetLastError());
    if (g->ev_after) MOC_CUDA(cudaEventRecord(g->ev_after, st));
    return MOC_OK;
}

// Each block of the self-addressing kernel re-reads the lengths in front of its range: worth it
// while that redundant traffic (grid * B/2 * 4 bytes from L2) stays small next to a second launch.
bool rows_without_scratch(const Plan& pl, int32_t B) {
    return (pl.pair || pl.lane || pl.quad) && (int64_t)pl.grid * B * 2 <= (int64_t)16 << 20;
}

// The plan for a batch of B, made when a batch first needs it: looking a kernel up loads it, and a kernel that is never
// launched should cost a program nothing (first evaluation of a handle, kernels loaded: 28 us with every kernel that may
// serve it looked up, 25 with one; the next evaluation takes 18).  `walk`: the backward walk may serve it (which is
// told by live_fn); nullptr: the error is in *rc.
const Plan* plan_for(const moc_graph* g, int32_t B, bool walk, int* rc) {
    *rc = MOC_OK;
    if (walk && live_serves(g, B)) {
        if (!g->plan_live.valid) plan_live(g, &g->plan_live);
        if (g->plan_live.live_fn) return &g->plan_live;
    }
    const bool wide = g->sum_m > (int64_t)INT32_MAX / g->C;
    const size_t cap = g->smem_optin > 1024 ? g->smem_optin - 1024 : 0;
    auto quad = [&](Plan& kept, int mode) -> const Plan* {
        if (!kept.valid) {
            Plan pl;
            pl.wide = wide;
            plan_quad(g, cap, false, mode, &pl);
            pl.valid = true;
            kept = pl;
        }
        return kept.quad ? &kept : nullptr;
    };
    const bool any_block = g->want_kind == MOC_KERNEL_BLOCK || (g->want_kind == MOC_KERNEL_AUTO && !g->want_G && !g->want_gpc && g->C >= 3);
    if (any_block)
        if (const int team = quad_shape(g, B, false).team)
            if (const Plan* pl = team > 1 || g->C < 3 ? quad(g->plan_chip, moc::kQuadTeams) : quad(g->plan_warps, moc::kQuadWarps)) return pl;
    if (team_shape(g, B).team > 1) {
        Plan& kept = g->plan_team;
        if (!kept.valid) {
            Plan pl;
            pl.wide = wide;
            pair_bytes(g, &pl);
            pl.pair_fn = pair_fn(wide, -1);
            pl.pair = pl.pair_team = raise_smem_limit((const void*)pl.pair_fn, g->smem_optin) == cudaSuccess;
            if (!pl.pair) cudaGetLastError();
            pl.sm_count = g->sm_count;
            pl.grid = 2 * g->sm_count;
            pl.gpc = 1;
            pl.valid = true;
            kept = pl;
        }
        if (kept.pair) return &kept;
    }
    if (!g->plan_eval.valid) *rc = make_plan(g, false, &g->plan_eval);
    return *rc == MOC_OK ? &g->plan_eval : nullptr;
}

void forget_plans(moc_graph* g) { g->plan_eval = g->plan_team = g->plan_chip = g->plan_warps = g->plan_live = Plan(); }

int launch_eval(const moc_graph* g, const int32_t* seqs, const int32_t* lens, int32_t B, int64_t M,
                int64_t* out_peak, int64_t* out_dur, int32_t* out_feasible, cudaStream_t st) {
    int rc;
    const Plan* plan = plan_for(g, B, true, &rc);
    if (!plan) return rc;
    const Plan& pl = *plan;
    if (pl.live_fn) return enqueue_live(g, pl, nullptr, seqs, lens, B, M, out_peak, out_dur, out_feasible, st);
    if (rows_without_scratch(pl, B))
        return enqueue_eval(g, pl, nullptr, false, seqs, lens, B, M, out_peak, out_dur, out_feasible, st);
    rc = ensure((void**)&g->d_offs, &g->offs_cap, ((size_t)B + 1) * sizeof(int64_t));
    if (rc != MOC_OK) return rc;
    if (pl.global_state) {
        rc = ensure((void**)&g->d_state, &g->state_cap, (size_t)pl.grid * pl.group_bytes);
        if (rc != MOC_OK) return rc;
    }
    return enqueue_eval(g, pl, g->d_offs, true, seqs, lens, B, M, out_peak, out_dur, out_feasible, st);
}

}  // namespace

namespace moc_host {
int eval_rows(const moc_graph* g, const int64_t* offs, const int32_t* seqs, const int32_t* lens, int32_t B,
              int64_t M, int64_t* out_peak, int64_t* out_dur, int32_t* out_feasible, cudaStream_t st) {
    int rc;
    const Plan* plan = plan_for(g, B, true, &rc);
    if (!plan) return rc;
    const Plan& pl = *plan;
    if (pl.live_fn) return enqueue_live(g, pl, offs, seqs, lens, B, M, out_peak, out_dur, out_feasible, st);
    if (pl.global_state) {
        rc = ensure((void**)&g->d_state, &g->state_cap, (size_t)pl.grid * pl.group_bytes);
        if (rc != MOC_OK) return rc;
    }
    return enqueue_eval(g, pl, const_cast<int64_t*>(offs), false, seqs, lens, B, M, out_peak, out_dur, out_feasible, st);
}
}  // namespace moc_host

extern "C" {

const char* moc_last_error(void) { return g_err; }
int moc_last_launch_count(void) { return g_launches; }

int moc_graph_create(int32_t n, int64_t n_edges, const int32_t* edges, const int64_t* w,
                     const int64_t* m, moc_graph** out) {
    g_err[0] = 0;
    if (out) *out = nullptr;
    if (!out || !w || !m || n < 1 || n_edges < 0 || (n_edges > 0 && !edges))
        return fail(MOC_ERR_ARG, "moc_graph_create: null pointer, n < 1 or n_edges < 0");
    if (n > (1 << 27) || n_edges > (int64_t)INT32_MAX - 1)
        return fail(MOC_ERR_ARG, "moc_graph_create: n > 2^27 or n_edges >= 2^31-1");
    int64_t sum_w = 0, sum_m = 0;
    const int64_t lim = (int64_t(1) << 62) / 8;
    for (int32_t v = 0; v < n; ++v) {
        if (w[v] < 0 || m[v] < 0) return fail(MOC_ERR_OVERFLOW, "negative weight at node %d", v);
        if (w[v] >= lim - sum_w || m[v] >= lim - sum_m)
            return fail(MOC_ERR_OVERFLOW, "8*sum(w) or 8*sum(m) reaches 2^62");
        sum_w += w[v];
        sum_m += m[v];
    }
    std::vector<uint64_t> keys;
    try {
        keys.reserve((size_t)n_edges);
        for (int64_t e = 0; e < n_edges; ++e) {
            const int32_t u = edges[2 * e], v = edges[2 * e + 1];
            if (u < 0 || u >= n || v < 0 || v >= n)
                return fail(MOC_ERR_RANGE, "edge %lld = (%d,%d) outside [0,%d)", (long long)e, u, v, n);
            if (u == v) return fail(MOC_ERR_CYCLE, "self-loop at node %d", u);
            keys.push_back(((uint64_t)(uint32_t)u << 32) | (uint32_t)v);
        }
        std::sort(keys.begin(), keys.end());
        keys.erase(std::unique(keys.begin(), keys.end()), keys.end());
    } catch (const std::bad_alloc&) {
        return fail(MOC_ERR_NOMEM, "host allocation failed");
    }
    const int64_t ne = (int64_t)keys.size();
    std::vector<int32_t> succ_start, succ, indeg, queue, m32;
    try {
        succ_start.assign((size_t)n + 1, 0);
        succ.resize((size_t)std::max<int64_t>(ne, 1));
        indeg.assign((size_t)n, 0);
        m32.resize((size_t)n);
        for (int64_t e = 0; e < ne; ++e) {
            const int32_t u = (int32_t)(keys[e] >> 32), v = (int32_t)(keys[e] & 0xFFFFFFFFu);
            succ_start[u + 1]++;
            succ[e] = v;  // keys are sorted by (u, v): already grouped by producer
            indeg[v]++;
        }
        for (int32_t v = 0; v < n; ++v) succ_start[v + 1] += succ_start[v];
        // Kahn: the graph is a DAG iff every node gets removed
        queue.reserve((size_t)n);
        for (int32_t v = 0; v < n; ++v)
            if (indeg[v] == 0) queue.push_back(v);
        for (size_t h = 0; h < queue.size(); ++h) {
            const int32_t u = queue[h];
            for (int32_t e = succ_start[u]; e < succ_start[u + 1]; ++e)
                if (--indeg[succ[e]] == 0) queue.push_back(succ[e]);
        }
        if ((int32_t)queue.size() != n) return fail(MOC_ERR_CYCLE, "the edges contain a directed cycle");
        for (int32_t v = 0; v < n; ++v) m32[v] = (int32_t)std::min<int64_t>(m[v], INT32_MAX);
    } catch (const std::bad_alloc&) {
        return fail(MOC_ERR_NOMEM, "host allocation failed");
    }

    moc_graph* g = new (std::nothrow) moc_graph();
    if (!g) return fail(MOC_ERR_NOMEM, "host allocation failed");
    g->n = n;
    g->n_edges = ne;
    g->sum_m = sum_m;
    g->sum_w = sum_w;
    cudaError_t e = cudaGetDevice(&g->device);
    int smem = 0;
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&g->sm_count, cudaDevAttrMultiProcessorCount, g->device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, g->device);
    g->smem_optin = (size_t)smem;
    if (e != cudaSuccess) {
        delete g;
        return fail(MOC_ERR_CUDA, "moc_graph_create: %s", cudaGetErrorString(e));
    }
    try {
        g->h_w.assign(w, w + n);
        Tables tables;
        build_tables(g, keys, succ_start, succ, w, m, m32, &tables);
        e = tables.upload(&g->d_tables);
    } catch (const std::bad_alloc&) {
        moc_graph_destroy(g);
        return fail(MOC_ERR_NOMEM, "host allocation failed");
    }
    if (e != cudaSuccess) {
        const int rc = fail(e == cudaErrorMemoryAllocation ? MOC_ERR_NOMEM : MOC_ERR_CUDA, "moc_graph_create: %s", cudaGetErrorString(e));
        cudaGetLastError();
        moc_graph_destroy(g);
        return rc;
    }
    *out = g;
    return MOC_OK;
}

int moc_graph_set_max_copies(moc_graph* g, int32_t C) {
    g_err[0] = 0;
    if (!g || C < 1 || C > MOC_MAX_COPIES) return fail(MOC_ERR_ARG, "moc_graph_set_max_copies: C must be 1..%d", MOC_MAX_COPIES);
    if (!g->h_cap.empty()) {   // caps refer to the old C: back to a uniform cap
        int rc = moc_graph_set_node_caps(g, nullptr);
        if (rc != MOC_OK) return rc;
    }
    g->C = C;
    ++g->generation;
    forget_plans(g);
    g->plan_profile.valid = false;
    return MOC_OK;
}

int moc_graph_set_node_caps(moc_graph* g, const int32_t* caps) {
    g_err[0] = 0;
    if (!g) return fail(MOC_ERR_ARG, "moc_graph_set_node_caps: null handle");
    DeviceGuard dg(g->device);
    if (!dg.ok) return fail(MOC_ERR_CUDA, "cannot select device %d", g->device);
    // work queued on any stream may still read the old caps
    MOC_CUDA(cudaDeviceSynchronize());
    try {
        if (!caps) {
            g->h_cap.clear();
        } else {
            for (int32_t v = 0; v < g->n; ++v)
                if (caps[v] < 1 || caps[v] > g->C)
                    return fail(MOC_ERR_ARG, "moc_graph_set_node_caps: cap %d of node %d outside [1, C = %d]", caps[v], v, g->C);
            g->h_cap.assign(caps, caps + g->n);
        }
    } catch (const std::bad_alloc&) {
        return fail(MOC_ERR_NOMEM, "host allocation failed");
    }
    ++g->generation;
    if (caps) {
        if (!g->d_cap) MOC_CUDA(cudaMalloc((void**)&g->d_cap, std::max<size_t>((size_t)g->n * 4, 16)));
        MOC_CUDA(cudaMemcpy(g->d_cap, caps, (size_t)g->n * 4, cudaMemcpyHostToDevice));
    } else if (g->d_cap) {
        MOC_CUDA(cudaFree(g->d_cap));
        g->d_cap = nullptr;
    }
    // the caps are part of the node data of two layouts
    try {
        if (g->d_wslot) {
            const std::vector<uint64_t> wslot = slot_durations(g);
            MOC_CUDA(cudaMemcpy(g->d_wslot, wslot.data(), wslot.size() * 8, cudaMemcpyHostToDevice));
        }
    } catch (const std::bad_alloc&) {
        return fail(MOC_ERR_NOMEM, "host allocation failed");
    }
    set_lane_caps(g);
    for (const LaneLayout& L : g->lane) {
        if (!L.ok) continue;
        MOC_CUDA(cudaMemcpy(L.d_rec32, L.h_rec32.data(), L.h_rec32.size() * 4, cudaMemcpyHostToDevice));
        MOC_CUDA(cudaMemcpy(L.d_rec64, L.h_rec64.data(), L.h_rec64.size() * 4, cudaMemcpyHostToDevice));
    }
    return MOC_OK;
}

int moc_graph_set_kernel(moc_graph* g, int32_t kind, int32_t a, int32_t b) {
    g_err[0] = 0;
    if (!g) return fail(MOC_ERR_ARG, "moc_graph_set_kernel: null handle");
    bool ok = false;
    switch (kind) {
        case MOC_KERNEL_AUTO: ok = a == 0 && b == 0; break;
        case MOC_KERNEL_GROUP:
            ok = (a == 0 || a == 32 || a == 64 || a == 128 || a == 256 || a == 512 || a == 1024) && b >= 0 && b <= 32 &&
                 !(a && b && a * b > 1024);
            break;
        case MOC_KERNEL_WARP: ok = a == 0 && (b == 0 || (b >= 4 && b <= 16)); break;
        case MOC_KERNEL_BLOCK: ok = (a == 0 || (a >= 64 && a <= 1024 && a % 32 == 0)) && b == 0; break;
        case MOC_KERNEL_LANE: ok = (a == 0 || a == 8 || a == 16 || a == 32) && (b == 0 || (b >= 8 && b <= 32 && b % 8 == 0)); break;
        default: break;
    }
    if (!ok) return fail(MOC_ERR_ARG, "moc_graph_set_kernel: unsupported kind or shape (%d, %d, %d)", kind, a, b);
    g->want_kind = kind;
    g->want_a = a;
    g->want_b = b;
    g->want_G = kind == MOC_KERNEL_GROUP ? a : 0;
    g->want_gpc = (kind == MOC_KERNEL_GROUP || kind == MOC_KERNEL_WARP) ? b : 0;
    forget_plans(g);
    return MOC_OK;
}

int moc_graph_set_launch(moc_graph* g, int32_t tps, int32_t spb) {
    g_err[0] = 0;
    const bool ok_g = tps == 0 || tps == 32 || tps == 64 || tps == 128 || tps == 256 || tps == 512 || tps == 1024;
    if (!g || !ok_g || spb < 0 || spb > 32 || (tps && spb && tps * spb > 1024))
        return fail(MOC_ERR_ARG, "moc_graph_set_launch: unsupported shape (%d threads x %d sequences)", tps, spb);
    g->want_kind = MOC_KERNEL_AUTO;
    g->want_a = g->want_b = 0;
    g->want_G = tps;
    g->want_gpc = spb;
    forget_plans(g);
    return MOC_OK;
}

int moc_graph_set_timing_events(moc_graph* g, void* before, void* after) {
    g_err[0] = 0;
    if (!g || ((before == nullptr) != (after == nullptr)))
        return fail(MOC_ERR_ARG, "moc_graph_set_timing_events: null handle, or only one of the two events given");
    g->ev_before = (cudaEvent_t)before;
    g->ev_after = (cudaEvent_t)after;
    return MOC_OK;
}

void moc_graph_destroy(moc_graph* g) {
    if (!g) return;
    DeviceGuard dg(g->device);
    cudaFree(g->d_tables);
    cudaFree(g->d_cap);
    cudaFree(g->d_offs);
    cudaFree(g->d_state);
    cudaFree(g->d_stage_seqs);
    cudaFree(g->d_stage_u16);
    cudaFree(g->d_stage_io);
    if (g->h_stage) cudaFreeHost(g->h_stage);
    if (g->copy_stream) cudaStreamDestroy(g->copy_stream);
    for (cudaEvent_t ev : g->chunk_ev)
        if (ev) cudaEventDestroy(ev);
    delete g;
}

int moc_graph_info(const moc_graph* g, int32_t* n, int64_t* n_edges, int32_t* C, int32_t* wide) {
    g_err[0] = 0;
    if (!g) return fail(MOC_ERR_ARG, "moc_graph_info: null handle");
    if (n) *n = g->n;
    if (n_edges) *n_edges = g->n_edges;
    if (C) *C = g->C;
    if (wide) *wide = g->sum_m > (int64_t)INT32_MAX / g->C ? 1 : 0;
    return MOC_OK;
}

int moc_eval_batch(const moc_graph* g, const int32_t* seqs, const int32_t* lens, int32_t B, int64_t M,
                   int64_t* out_peak, int64_t* out_dur, int32_t* out_feasible, void* stream) {
    g_err[0] = 0;
    g_launches = 0;
    if (!g || B < 0) return fail(MOC_ERR_ARG, "moc_eval_batch: null handle or B < 0");
    if (B == 0) return MOC_OK;
    if (!seqs || !lens || !out_peak || !out_dur || !out_feasible)
        return fail(MOC_ERR_ARG, "moc_eval_batch: null array");
    if (reinterpret_cast<uintptr_t>(seqs) & 3) return fail(MOC_ERR_ARG, "moc_eval_batch: seqs not 4-byte aligned");
    DeviceGuard dg(g->device);
    if (!dg.ok) return fail(MOC_ERR_CUDA, "cannot select device %d", g->device);
    return launch_eval(g, seqs, lens, B, M, out_peak, out_dur, out_feasible, (cudaStream_t)stream);
}

// Host entry points.
//
// A large batch travels in three parts of 11/16, 4/16 and 1/16 of the ids on a copy stream owned by the handle, and the
// caller's stream evaluates the sequences that have arrived in full while the next part is under way: the link is
// busy throughout, every further part would cost it 4 us, and only the evaluation of the last sixteenth is exposed.  A
// batch whose copy is shorter than the calls that would cut it goes in one piece on the caller's stream.
//
// A caller's buffer may be much larger than the batch in it, and only the ids that the lengths add up to should travel.  Adding
// up 16384 lengths takes 3.4 us, so the first part starts before that where a sample of the lengths says that
// the batch fills the buffer (a wrong guess costs time, nothing else); otherwise, and for short batches, the lengths
// come first.  Buffers of 2 and 4 times the batch: 673 and 1303 us with the whole buffer sent, 410 and 408 now.
//
// Results go to pinned arrays of the caller straight from the device, behind the copies of later parts; to
// pageable ones with one copy into a pinned block of the handle and a memcpy.  Short batches in pinned memory
// are also fetched by a kernel: one launch instead of two copies and the widening.
//
// n = 442, B = 16384, ids as 16-bit words (17.4 MB, 318 us at the link's 54.8 GB/s; one copy alone
// takes 327): 445 -> 385 us a call.  B = 8: 49 -> 24 us, B = 200: 59 -> 32.
namespace {
constexpr int kHostPart[kHostParts] = {11, 4, 1};       // sixteenths
constexpr int64_t kHostCutSteps = (int64_t)1 << 21;      // from here on in parts (4 MB of 16-bit ids: 80 us of copy)
constexpr int64_t kHostFetchBytes = 256 << 10;           // up to here fetched by a kernel (about 45 GB/s, no call per array)
constexpr int32_t kHostDirect = 2048;                    // up to here sequences' results are written by the evaluation itself
constexpr int32_t kHostSumFirst = 4096;                  // up to here the lengths are always added up first (1 us)

int host_streams(const moc_graph* g) {
    if (!g->copy_stream) MOC_CUDA(cudaStreamCreateWithFlags(&g->copy_stream, cudaStreamNonBlocking));
    for (cudaEvent_t& ev : g->chunk_ev)
        if (!ev) MOC_CUDA(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
    return MOC_OK;
}

// Address under which kernels reach a host array of `bytes` bytes (at least one), or nullptr unless every byte of it lies
// in pinned memory that is mapped at its own address.  The array is followed from one registration to the next: an
// array whose two ends are registered may still have a hole.
void* mapped_address(const void* host, size_t bytes) {
    using Query = CUresult (*)(unsigned int, CUpointer_attribute*, void**, CUdeviceptr);
    static const Query query = [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult found{};
        if (cudaGetDriverEntryPointByVersion("cuPointerGetAttributes", &fn, 12000, cudaEnableDefault, &found) != cudaSuccess) cudaGetLastError();
        return found == cudaDriverEntryPointSuccess ? (Query)fn : nullptr;
    }();
    if (!query) return nullptr;
    const CUdeviceptr first = (CUdeviceptr)(uintptr_t)host, end = first + bytes;
    for (CUdeviceptr at = first; at < end;) {
        unsigned int type = 0, managed = 0;
        CUdeviceptr device = 0, start = 0;
        size_t size = 0;
        CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                      CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
        void* out[] = {&type, &managed, &device, &start, &size};
        if (query(5, what, out, at) != CUDA_SUCCESS) return nullptr;
        if (type != CU_MEMORYTYPE_HOST || managed || device != at || at < start || at - start >= size) return nullptr;
        at = start + size;
    }
    return const_cast<void*>(host);
}

// Work of a host entry point that reads or writes the caller's arrays: whatever way the call returns, it is over by then.
struct HostWork {
    cudaStream_t copies = nullptr, work = nullptr;
    bool begun = false;
    HostWork() = default;
    HostWork(const HostWork&) = delete;
    ~HostWork() {
        if (!begun) return;
        cudaStreamSynchronize(copies);
        if (work != copies) cudaStreamSynchronize(work);
    }
};

// Ids of the sequences b0 .. b1 - 1: the sum of max(lens, 0), in two 16-bit halves that the compiler adds up in vectors.
int64_t steps_of(const int32_t* lens, int32_t b0, int32_t b1) {
    int64_t sum = 0;
    for (int32_t b = b0; b < b1;) {
        const int32_t e = (int32_t)std::min<int64_t>(b1, (int64_t)b + 32768);
        uint32_t lo = 0, hi = 0;
        for (; b < e; ++b) {
            const uint32_t x = (uint32_t)std::max(lens[b], 0);
            lo += x & 0xFFFFu;
            hi += x >> 16;
        }
        sum += (int64_t)lo + ((int64_t)hi << 16);
    }
    return sum;
}

// What 64 of the lengths, evenly spread, let the sum of all be.
int64_t sampled_steps(const int32_t* lens, int32_t B) {
    int64_t sum = 0;
    for (int32_t k = 0; k < 64; ++k) sum += std::max(lens[(int64_t)B * k / 64], 0);
    return (int64_t)((double)sum / 64 * B);
}

// ids: host array of n_steps node ids, 4 bytes each (wide_ids) or 2 bytes each, of which the sequences take the first.
int eval_host(const moc_graph* g, const void* ids, bool wide_ids, int64_t n_steps, const int32_t* lens, int32_t B,
              int64_t M, int64_t* out_peak, int64_t* out_dur, int32_t* out_feasible, cudaStream_t st, const char* who) {
    const size_t id_b = wide_ids ? 4 : 2, bB = (size_t)B;
    DeviceGuard dg(g->device);
    if (!dg.ok) return fail(MOC_ERR_CUDA, "cannot select device %d", g->device);
    int rc = MOC_OK;
    const size_t o_peak = 0, o_dur = bB * 8, o_st = 2 * bB * 8, o_lens = align16(o_st + bB * 4), res_bytes = o_st + bB * 4, io_bytes = o_lens + bB * 4;
    rc = ensure((void**)&g->d_stage_io, &g->stage_io_cap, io_bytes);
    if (rc != MOC_OK) return rc;
    int64_t* d_peak = (int64_t*)(g->d_stage_io + o_peak);
    int64_t* d_dur = (int64_t*)(g->d_stage_io + o_dur);
    int32_t* d_st = (int32_t*)(g->d_stage_io + o_st);
    int32_t* d_lens = (int32_t*)(g->d_stage_io + o_lens);
    auto too_long = [&](int64_t sum) {
        return fail(MOC_ERR_ARG, "%s: lens sum to %lld > n_steps %lld", who, (long long)sum, (long long)n_steps);
    };
    const bool room = g->stage_seqs_cap >= (size_t)n_steps * 4 + 16 && (wide_ids || g->stage_u16_cap >= (size_t)n_steps * 2 + 16);
    int64_t need = -1;                         // ids of the batch: not known yet
    if (B <= kHostSumFirst || !room || sampled_steps(lens, B) / 32 * 33 < n_steps) {
        need = steps_of(lens, 0, B);
        if (need > n_steps) return too_long(need);
        rc = ensure((void**)&g->d_stage_seqs, &g->stage_seqs_cap, (size_t)need * 4 + 16);
        if (rc != MOC_OK) return rc;
    }
    const int64_t send = need >= 0 ? need : n_steps;
    // how the ids come: fetched by a kernel, copied in one piece, or in parts
    const void* m_ids = nullptr;
    const int32_t* m_lens = nullptr;
    if (send > 0 && send * (int64_t)id_b <= kHostFetchBytes && (m_ids = mapped_address(ids, (size_t)send * id_b)) != nullptr)
        m_lens = (const int32_t*)mapped_address(lens, bB * 4);
    if (!m_lens && !wide_ids) {
        rc = ensure((void**)&g->d_stage_u16, &g->stage_u16_cap, (size_t)send * 2 + 16);
        if (rc != MOC_OK) return rc;
    }
    const bool parts = send >= kHostCutSteps;
    for (int k = 0; k < (parts ? kHostParts : 1); ++k)         // before anything is in flight: a first call looks its kernels up
        if (!plan_for(g, parts ? (int32_t)((int64_t)B * kHostPart[k] / 16) : B, true, &rc)) return rc;
    void* stage = wide_ids ? (void*)g->d_stage_seqs : (void*)g->d_stage_u16;
    cudaStream_t cs = st;
    HostWork in_flight;
    int64_t at[kHostParts + 1] = {0};         // ids on the device once part k has arrived
    auto copy_part = [&](int k) -> int {       // part k of the ids, and the lengths behind the first
        const int64_t cnt = at[k + 1] - at[k];
        if (cnt) MOC_CUDA(cudaMemcpyAsync((char*)stage + at[k] * id_b, (const char*)ids + at[k] * id_b, (size_t)cnt * id_b, cudaMemcpyHostToDevice, cs));
        if (k == 0) MOC_CUDA(cudaMemcpyAsync(d_lens, lens, bB * 4, cudaMemcpyHostToDevice, cs));
        if (parts) MOC_CUDA(cudaEventRecord(g->chunk_ev[k], cs));
        return MOC_OK;
    };
    const int n_parts = parts ? kHostParts : 1;
    for (int k = 0, sum = 0; k < n_parts; ++k) {
        sum += parts ? kHostPart[k] : 16;
        at[k + 1] = sum == 16 ? send : (send / 16 * sum) & ~int64_t(7);      // every part starts on a 16-byte boundary
    }
    if (parts) {
        rc = host_streams(g);
        if (rc != MOC_OK) return rc;
        cs = g->copy_stream;
        // the copy stream starts once the caller's stream has reached this call
        MOC_CUDA(cudaEventRecord(g->chunk_ev[kHostParts], st));
        MOC_CUDA(cudaStreamWaitEvent(cs, g->chunk_ev[kHostParts], 0));
    }
    in_flight.copies = cs;
    in_flight.work = st;
    in_flight.begun = true;
    if (!m_lens) {
        rc = copy_part(0);
        if (rc != MOC_OK) return rc;
    }
    // the rest while the first part is under way
    if (need < 0) {
        need = steps_of(lens, 0, B);
        if (need > n_steps) return too_long(need);
        for (int k = 1; k < n_parts; ++k) at[k + 1] = std::min(at[k + 1], std::max(need, at[1]));
    }
    for (int k = 1; k < n_parts && !m_lens; ++k) {
        rc = copy_part(k);
        if (rc != MOC_OK) return rc;
    }
    int launches = 0;
    if (m_lens) {                  // under way while the rest is prepared
        const int blocks = (int)std::min<int64_t>((std::max<int64_t>(need / 4, B) + 255) / 256, (int64_t)g->sm_count * 2);
        if (wide_ids) moc::fetch_kernel<int32_t><<<blocks, 256, 0, st>>>((const int32_t*)m_ids, need, g->d_stage_seqs, m_lens, B, d_lens);
        else moc::fetch_kernel<uint16_t><<<blocks, 256, 0, st>>>((const uint16_t*)m_ids, need, g->d_stage_seqs, m_lens, B, d_lens);
        MOC_CUDA(cudaGetLastError());
        ++launches;
    }
    // sequences that are complete with each part
    int32_t cb[kHostParts + 1] = {0};
    int64_t co[kHostParts + 1] = {0};
    cb[n_parts] = B;
    co[n_parts] = need;
    if (parts) {
        int64_t here = 0;
        int k = 0;
        for (int32_t b = 0; b < B && k + 1 < n_parts;) {
            const int32_t b1 = (int32_t)std::min<int64_t>(B, (int64_t)b + 64);
            const int64_t sum = steps_of(lens, b, b1);
            while (k + 1 < n_parts && here + sum > at[k + 1]) {      // this piece of 64 sequences reaches beyond part k
                cb[++k] = b;
                co[k] = here;
            }
            here += sum;
            b = b1;
        }
        for (++k; k < n_parts; ++k) {
            cb[k] = B;
            co[k] = need;
        }
    }
    int64_t *m_peak = (int64_t*)mapped_address(out_peak, bB * 8), *m_dur = m_peak ? (int64_t*)mapped_address(out_dur, bB * 8) : nullptr;
    int32_t* m_st = m_dur ? (int32_t*)mapped_address(out_feasible, bB * 4) : nullptr;
    if (!m_st && res_bytes > g->h_stage_cap) {
        if (g->h_stage) MOC_CUDA(cudaFreeHost(g->h_stage));
        g->h_stage = nullptr;
        g->h_stage_cap = 0;
        MOC_CUDA(cudaMallocHost((void**)&g->h_stage, res_bytes * 2));
        g->h_stage_cap = res_bytes * 2;
    }
    for (int k = 0; k < n_parts; ++k) {
        if (parts) MOC_CUDA(cudaStreamWaitEvent(st, g->chunk_ev[k], 0));
        const int64_t cnt = at[k + 1] - at[k];
        if (!m_lens && !wide_ids && cnt) {
            const int blocks = (int)std::min<int64_t>((cnt / 8 + 255) / 256 + 1, (int64_t)g->sm_count * 8);
            moc::widen_ids_kernel<<<blocks, 256, 0, st>>>(g->d_stage_u16 + at[k], g->d_stage_seqs + at[k], cnt);
            ++launches;
        }
        const int32_t b0 = cb[k], nb = cb[k + 1] - cb[k];
        if (nb <= 0) continue;
        const bool direct = m_st && nb <= kHostDirect;
        rc = launch_eval(g, g->d_stage_seqs + co[k], d_lens + b0, nb, M, (direct ? m_peak : d_peak) + b0, (direct ? m_dur : d_dur) + b0,
                         (direct ? m_st : d_st) + b0, st);
        if (rc != MOC_OK) return rc;
        if (m_st && !direct) {
            moc::deliver_kernel<<<std::min((nb + 255) / 256, g->sm_count), 256, 0, st>>>(d_peak + b0, d_dur + b0, d_st + b0, nb, m_peak + b0,
                                                                                       m_dur + b0, m_st + b0);
            MOC_CUDA(cudaGetLastError());
            ++launches;
        }
    }
    g_launches += launches;      // the evaluation launches were counted as they were enqueued
    if (!m_st) MOC_CUDA(cudaMemcpyAsync(g->h_stage, g->d_stage_io, res_bytes, cudaMemcpyDeviceToHost, st));
    MOC_CUDA(cudaStreamSynchronize(st));       // which waits for the copy stream's events
    in_flight.begun = false;
    if (m_st) return MOC_OK;
    memcpy(out_peak, g->h_stage + o_peak, bB * 8);
    memcpy(out_dur, g->h_stage + o_dur, bB * 8);
    memcpy(out_feasible, g->h_stage + o_st, bB * 4);
    return MOC_OK;
}
}  // namespace

int moc_eval_batch_host(const moc_graph* g, const int32_t* seqs, int64_t n_steps, const int32_t* lens,
                        int32_t B, int64_t M, int64_t* out_peak, int64_t* out_dur,
                        int32_t* out_feasible, void* stream) {
    g_err[0] = 0;
    g_launches = 0;
    if (!g || B < 0 || n_steps < 0) return fail(MOC_ERR_ARG, "moc_eval_batch_host: null handle or negative size");
    if (B == 0) return MOC_OK;
    if (!lens || !out_peak || !out_dur || !out_feasible || (n_steps > 0 && !seqs))
        return fail(MOC_ERR_ARG, "moc_eval_batch_host: null array");
    return eval_host(g, seqs, true, n_steps, lens, B, M, out_peak, out_dur, out_feasible, (cudaStream_t)stream, "moc_eval_batch_host");
}

int moc_eval_batch_host16(const moc_graph* g, const uint16_t* seqs, int64_t n_steps, const int32_t* lens,
                          int32_t B, int64_t M, int64_t* out_peak, int64_t* out_dur,
                          int32_t* out_feasible, void* stream) {
    g_err[0] = 0;
    g_launches = 0;
    if (!g || B < 0 || n_steps < 0) return fail(MOC_ERR_ARG, "moc_eval_batch_host16: null handle or negative size");
    if (g->n > 65535) return fail(MOC_ERR_ARG, "moc_eval_batch_host16: n = %d does not fit 16-bit node ids", g->n);
    if (B == 0) return MOC_OK;
    if (!lens || !out_peak || !out_dur || !out_feasible || (n_steps > 0 && !seqs))
        return fail(MOC_ERR_ARG, "moc_eval_batch_host16: null array");
    return eval_host(g, seqs, false, n_steps, lens, B, M, out_peak, out_dur, out_feasible, (cudaStream_t)stream, "moc_eval_batch_host16");
}

// ---- evaluation without any allocation -----------------------------------------------------------
// Packing offsets for moc_eval_batch_noalloc live in this array of the library's device image.  In
// host code `g_noalloc_offs` is only a stand-in for the symbol, not a device address: the address a
// kernel can use comes from cudaGetSymbolAddress, asked once per device with that device current.
static __device__ __align__(256) long long g_noalloc_offs[MOC_NOALLOC_MAX_B + 1];

namespace {
constexpr int kMaxDevices = 64;
int64_t* g_noalloc_ptr[kMaxDevices] = {};  // device address of g_noalloc_offs, per device ordinal

// Caller has made `device` current.
int noalloc_offsets(int device, int64_t** out) {
    if (device < 0 || device >= kMaxDevices) return fail(MOC_ERR_ARG, "device ordinal %d not supported", device);
    int64_t* ptr = __atomic_load_n(&g_noalloc_ptr[device], __ATOMIC_ACQUIRE);
    if (!ptr) {
        cudaError_t e = cudaGetSymbolAddress((void**)&ptr, g_noalloc_offs);
        if (e != cudaSuccess || !ptr)
            return fail(MOC_ERR_CUDA, "cudaGetSymbolAddress(scratch): %s", cudaGetErrorString(e));
        __atomic_store_n(&g_noalloc_ptr[device], ptr, __ATOMIC_RELEASE);
    }
    *out = ptr;
    return MOC_OK;
}
}  // namespace

int moc_eval_batch_noalloc(const moc_graph* g, const int32_t* seqs, const int32_t* lens, int32_t B,
                           int64_t M, int64_t* out_peak, int64_t* out_dur, int32_t* out_feasible,
                           void* stream) {
    g_err[0] = 0;
    g_launches = 0;
    if (!g || B < 0) return fail(MOC_ERR_ARG, "moc_eval_batch_noalloc: null handle or B < 0");
    if (B == 0) return MOC_OK;
    if (B > MOC_NOALLOC_MAX_B)
        return fail(MOC_ERR_ARG, "moc_eval_batch_noalloc: B = %d exceeds the fixed scratch of %d sequences; "
                    "split the batch or use moc_eval_batch", B, MOC_NOALLOC_MAX_B);
    if (!seqs || !lens || !out_peak || !out_dur || !out_feasible)
        return fail(MOC_ERR_ARG, "moc_eval_batch_noalloc: null array");
    if (reinterpret_cast<uintptr_t>(seqs) & 3) return fail(MOC_ERR_ARG, "moc_eval_batch_noalloc: seqs not 4-byte aligned");
    DeviceGuard dg(g->device);
    if (!dg.ok) return fail(MOC_ERR_CUDA, "cannot select device %d", g->device);
    int64_t* offs = nullptr;
    int rc = noalloc_offsets(g->device, &offs);
    if (rc != MOC_OK) return rc;
    const Plan* plan = plan_for(g, B, false, &rc);  // attribute and occupancy queries only
    if (!plan) return rc;
    const Plan& pl = *plan;
    if (pl.global_state)
        return fail(MOC_ERR_ARG, "moc_eval_batch_noalloc: this graph needs a global workspace "
                    "(per-sequence state exceeds shared memory); use moc_eval_batch");
    // the offsets kernel rewrites offs[0..B] before the evaluation kernel reads them
    return enqueue_eval(g, pl, offs, true, seqs, lens, B, M, out_peak, out_dur, out_feasible, (cudaStream_t)stream);
}

int moc_mem_profile(const moc_graph* g, const int32_t* seq, int32_t len, int64_t* out_profile,
                    int32_t* out_free, int32_t* out_status, void* stream) {
    g_err[0] = 0;
    g_launches = 0;
    if (!g || len < 0 || !out_status || (len > 0 && (!seq || !out_profile)))
        return fail(MOC_ERR_ARG, "moc_mem_profile: null pointer or len < 0");
    if (reinterpret_cast<uintptr_t>(seq) & 3) return fail(MOC_ERR_ARG, "moc_mem_profile: seq not 4-byte aligned");
    DeviceGuard dg(g->device);
    if (!dg.ok) return fail(MOC_ERR_CUDA, "cannot select device %d", g->device);
    cudaStream_t st = (cudaStream_t)stream;
    if (!g->plan_profile.valid) {
        int rc = make_plan(g, true, &g->plan_profile);
        if (rc != MOC_OK) return rc;
    }
    const Plan& pl = g->plan_profile;
    if (pl.quad) {
        moc::QuadParams q = quad_params(g, pl);
        q.B = 1;
        q.M = INT64_MAX;
        q.seqs = seq;
        q.single_len = len;
        q.out_status = out_status;
        q.out_profile = out_profile;
        q.out_free = out_free;
        // threads (us per call with 128 / 256 / 512 / 1024; calls of 5.6 are the host's time): n = 60 5.6 / 5.6 / 5.6 / 5.6, 442 6.7 / 5.7 / 5.7 / 6.2, 1000 10.3 / 8.2 /
        // 6.2 / 7.2, 2600 17.5 / 12.3 / 10.9 / 12.3, 4800 27.7 / 18.5 / 16.4 / 15.9
        const int thr = g->n < 200 ? 256 : (g->n < 3000 ? 512 : 1024);
        q.team = thr / 32;
        pl.quad_fn<<<1, thr, pl.smem, st>>>(q);
        ++g_launches;
        MOC_CUDA(cudaGetLastError());
        return MOC_OK;
    }
    if (pl.global_state) {
        int rc = ensure((void**)&g->d_state, &g->state_cap, (size_t)pl.group_bytes);
        if (rc != MOC_OK) return rc;
    }
    moc::EvalParams p = base_params(g, pl);
    p.seqs = seq;
    p.single_len = len;
    p.B = 1;
    p.M = INT64_MAX;
    p.out_status = out_status;
    p.out_profile = out_profile;
    p.out_free = out_free;
    p.gstate = g->d_state;
    pl.fn<<<1, pl.block, pl.smem, st>>>(p);
    ++g_launches;
    MOC_CUDA(cudaGetLastError());
    return MOC_OK;
}

}  // extern "C"
