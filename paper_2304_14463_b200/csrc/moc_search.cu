// Host side of the search entry points of libmoc_b200.so (declared in include/moc.h): state of the
// chains on the device and the per-generation launch sequence.  Proposals, scoring and selection
// all run in kernels (moc_search_kernels.cuh and the evaluation kernels).
#include <algorithm>
#include <new>

#include <vector>

#include "moc_cache_host.cuh"
#include "moc_search_kernels.cuh"
#include "moc_search_score_kernel.cuh"
#include "moc_search_walk_kernel.cuh"

using namespace moc_host;

struct moc_search {
    const moc_graph* g = nullptr;
    int device = 0;
    int32_t P = 0, stride = 0;
    int64_t M = 0;
    uint64_t seed = 0;
    uint32_t generation = 0;   // generations completed (proposed, scored and settled)
    char* d_block = nullptr;   // one allocation, carved up below
    int32_t* d_bad = nullptr;
    moc::SearchParams p{};
    // search on the incremental evaluation (off until moc_search_set_samples switches it on)
    bool incremental = false;
    int32_t samples = 1;
    moc_cache* cache = nullptr;
    char* d_inc = nullptr;
    moc::SearchIncParams ip{};
    // one kernel per generation with a warp per chain (moc_search_score_kernel.cuh) instead of draw, score, pick
    bool fused = false;
    moc::ScoreParams sp{};
    int score_wpb = 0, score_grid_cap = 0;
    const void* score_fn = nullptr;
    size_t score_smem = 0;
    // all generations of a call in one kernel (moc_search_walk_kernel.cuh)
    uint64_t graph_generation = 0;     // the graph's C and caps when the chains were evaluated
    moc::WalkParams wp{};
    bool walk_planned = false, walk_fits = false;
    bool walk_wide = false, walk_lists = false;
    const void* walk_fn[2] = {};       // without and with the bound on the new peak; null: not prepared (walk_variant)
    bool walk_scores = false;          // incremental, and the walk kernel does it (no cache)
    bool walk_sizes = false;           // with the bound on the new peak, the output sizes lie on chip
    int walk_wpb = 0, walk_grid = 0;
    size_t walk_smem = 0, walk_smem_floor = 0;
};

namespace {

size_t up256(size_t x) { return (x + 255) & ~size_t(255); }

int chain_blocks(int32_t P) { return (P + moc::kSearchThreads / 32 - 1) / (moc::kSearchThreads / 32); }

// Launch shape of the warp-per-chain generation kernel; false when the graph's largest in-degree or the row
// length leaves fewer than four warps on an SM.
bool plan_fused(moc_search* s) {
    const moc_graph* g = s->g;
    const moc_cache* h = s->cache;
    moc::ScoreParams& sp = s->sp;
    const size_t msz = h->wide ? 8 : 4;
    const int32_t worst = 4 + 2 * g->max_indeg;
    sp.list_cap = std::max(128, (worst + 31) & ~31);
    sp.warp_bytes = (uint32_t)moc::score_warp_bytes(h->c.occ_stride, h->c.stride, msz, sp.list_cap, &sp.fre_b, &sp.row_b, &sp.prof_b,
                                                   &sp.lh_b, &sp.val_b, &sp.diff_b);
    const size_t cap = g->smem_optin > 2048 ? g->smem_optin - 2048 : 0;
    if ((size_t)sp.warp_bytes * 4 > cap) return false;
    // with the block's own copy of the graph when that still leaves eight warps on an SM, else from global memory
    const int64_t E = g->n_edges;
    const size_t graph_b = moc::score_graph_bytes(g->n, E, msz, &sp.gs_pred_b, &sp.gs_m_b, &sp.gs_succ_b, &sp.gs_predl_b);
    sp.graph_bytes = (uint32_t)std::min<size_t>(graph_b, 0xFFFFFFF0u);
    int best = 0;
    for (int chip = 1; chip >= 0; --chip) {
        if (chip && (g->n > 65535 || graph_b > cap / 4)) continue;
        s->score_fn = score_fn(h->wide, chip != 0);
        if (cudaFuncSetAttribute(s->score_fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(g->smem_optin - 1024)) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        const size_t fixed = chip ? sp.graph_bytes : 0;
        best = 0;
        for (int k = 1; k <= moc::kScoreThreads / 32; ++k) {
            const size_t blk = fixed + (size_t)sp.warp_bytes * k;
            if (blk > cap) break;
            int nb = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, s->score_fn, 32 * k, blk) != cudaSuccess) {
                cudaGetLastError();
                return false;
            }
            if (nb * k >= best && nb > 0) { best = nb * k; s->score_wpb = k; }     // ties: the larger block (one copy of the graph)
        }
        s->score_smem = fixed + (size_t)sp.warp_bytes * s->score_wpb;
        if (best >= 8) break;
    }
    if (best < 4) return false;
    s->score_grid_cap = g->sm_count * (best / s->score_wpb);
    return true;
}

// Launch shape of the kernel that takes a warp per chain through all generations; leaves walk_fits false when the
// graph has no warp-per-sequence layout (C > 2, very uneven degrees) or fewer than four warps fit an SM.
void plan_walk(moc_search* s) {
    s->walk_planned = true;
    s->walk_fits = false;
    const moc_graph* g = s->g;
    if (g->C > 2 || g->d_rec32 == nullptr) return;
    const bool wide = g->sum_m > (int64_t)INT32_MAX / g->C;
    if (wide && !g->split_ok) return;
    const size_t per_vec = wide ? 2 : 4, nvec = ((size_t)g->C * g->n + 2 + per_vec - 1) / per_vec, v_max = ((nvec + 31) / 32) | 1;
    moc::WalkParams& w = s->wp;
    for (uint32_t r = 0; r < 10; ++r) {
        w.round_key[2 * r] = s->p.seed_lo + r * moc::kPhiloxWeyl0;
        w.round_key[2 * r + 1] = s->p.seed_hi + r * moc::kPhiloxWeyl1;
    }
    w.n = g->n;
    w.C = g->C;
    w.n_tiles = g->n_tiles;
    w.split = g->split;
    w.rec = wide ? g->d_rec64 : g->d_rec32;
    w.sell = g->d_sell;
    w.succ_start = g->d_succ_start;
    w.succ = g->d_succ;
    w.pred_start = g->d_pred_start;
    w.pred = g->d_pred;
    w.w = g->d_w;
    w.m = g->d_m64;
    w.rec_bytes = (wide ? 16u : 8u) * 64u * (uint32_t)g->n_tiles;
    w.sell_bytes = (4u * (uint32_t)g->sell_len + 15u) & ~15u;
    w.word_bytes = (4u * ((uint32_t)g->n + 2u) + 15u) & ~15u;
    w.delta_bytes = (uint32_t)(moc::kPairDeltaFront + 32 * v_max * 16);
    const size_t warp_b = moc::walk_warp_bytes(w.word_bytes, w.delta_bytes), graph_b = (size_t)w.rec_bytes + w.sell_bytes;
    const size_t cap = g->smem_optin;
    if (graph_b + 4 * warp_b > cap) return;
    // Chains that fit the device at once get one round with as few warps per SM as that takes; larger
    // populations the shape with the smallest rounds * (warps + 10): a round is a chain's latency and the SM's work.
    const int sm = g->sm_count, most = (int)std::min<size_t>(moc::kWalkThreads / 32, (cap - graph_b) / warp_b);
    int best = 0;
    int64_t best_cost = 0;
    for (int k = most; k >= 1; --k) {
        const int64_t rounds = ((int64_t)s->P + (int64_t)sm * k - 1) / ((int64_t)sm * k);
        const int64_t cost = rounds * (k + 10);
        if (best == 0 || cost < best_cost) { best = k; best_cost = cost; }
    }
    // the neighbours' lists where they fit beside that many warps (10 generations, with / without: 64-bit sums, n = 510, 16000 chains x 32 809 / 878 us, n = 600,
    // 8000 x 1 135 / 145, n = 430 x 32 the same; 32-bit sums, n = 620, 8000 x 1 102 / 110); behind them, where they fit too, the output sizes for the one
    // variant that reads them from there (32-bit sums, bound on the new peak).  Copied and counted for all, their 4 n bytes displaced lists.
    w.n_edges = (int32_t)g->n_edges;
    const size_t used = graph_b + (size_t)best * warp_b;
    const bool lists = g->d_near != nullptr && used + g->near_bytes <= cap;
    s->walk_sizes = lists && !wide && used + g->near_size_bytes <= cap;
    w.lists = g->d_near;
    s->walk_wide = wide;
    s->walk_lists = lists;
    s->walk_wpb = best;
    s->walk_grid = (int)std::min<int64_t>(sm, ((int64_t)s->P + best - 1) / best);
    s->walk_smem = used + (lists ? g->near_bytes : 0);
    s->walk_smem_floor = s->walk_sizes ? used + g->near_size_bytes : s->walk_smem;
    s->walk_fits = true;
}

// Whether the generations from `generation` on are tested with a bound on the new peak: where enough evaluations fall away for what it costs, with many
// proposals of a generation or expensive evaluations.  Time of 10 generations with / without it, of that of the kernel before there was one (geometric mean over layered, training and
// convolutional graphs, 203 to 24576 chains, both sums, call after 0 to 440 generations): 8 proposals, n = 30 0.90 / 0.96, n = 60 0.95 / 0.96, n = 92 0.85 / 0.96,
// n = 200 0.80 / 0.97, n = 442 0.81 / 0.97; n > 256: 5 proposals 0.88 / 0.97, 3 0.94 / 0.97.  With one proposal, n > 256: 1.04 / 0.97 in the first
// 500 generations, 1.00 / 0.96 behind 1000 and 2000, 0.92 / 0.97 behind 10000, when few proposals gain anything and the bound refuses the others (n = 442, 4096 chains
// x 20, behind 100000: 31.0 us, 37.8 before).  n <= 256: 2 proposals 1.00 / 0.95, 5 at n = 60 0.98 / 0.96.
// Two proposals: 1.00 / 0.96 in the first 500 generations (64-bit sums, a layered graph, n = 442, 24576 chains 1.05), 0.93 / 0.97 behind 1000, 0.83 / 0.97 behind 10000 at n = 442.
bool walk_floor(const moc_search* s, uint32_t generation) {
    const uint32_t settled = s->samples == 1 ? 4096u : s->samples == 2 ? 1024u : 0u;
    return s->samples >= 8 || (s->g->n_tiles > 4 && generation >= settled);
}

// The variant to launch, prepared when it is first asked for: preparing loads it.  Null: it cannot be.
const void* walk_variant(moc_search* s, bool floor) {
    if (!s->walk_fits) return nullptr;
    if (!s->walk_fn[floor]) {
        const void* f = floor ? walk_floor_fn(s->walk_wide, s->walk_lists) : walk_fn(s->walk_wide, s->walk_lists);
        if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)s->g->smem_optin) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        s->walk_fn[floor] = f;
    }
    return s->walk_fn[floor];
}

// Proposals per chain of one launch: enough that the launch does not show, few enough for a caller who waits.
constexpr int32_t kWalkProposals = 4096;

}  // namespace

extern "C" {

int moc_search_create(const moc_graph* g, const int32_t* seqs, const int32_t* lens, int32_t P, int64_t M,
                      uint64_t seed, uint32_t first_chain, void* stream, moc_search** out) {
    clear_error();
    launch_counter() = 0;
    if (out) *out = nullptr;
    if (!g || !out || !seqs || !lens || P < 1) return fail(MOC_ERR_ARG, "moc_search_create: null pointer or P < 1");
    if (reinterpret_cast<uintptr_t>(seqs) & 3) return fail(MOC_ERR_ARG, "moc_search_create: seqs not 4-byte aligned");
    const int64_t max_T = (int64_t)g->C * g->n;
    const int64_t stride = (max_T + 3) & ~int64_t(3);
    if ((uint64_t)first_chain + (uint64_t)P > 0x100000000ull)
        return fail(MOC_ERR_ARG, "moc_search_create: first_chain + P exceeds 2^32");
    if (2 * (int64_t)P * stride > ((int64_t)1 << 40)) return fail(MOC_ERR_ARG, "moc_search_create: population too large");
    DeviceGuard dg(g->device);
    if (!dg.ok) return fail(MOC_ERR_CUDA, "cannot select device %d", g->device);
    cudaStream_t st = (cudaStream_t)stream;
    moc_search* s = new (std::nothrow) moc_search();
    if (!s) return fail(MOC_ERR_NOMEM, "host allocation failed");
    s->g = g;
    s->device = g->device;
    s->P = P;
    s->stride = (int32_t)stride;
    s->M = M;
    s->seed = seed;
    s->graph_generation = g->generation;
    const size_t bP = (size_t)P;
    const size_t o_rows = 0, o_offs = o_rows + up256(2 * bP * (size_t)stride * 4), o_peak = o_offs + up256((bP + 1) * 8),
                 o_dur = o_peak + up256(bP * 8), o_cpeak = o_dur + up256(bP * 8), o_cdur = o_cpeak + up256(bP * 8),
                 o_cur = o_cdur + up256(bP * 8), o_lens = o_cur + up256(bP * 4), o_st = o_lens + up256(bP * 4),
                 o_acc = o_st + up256(bP * 4), o_clens = o_acc + up256(bP * 4), o_cst = o_clens + up256(bP * 4),
                 o_bad = o_cst + up256(bP * 4), o_at = o_bad + 256, total = o_at + up256(bP * 4);
    cudaError_t e = cudaMalloc((void**)&s->d_block, total);
    if (e != cudaSuccess) {
        delete s;
        cudaGetLastError();
        return fail(e == cudaErrorMemoryAllocation ? MOC_ERR_NOMEM : MOC_ERR_CUDA, "moc_search_create: %s", cudaGetErrorString(e));
    }
    char* b = s->d_block;
    moc::SearchParams& p = s->p;
    p.P = P;
    p.stride = (int32_t)stride;
    p.max_T = (int32_t)max_T;
    p.M = M;
    p.seed_lo = (uint32_t)(seed & 0xFFFFFFFFu);
    p.seed_hi = (uint32_t)(seed >> 32);
    p.generation = 0;
    p.chain0 = first_chain;
    p.kinds = 7u;
    p.rows = (int32_t*)(b + o_rows);
    p.c_offs = (int64_t*)(b + o_offs);
    p.peak = (int64_t*)(b + o_peak);
    p.dur = (int64_t*)(b + o_dur);
    p.c_peak = (int64_t*)(b + o_cpeak);
    p.c_dur = (int64_t*)(b + o_cdur);
    p.cur = (int32_t*)(b + o_cur);
    p.lens = (int32_t*)(b + o_lens);
    p.status = (int32_t*)(b + o_st);
    p.n_acc = (int32_t*)(b + o_acc);
    p.c_lens = (int32_t*)(b + o_clens);
    p.c_status = (int32_t*)(b + o_cst);
    s->d_bad = (int32_t*)(b + o_bad);
    s->wp.peak_at = (int32_t*)(b + o_at);
    int rc = MOC_OK;
    int32_t bad = 0;
    auto run = [&]() -> int {
        MOC_CUDA(cudaMemsetAsync(s->d_bad, 0, 256 + bP * 4, st));      // with the peaks' places behind it: not known
        // packed offsets of the caller's sequences, then the rows, then their evaluation
        moc::offsets_kernel<<<(P + moc::kOffsTile - 1) / moc::kOffsTile, moc::kOffsThreads, 0, st>>>(lens, P, p.c_offs);
        moc::search_init_kernel<<<chain_blocks(P), moc::kSearchThreads, 0, st>>>(p, seqs, lens, p.c_offs, s->d_bad);
        moc::search_offsets_kernel<<<(P + 255) / 256, 256, 0, st>>>(p);
        MOC_CUDA(cudaGetLastError());
        int r = eval_rows(g, p.c_offs, p.rows, p.lens, P, M, p.peak, p.dur, p.status, st);
        if (r != MOC_OK) return r;
        MOC_CUDA(cudaMemcpyAsync(&bad, s->d_bad, 4, cudaMemcpyDeviceToHost, st));
        MOC_CUDA(cudaStreamSynchronize(st));
        return MOC_OK;
    };
    rc = run();
    if (rc == MOC_OK && bad)
        rc = fail(MOC_ERR_ARG, "moc_search_create: a sequence length lies outside [0, C*n = %lld]", (long long)max_T);
    if (rc != MOC_OK) {
        cudaFree(s->d_block);
        delete s;
        return rc;
    }
    *out = s;
    return MOC_OK;
}

int moc_search_run(moc_search* s, int32_t n_generations, void* stream) {
    clear_error();
    launch_counter() = 0;
    if (!s || n_generations < 0) return fail(MOC_ERR_ARG, "moc_search_run: null handle or negative count");
    if ((uint64_t)s->generation + (uint64_t)n_generations > 0xFFFFFFFFull)
        return fail(MOC_ERR_ARG, "moc_search_run: generation counter would pass 2^32 - 1");
    if (n_generations == 0) return MOC_OK;
    DeviceGuard dg(s->device);
    if (!dg.ok) return fail(MOC_ERR_CUDA, "cannot select device %d", s->device);
    cudaStream_t st = (cudaStream_t)stream;
    moc::SearchParams& p = s->p;
    const int blocks = chain_blocks(s->P);
    int launches = 0;
    // The walk kernel relies on the chains' evaluations: not after a change of the graph's C or caps, and without
    // samples not when the caller chose another evaluation kernel for the graph.
    const moc_graph* g = s->g;
    if (s->walk_scores && g->generation != s->graph_generation)
        return fail(MOC_ERR_ARG, "moc_search_run: the graph's C or node caps changed after the search's chains were evaluated");
    if (!s->walk_planned) plan_walk(s);
    if (s->incremental ? s->walk_scores
                       : s->walk_fits && g->generation == s->graph_generation && g->want_G == 0 &&
                             (g->want_kind == MOC_KERNEL_AUTO || g->want_kind == MOC_KERNEL_WARP) && walk_variant(s, walk_floor(s, s->generation))) {
        moc::WalkParams& w = s->wp;
        w.samples = s->samples;
        w.lanes_per_gen = 1;
        while (w.lanes_per_gen < std::min(s->samples, 32)) w.lanes_per_gen *= 2;
        w.cap = g->d_cap;
        const int32_t most = std::max(1, kWalkProposals / s->samples);
        // the variants of the first and of the last launch, before either
        const int32_t last = n_generations > 0 ? (n_generations - 1) / most * most : 0;
        if (!walk_variant(s, walk_floor(s, s->generation)) || !walk_variant(s, walk_floor(s, s->generation + (uint32_t)last)))
            return fail(MOC_ERR_CUDA, "moc_search_run: the search kernel cannot be prepared");
        for (int32_t k = 0; k < n_generations; k += most) {
            w.s = p;
            w.s.generation = s->generation + (uint32_t)k;
            w.n_gen = std::min(most, n_generations - k);
            const bool floor = walk_floor(s, w.s.generation);
            w.sizes = floor && s->walk_sizes;
            w.list_bytes = (uint32_t)(w.sizes ? g->near_size_bytes : g->near_bytes);
            void* args[] = {&w};
            MOC_CUDA(cudaLaunchKernel(s->walk_fn[floor], dim3(s->walk_grid), dim3(32 * s->walk_wpb), args, floor ? s->walk_smem_floor : s->walk_smem, st));
            ++launches;
        }
        s->generation += (uint32_t)n_generations;
        launch_counter() = launches;
        return MOC_OK;
    }
    MOC_CUDA(cudaMemsetAsync(s->wp.peak_at, 0, (size_t)s->P * 4, st));       // the kernels below do not keep it
    if (s->incremental && s->fused) {
        moc_cache* h = s->cache;
        if (h->graph_generation != h->g->generation)
            return fail(MOC_ERR_ARG, "moc_search_run: the graph's C or node caps changed after the search's cache was built");
        const int wpb = s->score_wpb;
        const int grid = (int)std::min<int64_t>(s->score_grid_cap, ((int64_t)s->P + wpb - 1) / wpb);
        for (int32_t k = 0; k < n_generations; ++k) {
            p.generation = s->generation + (uint32_t)k;
            s->sp.s = p;
            s->sp.c = h->c;
            s->sp.c.cap = h->g->d_cap;
            void* args[] = {&s->sp};
            MOC_CUDA(cudaLaunchKernel(s->score_fn, dim3(grid), dim3(32 * wpb), args, s->score_smem, st));
            int rc = cache_prepare(h, p.rows, p.lens, s->ip.row_offs, s->P, s->ip.todo, s->ip.todo_count + (p.generation & 1u),
                                   s->M, nullptr, nullptr, nullptr, st);
            if (rc != MOC_OK) return rc;
            launches += 2;
        }
        MOC_CUDA(cudaGetLastError());
        s->generation += (uint32_t)n_generations;
        launch_counter() = launches;
        return MOC_OK;
    }
    if (s->incremental) {
        const int64_t nE = (int64_t)s->P * s->samples;
        for (int32_t k = 0; k < n_generations; ++k) {
            p.generation = s->generation + (uint32_t)k;
            s->ip.s = p;
            moc::search_draw_kernel<<<(unsigned)((nE + 255) / 256), 256, 0, st>>>(s->ip);
            int rc = moc_eval_edits(s->cache, s->ip.e_parent, s->ip.e_op, s->ip.e_q, s->ip.e_j, (int32_t)nE, s->M,
                                    s->ip.r_peak, s->ip.r_dur, s->ip.r_status, nullptr, stream);
            if (rc != MOC_OK) return rc;
            moc::search_pick_kernel<<<blocks, moc::kSearchThreads, 0, st>>>(s->ip);
            rc = cache_prepare(s->cache, p.rows, p.lens, s->ip.row_offs, s->P, s->ip.todo, s->ip.todo_count, s->M,
                               nullptr, nullptr, nullptr, st);
            if (rc != MOC_OK) return rc;
            launches += 4;
        }
        MOC_CUDA(cudaGetLastError());
        s->generation += (uint32_t)n_generations;
        launch_counter() = launches;
        return MOC_OK;
    }
    for (int32_t k = 0; k < n_generations; ++k) {
        p.generation = s->generation + (uint32_t)k;
        // settle the previous generation's proposals (none before the first one), propose the next
        if (k == 0) moc::search_step_kernel<false, true><<<blocks, moc::kSearchThreads, 0, st>>>(p);
        else moc::search_step_kernel<true, true><<<blocks, moc::kSearchThreads, 0, st>>>(p);
        ++launches;
        int rc = eval_rows(s->g, p.c_offs, p.rows, p.c_lens, s->P, s->M, p.c_peak, p.c_dur, p.c_status, st);
        launches += launch_counter();
        launch_counter() = 0;
        if (rc != MOC_OK) return rc;
    }
    moc::search_step_kernel<true, false><<<blocks, moc::kSearchThreads, 0, st>>>(p);
    ++launches;
    MOC_CUDA(cudaGetLastError());
    s->generation += (uint32_t)n_generations;
    launch_counter() = launches;
    return MOC_OK;
}

int moc_search_set_kinds(moc_search* s, uint32_t kinds) {
    clear_error();
    if (!s || kinds == 0 || kinds > 7u) return fail(MOC_ERR_ARG, "moc_search_set_kinds: null handle or mask outside 1..7");
    s->p.kinds = kinds;
    return MOC_OK;
}

int moc_search_set_samples(moc_search* s, int32_t samples, int32_t incremental) {
    clear_error();
    if (!s || samples < 1 || samples > 4096 || incremental < 0 || incremental > 3)
        return fail(MOC_ERR_ARG, "moc_search_set_samples: null handle, samples outside [1, 4096] or mode outside 0..3");
    if (samples > 1 && !incremental)
        return fail(MOC_ERR_ARG, "moc_search_set_samples: more than one proposal per chain needs the incremental evaluation");
    if ((int64_t)s->P * samples > INT32_MAX) return fail(MOC_ERR_ARG, "moc_search_set_samples: P * samples exceeds 2^31 - 1");
    DeviceGuard dg(s->device);
    if (!dg.ok) return fail(MOC_ERR_CUDA, "cannot select device %d", s->device);
    MOC_CUDA(cudaDeviceSynchronize());          // generations in flight still use the old buffers
    if (!incremental) {
        s->incremental = false;
        s->fused = false;
        s->walk_scores = false;
        s->samples = 1;
        return MOC_OK;
    }
    // every chain needs a valid evaluation to start from
    std::vector<int32_t> st;
    try {
        st.resize((size_t)s->P);
    } catch (const std::bad_alloc&) {
        return fail(MOC_ERR_NOMEM, "host allocation failed");
    }
    MOC_CUDA(cudaMemcpy(st.data(), s->p.status, (size_t)s->P * 4, cudaMemcpyDeviceToHost));
    for (int32_t c = 0; c < s->P; ++c)
        if (st[c] < 0)
            return fail(MOC_ERR_ARG, "moc_search_set_samples: chain %d has no valid sequence (status %d); the incremental "
                        "evaluation starts from valid sequences only", c, st[c]);
    // by default the kernel that takes a warp per chain through all generations (no cache), where the graph fits it
    if (!s->walk_planned) plan_walk(s);
    s->walk_scores = false;
    if (incremental == MOC_SEARCH_SCORE_AUTO && s->walk_fits && s->g->generation == s->graph_generation) {
        const int32_t before = s->samples;
        s->samples = samples;
        if (walk_variant(s, walk_floor(s, s->generation))) {
            s->walk_scores = true;
            s->incremental = true;
            return MOC_OK;
        }
        s->samples = before;
    }
    if (!s->cache) {
        moc_cache* h = nullptr;
        int rc = moc_cache_create(s->g, s->P, &h);
        if (rc != MOC_OK) return rc;
        s->cache = h;
    }
    const size_t nE = (size_t)s->P * samples, bP = (size_t)s->P;
    const size_t o_par = 0, o_op = o_par + up256(nE * 4), o_q = o_op + up256(nE * 4), o_j = o_q + up256(nE * 4),
                 o_st = o_j + up256(nE * 4), o_pk = o_st + up256(nE * 4), o_du = o_pk + up256(nE * 8),
                 o_offs = o_du + up256(nE * 8), o_todo = o_offs + up256((bP + 1) * 8), o_cnt = o_todo + up256(bP * 4),
                 total = o_cnt + 256;          // o_cnt: two counters, used in turn by the warp-per-chain kernel
    if (s->d_inc) MOC_CUDA(cudaFree(s->d_inc));
    s->d_inc = nullptr;
    s->incremental = false;
    cudaError_t e = cudaMalloc((void**)&s->d_inc, total);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(e == cudaErrorMemoryAllocation ? MOC_ERR_NOMEM : MOC_ERR_CUDA, "moc_search_set_samples: %s", cudaGetErrorString(e));
    }
    char* b = s->d_inc;
    moc::SearchIncParams& ip = s->ip;
    ip.s = s->p;
    ip.samples = samples;
    ip.e_parent = (int32_t*)(b + o_par);
    ip.e_op = (int32_t*)(b + o_op);
    ip.e_q = (int32_t*)(b + o_q);
    ip.e_j = (int32_t*)(b + o_j);
    ip.r_status = (int32_t*)(b + o_st);
    ip.r_peak = (int64_t*)(b + o_pk);
    ip.r_dur = (int64_t*)(b + o_du);
    ip.row_offs = (int64_t*)(b + o_offs);
    ip.todo = (int32_t*)(b + o_todo);
    ip.todo_count = (int32_t*)(b + o_cnt);
    MOC_CUDA(cudaMemset(ip.todo_count, 0, 8));
    // scoring kernel: a warp per chain when asked for, or by default from 24 proposals per chain on
    // (below that the lane-per-edit kernel of moc_eval_edits, with more warps per SM, is as fast or faster)
    s->fused = false;
    if (incremental == MOC_SEARCH_SCORE_CHAIN || (incremental == MOC_SEARCH_SCORE_AUTO && samples >= 24)) {
        s->fused = plan_fused(s);
        if (!s->fused && incremental == MOC_SEARCH_SCORE_CHAIN) {
            cudaFree(s->d_inc);
            s->d_inc = nullptr;
            return fail(MOC_ERR_ARG, "moc_search_set_samples: the warp-per-chain kernel cannot hold this graph's rows and "
                        "correction lists (n = %d, largest in-degree %d) in shared memory", s->g->n, s->g->max_indeg);
        }
    }
    s->sp.samples = samples;
    s->sp.row_offs = ip.row_offs;
    s->sp.todo = ip.todo;
    s->sp.todo_count = ip.todo_count;
    // cache of all chains from their current rows
    moc::search_row_offsets_kernel<<<(s->P + 255) / 256, 256>>>(ip);
    int rc = cache_prepare(s->cache, s->p.rows, s->p.lens, ip.row_offs, s->P, nullptr, nullptr, s->M, nullptr, nullptr, nullptr, nullptr);
    if (rc != MOC_OK) return rc;
    MOC_CUDA(cudaDeviceSynchronize());
    s->samples = samples;
    s->incremental = true;
    return MOC_OK;
}

static int export_state(const moc_search* s, int32_t* out_rows, bool fill, int32_t* out_lens, int64_t* out_peak, int64_t* out_dur,
                        int32_t* out_status, int32_t* out_accepted, void* stream) {
    clear_error();
    if (!s) return fail(MOC_ERR_ARG, "moc_search_state: null handle");
    DeviceGuard dg(s->device);
    if (!dg.ok) return fail(MOC_ERR_CUDA, "cannot select device %d", s->device);
    moc::search_export_kernel<<<chain_blocks(s->P), moc::kSearchThreads, 0, (cudaStream_t)stream>>>(
        s->p, out_rows, fill, out_lens, out_peak, out_dur, out_status, out_accepted);
    MOC_CUDA(cudaGetLastError());
    return MOC_OK;
}

int moc_search_state(const moc_search* s, int32_t* out_rows, int32_t* out_lens, int64_t* out_peak,
                     int64_t* out_dur, int32_t* out_status, int32_t* out_accepted, void* stream) {
    return export_state(s, out_rows, false, out_lens, out_peak, out_dur, out_status, out_accepted, stream);
}

// For the torch side of the binding: the whole of out_rows is written, zeros behind the sequences.
int moc_search_state_filled(const moc_search* s, int32_t* out_rows, int32_t* out_lens, int64_t* out_peak,
                            int64_t* out_dur, int32_t* out_status, int32_t* out_accepted, void* stream) {
    return export_state(s, out_rows, true, out_lens, out_peak, out_dur, out_status, out_accepted, stream);
}

int moc_search_best(const moc_search* s, int32_t* out_seq, int64_t* out_best, void* stream) {
    clear_error();
    if (!s || !out_best) return fail(MOC_ERR_ARG, "moc_search_best: null handle or null out_best");
    DeviceGuard dg(s->device);
    if (!dg.ok) return fail(MOC_ERR_CUDA, "cannot select device %d", s->device);
    moc::search_best_kernel<<<1, moc::kBestThreads, 0, (cudaStream_t)stream>>>(s->p, out_seq, out_best);
    MOC_CUDA(cudaGetLastError());
    return MOC_OK;
}

int moc_search_info(const moc_search* s, int32_t* P, int32_t* stride, uint32_t* generation) {
    clear_error();
    if (!s) return fail(MOC_ERR_ARG, "moc_search_info: null handle");
    if (P) *P = s->P;
    if (stride) *stride = s->stride;
    if (generation) *generation = s->generation;
    return MOC_OK;
}

void moc_search_destroy(moc_search* s) {
    if (!s) return;
    DeviceGuard dg(s->device);
    moc_cache_destroy(s->cache);
    cudaFree(s->d_inc);
    cudaFree(s->d_block);
    delete s;
}

}  // extern "C"
