// Host side of moc_check_intervals (declared in include/moc.h): argument checks and the launch.
#include <algorithm>

#include "moc_host.cuh"
#include "moc_interval_kernels.cuh"
#include "moc_interval_plain_kernel.cuh"

using namespace moc_host;

namespace {

// Launch of the kernel for the plain domain with two slots per node; false when the case is not its own.
bool launch_plain(const moc_graph* g, const moc::IntervalParams& q, bool fill, cudaStream_t st, cudaError_t* err) {
    const bool wide = g->sum_m > (int64_t)INT32_MAX / g->C;
    if (q.topo_index || g->C != 2 || q.D > 32766 || !g->d_rec32 || (wide && !g->split_ok)) return false;
    if ((reinterpret_cast<uintptr_t>(q.s) | reinterpret_cast<uintptr_t>(q.e) | reinterpret_cast<uintptr_t>(q.a)) & 7) return false;
    moc::IntervalPlainParams p{};
    p.q = q;
    p.n_tiles = g->n_tiles;
    p.split = g->split;
    p.rec = wide ? g->d_rec64 : g->d_rec32;
    p.sell = g->d_sell_iv;
    p.rec_bytes = (wide ? 16u : 8u) * 64u * (uint32_t)g->n_tiles;
    p.sell_bytes = (4u * (uint32_t)g->sell_len + 15u) & ~15u;
    p.word_bytes = (4u * ((uint32_t)g->n + 2u) + 15u) & ~15u;
    p.event_bytes = (uint32_t)moc::interval_plain_event_bytes(q.D, wide ? 8 : 4);
    p.fill = fill;
    const size_t warp_b = 2 * ((size_t)p.word_bytes + moc::kPairWordTail) + p.event_bytes, graph_b = (size_t)p.rec_bytes + p.sell_bytes;
    if (graph_b + 4 * warp_b > g->smem_optin) return false;
    const void* fn = check_plain_fn(wide);
    *err = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g->smem_optin);
    if (*err != cudaSuccess) return true;
    // one block per SM; warps: the rounds a full block needs, evenly filled, at least eight to stage the graph
    const int most = (int)std::min<size_t>(moc::kIvPlainThreads / 32, (g->smem_optin - graph_b) / warp_b);
    const int64_t per_sm = ((int64_t)q.B + g->sm_count - 1) / g->sm_count, rounds = (per_sm + most - 1) / most;
    const int wpb = (int)std::min<int64_t>(most, std::max<int64_t>(8, (per_sm + rounds - 1) / rounds));
    const int grid = (int)std::min<int64_t>(g->sm_count, q.B);
    void* args[] = {&p};
    *err = cudaLaunchKernel(fn, dim3(grid), dim3(32 * wpb), args, graph_b + (size_t)wpb * warp_b, st);
    return true;
}

int check_intervals(const moc_graph* g, const int32_t* s, const int32_t* e, const int32_t* a, int32_t B, int64_t D,
                    const int32_t* topo_index, int64_t M, int64_t* out_peak, int64_t* out_dur, int32_t* out_mask, int32_t* out_seqs,
                    int32_t* out_lens, bool fill, void* stream) {
    clear_error();
    launch_counter() = 0;
    if (!g || B < 0) return fail(MOC_ERR_ARG, "moc_check_intervals: null handle or B < 0");
    if (B == 0) return MOC_OK;
    if (!s || !e || !a || !out_peak || !out_dur || !out_mask)
        return fail(MOC_ERR_ARG, "moc_check_intervals: null array");
    if (D < 1 || D > ((int64_t)1 << 30)) return fail(MOC_ERR_ARG, "moc_check_intervals: D outside [1, 2^30]");
    if (g->C > moc::kIvMaxC) return fail(MOC_ERR_ARG, "moc_check_intervals: C > %d", moc::kIvMaxC);
    const int64_t n = g->n, K = n * g->C;
    if (topo_index && D != n * (n + 1) / 2)
        return fail(MOC_ERR_ARG, "moc_check_intervals: the staged model needs D = n(n+1)/2 = %lld", (long long)(n * (n + 1) / 2));
    DeviceGuard dg(g->device);
    if (!dg.ok) return fail(MOC_ERR_CUDA, "cannot select device %d", g->device);
    moc::IntervalParams p{};
    p.n = g->n;
    p.C = g->C;
    p.succ_start = g->d_succ_start;
    p.succ = g->d_succ;
    p.w = g->d_w;
    p.m = g->d_m64;
    p.s = s;
    p.e = e;
    p.a = a;
    p.B = B;
    p.D = (int32_t)D;
    p.topo_index = topo_index;
    p.M = M;
    p.out_peak = out_peak;
    p.out_dur = out_dur;
    p.out_mask = out_mask;
    p.out_seqs = out_seqs;
    p.out_lens = out_lens;
    cudaError_t err = cudaSuccess;
    if (launch_plain(g, p, fill, (cudaStream_t)stream, &err)) {
        MOC_CUDA(err);
        launch_counter() = 1;
        return MOC_OK;
    }
    p.words = (uint32_t)(((D + 32) / 32 + 3) & ~int64_t(3));
    const bool plain = topo_index == nullptr;
    const bool wide = g->sum_m > (int64_t)INT32_MAX / g->C;     // C * sum(m) bounds every partial usage sum
    const size_t cap = g->smem_optin > 2048 ? g->smem_optin - 2048 : 0;
    const size_t base_b = moc::interval_clear_bytes(p.words, K, plain, wide ? 8 : 4), stage_b = moc::interval_stage_bytes(K, D < 65536 ? 2 : 4);
    if (base_b > cap || K > (int64_t)INT32_MAX / 2)
        return fail(MOC_ERR_ARG, "moc_check_intervals: domain of %lld events with %lld intervals needs %zu bytes of "
                    "shared memory per solution, the device offers %zu", (long long)D, (long long)K, base_b, cap);
    // keep the solution on chip after the first pass while two solutions per SM still fit: reading it again costs more than the
    // warps that its place would hold (staged, 4000 solutions: n = 600 344 -> 323 us, 700 582 -> 442, 1000 1658 -> 1271)
    p.byte_marks = plain && 2 * (((size_t)D + 1 + 15) & ~size_t(15)) <= ((((size_t)K + 2) * (wide ? 8 : 4) + 15) & ~size_t(15)) ? 1 : 0;
    const bool stage = (base_b + stage_b) * 2 <= cap;
    const size_t warp_b = base_b + (stage ? stage_b : 0);
    p.warp_bytes = (uint32_t)warp_b;
    // warps per block: the count that puts most warps on an SM (each block loses 1 KB to the system)
    int wpb = 1, best = 0;
    for (int k = 1; k <= moc::kIvMaxWarps; ++k) {
        const size_t blk = warp_b * k + 1024;
        const int fit = blk <= cap + 1024 ? (int)((g->smem_optin) / blk) * k : 0;
        if (fit > best) { best = fit; wpb = k; }
    }
    // Several warps on a solution where an SM would have few at work (bitmaps of a large domain, or a small batch), as many as leave it some
    // 48 and each 16 nodes.  Staged, 1 / 2 / 4 / 8 / 16 warps (us): n = 111, B = 500 14.8 / 12.3 / 10.6 / 11.0 / 14.7; n = 300, B = 6000 80 / 62 / 68 / 85 / 107;
    // n = 442, B = 1500 77 / 47 / 33 / 33 / 38, B = 148 40 / 24 / 17 / 13 / 11; n = 932, B = 1500 433 / 231 / 136 / 89 / 68.
    const int64_t per_sm = ((int64_t)B + g->sm_count - 1) / g->sm_count, at_work = std::max<int64_t>(1, std::min<int64_t>(best, per_sm));
    int team = 1;
    while (team < moc::kIvMaxTeam && 2 * team * at_work <= 48 && 32 * team <= n) team *= 2;
    p.team = team > 1 ? 1 : 0;
    if (team > 1) wpb = team;
    if (fill && out_seqs) MOC_CUDA(cudaMemsetAsync(out_seqs, 0xFF, (size_t)B * (size_t)K * 4, (cudaStream_t)stream));
    const size_t smem = team > 1 ? warp_b : warp_b * wpb;
    const int cp = g->C <= 2 ? 2 : (g->C <= 4 ? 4 : 8), kept = !stage ? 0 : (D < 65536 ? 2 : 4);      // bytes per kept event
    const IntervalFn fn = plain ? check_general_fn(cp, wide, kept, team > 1) : check_staged_fn(cp, wide, kept, team > 1);
    MOC_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cap));
    int nb = 0;
    MOC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, 32 * wpb, smem));
    if (nb < 1) return fail(MOC_ERR_CUDA, "moc_check_intervals: kernel does not fit on an SM");
    const int grid = (int)std::min<int64_t>((int64_t)g->sm_count * nb, team > 1 ? (int64_t)B : ((int64_t)B + wpb - 1) / wpb);
    fn<<<grid, 32 * wpb, smem, (cudaStream_t)stream>>>(p);
    MOC_CUDA(cudaGetLastError());
    launch_counter() = 1;
    return MOC_OK;
}

}  // namespace

extern "C" int moc_check_intervals(const moc_graph* g, const int32_t* s, const int32_t* e, const int32_t* a, int32_t B, int64_t D,
                                   const int32_t* topo_index, int64_t M, int64_t* out_peak, int64_t* out_dur, int32_t* out_mask,
                                   int32_t* out_seqs, int32_t* out_lens, void* stream) {
    return check_intervals(g, s, e, a, B, D, topo_index, M, out_peak, out_dur, out_mask, out_seqs, out_lens, false, stream);
}

// For the torch side of the binding: the whole of out_seqs is written, -1 behind the sequences.
extern "C" int moc_check_intervals_filled(const moc_graph* g, const int32_t* s, const int32_t* e, const int32_t* a, int32_t B, int64_t D,
                                          const int32_t* topo_index, int64_t M, int64_t* out_peak, int64_t* out_dur, int32_t* out_mask,
                                          int32_t* out_seqs, int32_t* out_lens, void* stream) {
    return check_intervals(g, s, e, a, B, D, topo_index, M, out_peak, out_dur, out_mask, out_seqs, out_lens, true, stream);
}
