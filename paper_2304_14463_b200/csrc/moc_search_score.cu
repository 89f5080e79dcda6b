// Search generation with a warp per chain on the cached evaluation.
#include "moc_host.cuh"
#include "moc_search_score_kernel.cuh"

namespace moc_host {
const void* score_fn(bool wide, bool graph_on_chip) {
    if (graph_on_chip) return wide ? (const void*)moc::search_score_kernel<int64_t, true> : (const void*)moc::search_score_kernel<int32_t, true>;
    return wide ? (const void*)moc::search_score_kernel<int64_t, false> : (const void*)moc::search_score_kernel<int32_t, false>;
}
}  // namespace moc_host
