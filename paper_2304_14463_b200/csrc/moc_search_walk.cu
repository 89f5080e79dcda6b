// All generations of a search call with a warp per chain.
#include "moc_host.cuh"
#include "moc_search_walk_kernel.cuh"

namespace moc_host {
const void* walk_fn(bool wide, bool lists) {
    if (lists) return wide ? (const void*)moc::search_walk_kernel<int64_t, true> : (const void*)moc::search_walk_kernel<int32_t, true>;
    return wide ? (const void*)moc::search_walk_kernel<int64_t, false> : (const void*)moc::search_walk_kernel<int32_t, false>;
}
}  // namespace moc_host
