// All generations of a search call with a warp per chain.
#include "moc_host.cuh"
#include "moc_search_walk_kernel.cuh"

namespace moc_host {
const void* walk_fn(bool wide, bool lists) {
    if (lists) return wide ? (const void*)moc::search_walk_kernel<int64_t, true, false> : (const void*)moc::search_walk_kernel<int32_t, true, false>;
    return wide ? (const void*)moc::search_walk_kernel<int64_t, false, false> : (const void*)moc::search_walk_kernel<int32_t, false, false>;
}
}  // namespace moc_host
