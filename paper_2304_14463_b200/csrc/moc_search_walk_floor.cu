// All generations of a search call with a warp per chain and a bound on the new peak, in a module of its own: a search that does not use the
// bound does not load it (first run of a process with both in one module 1.1 ms instead of 0.7).
#include "moc_host.cuh"
#include "moc_search_walk_kernel.cuh"

namespace moc_host {
const void* walk_floor_fn(bool wide, bool lists) {
    if (lists) return wide ? (const void*)moc::search_walk_floor_kernel<int64_t, true> : (const void*)moc::search_walk_floor_kernel<int32_t, true>;
    return wide ? (const void*)moc::search_walk_floor_kernel<int64_t, false> : (const void*)moc::search_walk_floor_kernel<int32_t, false>;
}
}  // namespace moc_host
