// All generations of a search call with a warp per chain and a bound on the new peak, in a module of its own: a search that does not use the
// bound does not load it (first run of a process with both in one module 1.1 ms instead of 0.7).  The kernel is the same template, under
// another name: launches and modules tell the two apart by it.
#define search_walk_kernel search_walk_floor_kernel
#include "moc_host.cuh"
#include "moc_search_walk_kernel.cuh"

namespace moc_host {
const void* walk_floor_fn(bool wide, bool lists) {
    if (lists) return wide ? (const void*)moc::search_walk_floor_kernel<int64_t, true, true> : (const void*)moc::search_walk_floor_kernel<int32_t, true, true>;
    return wide ? (const void*)moc::search_walk_floor_kernel<int64_t, false, true> : (const void*)moc::search_walk_floor_kernel<int32_t, false, true>;
}
}  // namespace moc_host
