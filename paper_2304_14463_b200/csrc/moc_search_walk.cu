// All generations of a search call with a warp per chain.
#include "moc_host.cuh"
#include "moc_search_walk_kernel.cuh"

namespace moc_host {
template <typename MemT>
static const void* of(bool lists, bool floor) {
    if (lists) return floor ? (const void*)moc::search_walk_kernel<MemT, true, true> : (const void*)moc::search_walk_kernel<MemT, true, false>;
    return floor ? (const void*)moc::search_walk_kernel<MemT, false, true> : (const void*)moc::search_walk_kernel<MemT, false, false>;
}
const void* walk_fn(bool wide, bool lists, bool floor) { return wide ? of<int64_t>(lists, floor) : of<int32_t>(lists, floor); }
}  // namespace moc_host
