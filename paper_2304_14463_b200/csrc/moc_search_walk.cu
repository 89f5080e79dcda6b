// All generations of a search call with a warp per chain.
#include "moc_host.cuh"
#include "moc_search_walk_kernel.cuh"

namespace moc_host {
const void* walk_fn(bool wide) { return wide ? (const void*)moc::search_walk_kernel<int64_t> : (const void*)moc::search_walk_kernel<int32_t>; }
}  // namespace moc_host
