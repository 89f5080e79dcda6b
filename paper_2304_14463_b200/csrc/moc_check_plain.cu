// Interval checker for the plain domain with two slots per node.
#include "moc_host.cuh"
#include "moc_interval_plain_kernel.cuh"

namespace moc_host {
const void* check_plain_fn(bool wide) { return wide ? (const void*)moc::check_plain_kernel<int64_t> : (const void*)moc::check_plain_kernel<int32_t>; }
}  // namespace moc_host
