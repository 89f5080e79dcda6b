// Interval checker, plain domain: what the kernel for two slots per node does not serve.
#include "moc_host.cuh"
#include "moc_interval_kernels.cuh"

namespace moc_host {
namespace {
template <int CP, typename MemT>
IntervalFn kept_fn(int kept) {
    switch (kept) {
        case 0: return moc::check_intervals_kernel<true, CP, MemT, false, int32_t>;
        case 2: return moc::check_intervals_kernel<true, CP, MemT, true, uint16_t>;
        default: return moc::check_intervals_kernel<true, CP, MemT, true, int32_t>;
    }
}
template <int CP>
IntervalFn wide_fn(bool wide, int kept) {
    return wide ? kept_fn<CP, int64_t>(kept) : kept_fn<CP, int32_t>(kept);
}
}  // namespace

IntervalFn check_general_fn(int cp, bool wide, int kept) {
    return cp == 2 ? wide_fn<2>(wide, kept) : (cp == 4 ? wide_fn<4>(wide, kept) : wide_fn<8>(wide, kept));
}
}  // namespace moc_host
