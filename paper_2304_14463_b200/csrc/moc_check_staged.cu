// Interval checker, staged domain.
#include "moc_host.cuh"
#include "moc_interval_kernels.cuh"

namespace moc_host {
namespace {
template <int CP, typename MemT, bool kTeams>
IntervalFn kept_fn(int kept) {
    switch (kept) {
        case 0: return moc::check_intervals_kernel<false, CP, MemT, false, int32_t, kTeams>;
        case 2: return moc::check_intervals_kernel<false, CP, MemT, true, uint16_t, kTeams>;
        default: return moc::check_intervals_kernel<false, CP, MemT, true, int32_t, kTeams>;
    }
}
template <int CP, bool kTeams>
IntervalFn wide_fn(bool wide, int kept) {
    return wide ? kept_fn<CP, int64_t, kTeams>(kept) : kept_fn<CP, int32_t, kTeams>(kept);
}
}  // namespace

IntervalFn check_staged_fn(int cp, bool wide, int kept, bool team) {
    if (cp == 2) return team ? wide_fn<2, true>(wide, kept) : wide_fn<2, false>(wide, kept);
    return cp == 4 ? wide_fn<4, true>(wide, kept) : wide_fn<8, true>(wide, kept);      // one variant for both
}
}  // namespace moc_host
