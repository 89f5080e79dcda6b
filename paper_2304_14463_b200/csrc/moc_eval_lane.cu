// Sequence-per-lane kernel (C <= 2).
#include "moc_host.cuh"

namespace moc_host {
namespace {
template <typename MemT, int LG>
LaneFn lane_fn_kp(int kp) {
    switch (kp) {
        case 2: return (LaneFn)moc::eval_lane_kernel<MemT, LG, 2>;
        case 4: return (LaneFn)moc::eval_lane_kernel<MemT, LG, 4>;
        case 6: return (LaneFn)moc::eval_lane_kernel<MemT, LG, 6>;
        default: return (LaneFn)moc::eval_lane_kernel<MemT, LG, 8>;
    }
}
template <typename MemT>
LaneFn lane_fn_lg(int lg, int kp) {
    switch (lg) {
        case 5: return lane_fn_kp<MemT, 5>(kp);
        case 4: return lane_fn_kp<MemT, 4>(kp);
        default: return lane_fn_kp<MemT, 3>(kp);
    }
}
}  // namespace

LaneFn lane_fn(bool wide, int lg, int kp) { return wide ? lane_fn_lg<int64_t>(lg, kp) : lane_fn_lg<int32_t>(lg, kp); }
}  // namespace moc_host
