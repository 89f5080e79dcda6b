// Warp-per-sequence kernel (C <= 2).
#include "moc_host.cuh"

namespace moc_host {
namespace {
template <typename MemT>
PairFn pair_fn_t(int pre) {
    if (pre < 0) return (PairFn)moc::eval_pair_kernel<MemT, 0, true>;
    switch (pre) {
        case 0: return (PairFn)moc::eval_pair_kernel<MemT, 0, false>;
        case 1: return (PairFn)moc::eval_pair_kernel<MemT, 1, false>;
        case 2: return (PairFn)moc::eval_pair_kernel<MemT, 2, false>;
        case 3: return (PairFn)moc::eval_pair_kernel<MemT, 3, false>;
        case 4: return (PairFn)moc::eval_pair_kernel<MemT, 4, false>;
        default: return (PairFn)moc::eval_pair_kernel<MemT, 5, false>;
    }
}
}  // namespace

PairFn pair_fn(bool wide, int pre) { return wide ? pair_fn_t<int64_t>(pre) : pair_fn_t<int32_t>(pre); }
}  // namespace moc_host
