// Warp-per-sequence kernel (C <= 2).
#include "moc_host.cuh"

namespace moc_host {
namespace {
template <typename MemT>
PairFn pair_fn_t(int pre) {
    switch (pre) {
        case 0: return (PairFn)moc::eval_pair_kernel<MemT, 0>;
        case 1: return (PairFn)moc::eval_pair_kernel<MemT, 1>;
        case 2: return (PairFn)moc::eval_pair_kernel<MemT, 2>;
        case 3: return (PairFn)moc::eval_pair_kernel<MemT, 3>;
        case 4: return (PairFn)moc::eval_pair_kernel<MemT, 4>;
        default: return (PairFn)moc::eval_pair_kernel<MemT, 5>;
    }
}
}  // namespace

PairFn pair_fn(bool wide, int pre) { return wide ? pair_fn_t<int64_t>(pre) : pair_fn_t<int32_t>(pre); }
}  // namespace moc_host
