// Backward walk with a lane per sequence (n <= 128, C <= 4).
#include "moc_host.cuh"

namespace moc_host {
namespace {
template <typename SumT, int W>
LiveFn live_fn_k(int C) {
    return C <= 2 ? (LiveFn)moc::eval_live_kernel<SumT, W, 2> : (LiveFn)moc::eval_live_kernel<SumT, W, 4>;
}
template <typename SumT>
LiveFn live_fn_w(int words, int C) {
    switch (words) {
        case 1: return live_fn_k<SumT, 1>(C);
        case 2: return live_fn_k<SumT, 2>(C);
        default: return live_fn_k<SumT, 4>(C);
    }
}
}  // namespace

LiveFn live_fn(bool wide, int words, int C) { return wide ? live_fn_w<int64_t>(words, C) : live_fn_w<int32_t>(words, C); }
}  // namespace moc_host
