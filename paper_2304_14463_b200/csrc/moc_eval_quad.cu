// Block-per-sequence kernel (C <= 4).
#include "moc_host.cuh"

namespace moc_host {
namespace {
template <typename MemT, bool kTiles>
QuadFn quad_fn_c(int C, bool profile) {
    if (profile) return C <= 3 ? (QuadFn)moc::eval_quad_kernel<MemT, 3, kTiles, true> : (QuadFn)moc::eval_quad_kernel<MemT, 4, kTiles, true>;
    return C <= 3 ? (QuadFn)moc::eval_quad_kernel<MemT, 3, kTiles, false> : (QuadFn)moc::eval_quad_kernel<MemT, 4, kTiles, false>;
}
}  // namespace

QuadFn quad_fn(bool wide, int C, bool tiles, bool profile) {
    if (tiles) return wide ? quad_fn_c<int64_t, true>(C, profile) : quad_fn_c<int32_t, true>(C, profile);
    return wide ? quad_fn_c<int64_t, false>(C, profile) : quad_fn_c<int32_t, false>(C, profile);
}
}  // namespace moc_host
