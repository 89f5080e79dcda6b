// Block-per-sequence kernel (C <= 4).
#include "moc_host.cuh"

namespace moc_host {
namespace {
template <typename MemT, bool kTiles, bool kChip>
QuadFn quad_fn_c(int C, bool profile) {
    if (profile) return C <= 3 ? (QuadFn)moc::eval_quad_kernel<MemT, 3, kTiles, true, kChip> : (QuadFn)moc::eval_quad_kernel<MemT, 4, kTiles, true, kChip>;
    if (C <= 2) return (QuadFn)moc::eval_quad_kernel<MemT, 2, kTiles, false, kChip>;
    return C == 3 ? (QuadFn)moc::eval_quad_kernel<MemT, 3, kTiles, false, kChip> : (QuadFn)moc::eval_quad_kernel<MemT, 4, kTiles, false, kChip>;
}
}  // namespace

QuadFn quad_fn(bool wide, int C, bool tiles, bool chip, bool profile) {
    if (tiles && chip) return wide ? quad_fn_c<int64_t, true, true>(C, profile) : quad_fn_c<int32_t, true, true>(C, profile);
    if (tiles) return wide ? quad_fn_c<int64_t, true, false>(C, profile) : quad_fn_c<int32_t, true, false>(C, profile);
    return wide ? quad_fn_c<int64_t, false, false>(C, profile) : quad_fn_c<int32_t, false, false>(C, profile);
}
}  // namespace moc_host
