// Block-per-sequence kernel (C <= 4).
#include "moc_host.cuh"

namespace moc_host {
namespace {
template <typename MemT, bool kTiles, int kMode>
QuadFn quad_fn_c(int C, bool profile) {
    if (profile) return C <= 3 ? (QuadFn)moc::eval_quad_kernel<MemT, 3, kTiles, true, kMode> : (QuadFn)moc::eval_quad_kernel<MemT, 4, kTiles, true, kMode>;
    if (C <= 2) return (QuadFn)moc::eval_quad_kernel<MemT, 2, kTiles, false, kMode>;
    return C == 3 ? (QuadFn)moc::eval_quad_kernel<MemT, 3, kTiles, false, kMode> : (QuadFn)moc::eval_quad_kernel<MemT, 4, kTiles, false, kMode>;
}
}  // namespace

QuadFn quad_fn(bool wide, int C, bool tiles, bool chip, bool profile) {
    if (tiles && chip) return wide ? quad_fn_c<int64_t, true, moc::kQuadTeams>(C, profile) : quad_fn_c<int32_t, true, moc::kQuadTeams>(C, profile);
    if (tiles) return wide ? quad_fn_c<int64_t, true, moc::kQuadBlock>(C, profile) : quad_fn_c<int32_t, true, moc::kQuadBlock>(C, profile);
    return wide ? quad_fn_c<int64_t, false, moc::kQuadBlock>(C, profile) : quad_fn_c<int32_t, false, moc::kQuadBlock>(C, profile);
}
}  // namespace moc_host
