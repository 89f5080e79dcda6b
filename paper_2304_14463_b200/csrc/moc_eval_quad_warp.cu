// Block-per-sequence kernel's code with a warp per sequence (C = 3, 4).
#include "moc_host.cuh"

namespace moc_host {
QuadFn quad_warp_fn(bool wide, int C) {
    if (wide) return C <= 3 ? (QuadFn)moc::eval_quad_warp_kernel<int64_t, 3> : (QuadFn)moc::eval_quad_warp_kernel<int64_t, 4>;
    return C <= 3 ? (QuadFn)moc::eval_quad_warp_kernel<int32_t, 3> : (QuadFn)moc::eval_quad_warp_kernel<int32_t, 4>;
}
}  // namespace moc_host
