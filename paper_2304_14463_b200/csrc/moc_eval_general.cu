// General kernels: a thread group per sequence, any C, state on chip or in global memory.
#include "moc_host.cuh"

namespace moc_host {
namespace {
template <int G, typename MemT>
KernelFn shared_fn_cp(int CP, bool profile) {
    if (profile && G != 1024) return nullptr;
    switch (CP) {
        case 2: return profile ? (KernelFn)moc::eval_shared_kernel<1024, MemT, 2, true>
                               : (KernelFn)moc::eval_shared_kernel<G, MemT, 2, false>;
        case 4: return profile ? (KernelFn)moc::eval_shared_kernel<1024, MemT, 4, true>
                               : (KernelFn)moc::eval_shared_kernel<G, MemT, 4, false>;
        default: return profile ? (KernelFn)moc::eval_shared_kernel<1024, MemT, 8, true>
                                : (KernelFn)moc::eval_shared_kernel<G, MemT, 8, false>;
    }
}
template <typename MemT>
KernelFn shared_fn_g(int G, int CP, bool profile) {
    switch (G) {
        case 32: return shared_fn_cp<32, MemT>(CP, profile);
        case 64: return shared_fn_cp<64, MemT>(CP, profile);
        case 128: return shared_fn_cp<128, MemT>(CP, profile);
        case 256: return shared_fn_cp<256, MemT>(CP, profile);
        case 512: return shared_fn_cp<512, MemT>(CP, profile);
        case 1024: return shared_fn_cp<1024, MemT>(CP, profile);
        default: return nullptr;
    }
}
}  // namespace

KernelFn global_fn(int CP, bool profile) {
    switch (CP) {
        case 2: return profile ? (KernelFn)moc::eval_global_kernel<2, true> : (KernelFn)moc::eval_global_kernel<2, false>;
        case 4: return profile ? (KernelFn)moc::eval_global_kernel<4, true> : (KernelFn)moc::eval_global_kernel<4, false>;
        default: return profile ? (KernelFn)moc::eval_global_kernel<8, true> : (KernelFn)moc::eval_global_kernel<8, false>;
    }
}
KernelFn shared_fn(bool wide, int G, int CP, bool profile) {
    return wide ? shared_fn_g<int64_t>(G, CP, profile) : shared_fn_g<int32_t>(G, CP, profile);
}
}  // namespace moc_host
