// Mixed-precision forward kernels of order 25.
#include "lr_fwdmx.cuh"

namespace lr {

template <int T>
static void *kernel_ptr_mx(int kind)
{
    switch (kind) {
        case KIND_PROJECT: return (void *)k_mixed<T, KIND_PROJECT>;
        case KIND_TDI: return (void *)k_mixed<T, KIND_TDI>;
        case KIND_WIDE: return (void *)k_mixed<T, KIND_FUSED, MIXED_WIDE>;
        case KIND_LIKE: return (void *)k_mixed<T, KIND_LIKE>;
        case KIND_FUSED_GEN: return (void *)k_mixed<T, KIND_FUSED, MIXED_THREADS, true>;
        case KIND_LIKE_GEN: return (void *)k_mixed<T, KIND_LIKE, MIXED_THREADS, true>;
        default: return (void *)k_mixed<T, KIND_FUSED>;
    }
}

void *kernel_for_mx_p25(int kind, int order)
{
    switch (order) {
        case 25: return kernel_ptr_mx<26>(kind);
        default: return nullptr;
    }
}

}  // namespace lr
