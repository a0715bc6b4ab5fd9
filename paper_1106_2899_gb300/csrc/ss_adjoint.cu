// ss_adjoint.cu -- the reverse sweep of differentiation windows, by lane layout.
#include "ss_adjoint.cuh"
#include "ss_launch.h"

namespace ssk {
namespace {

template <typename T>
const void* adjoint_fn(int W, int B) {
    if constexpr (sizeof(T) == 4) {  // FP64 windows of that length run 16 x 2
        if (W == 8 && B == 3) return (const void*)adjoint_kernel<T, 8, 3>;
    }
    switch (W * 16 + B) {
        case 8 * 16 + 1: return (const void*)adjoint_kernel<T, 8, 1>;
        case 16 * 16 + 1: return (const void*)adjoint_kernel<T, 16, 1>;
        case 16 * 16 + 2: return (const void*)adjoint_kernel<T, 16, 2>;
        case 16 * 16 + 3: return (const void*)adjoint_kernel<T, 16, 3>;
        case 16 * 16 + 4: return (const void*)adjoint_kernel<T, 16, 4>;
        case 32 * 16 + 3: return (const void*)adjoint_kernel<T, 32, 3>;
        case 32 * 16 + 4: return (const void*)adjoint_kernel<T, 32, 4>;
        default: return nullptr;
    }
}

}  // namespace

const void* adjoint_fn_f32(int W, int B) { return adjoint_fn<float>(W, B); }
const void* adjoint_fn_f64(int W, int B) { return adjoint_fn<double>(W, B); }

}  // namespace ssk
