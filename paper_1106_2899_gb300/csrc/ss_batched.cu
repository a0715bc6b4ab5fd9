// ss_batched.cu -- the kernel over many elements, by lane layout.
#include "ss_kernels.cuh"
#include "ss_launch.h"

namespace ssk {
namespace {

template <typename T>
const void* batched_fn(int W, int B) {
    switch (W * 16 + B) {
        case 8 * 16 + 1: return (const void*)batched_kernel<T, 8, 1>;
        case 8 * 16 + 2: return (const void*)batched_kernel<T, 8, 2>;
        case 8 * 16 + 3: return (const void*)batched_kernel<T, 8, 3>;
        case 16 * 16 + 1: return (const void*)batched_kernel<T, 16, 1>;
        case 16 * 16 + 2: return (const void*)batched_kernel<T, 16, 2>;
        case 16 * 16 + 3: return (const void*)batched_kernel<T, 16, 3>;
        case 16 * 16 + 4: return (const void*)batched_kernel<T, 16, 4>;
        case 32 * 16 + 1: return (const void*)batched_kernel<T, 32, 1>;
        case 32 * 16 + 3: return (const void*)batched_kernel<T, 32, 3>;
        case 32 * 16 + 4: return (const void*)batched_kernel<T, 32, 4>;
        default: return nullptr;
    }
}

}  // namespace

const void* batched_fn_f32(int W, int B) { return batched_fn<float>(W, B); }
const void* batched_fn_f64(int W, int B) { return batched_fn<double>(W, B); }

}  // namespace ssk
