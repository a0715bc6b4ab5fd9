// chunk_kernel of one precision by lane layout, with or without the flow terms
// (included by the ss_chunk_*.cu units).
#include "ss_kernels.cuh"
#include "ss_launch.h"

namespace ssk {
namespace {

// 8 x 2 and 8 x 3 serve FP32 runs of the Euler-Maruyama step alone (layout_for)
template <int W, int B>
constexpr bool kNarrow = W == 8 && B > 1;

template <typename T, int W, int B, bool FLOW, bool ALT>
const void* chunk_of(int win, bool heun, bool corr) {
    if constexpr (!FLOW) {
        if (win == kWinRecord) return (const void*)chunk_kernel<T, W, B, kWinRecord, false, false, true>;
        if (win == kWinReplay) return (const void*)chunk_kernel<T, W, B, kWinReplay, false, false, true>;
    }
    // (without a series the two forms of the Heun step without flow are the same)
    constexpr bool E2 = ALT && has_second_form(W, B, false, FLOW), H2 = ALT && has_second_form(W, B, true, FLOW);
    if constexpr (kNarrow<W, B>) {
        if (heun) return nullptr;
    } else if (heun) {
        return corr ? (const void*)chunk_kernel<T, W, B, kWinOff, FLOW, true, true, H2>
                    : (const void*)chunk_kernel<T, W, B, kWinOff, FLOW, true, false, H2 && FLOW>;
    }
    return corr ? (const void*)chunk_kernel<T, W, B, kWinOff, FLOW, false, true, E2>
                : (const void*)chunk_kernel<T, W, B, kWinOff, FLOW, false, false, E2>;
}

template <typename T, int W, int B, bool FLOW>
const void* chunk_form(int win, bool heun, bool corr, bool alt) {
    if constexpr (sizeof(T) == 4 && (has_second_form(W, B, false, FLOW) || has_second_form(W, B, true, FLOW))) {
        if (alt && win == kWinOff) return chunk_of<T, W, B, FLOW, true>(win, heun, corr);
    }
    return chunk_of<T, W, B, FLOW, false>(win, heun, corr);
}

template <typename T, bool FLOW>
const void* chunk_fn(int W, int B, int win, bool heun, bool corr, bool alt) {
    if constexpr (sizeof(T) == 4) {
        if (W == 8 && B == 2) return chunk_form<T, 8, 2, FLOW>(win, heun, corr, alt);
        if (W == 8 && B == 3) return chunk_form<T, 8, 3, FLOW>(win, heun, corr, alt);
    }
    switch (W * 16 + B) {
        case 8 * 16 + 1: return chunk_form<T, 8, 1, FLOW>(win, heun, corr, alt);
        case 16 * 16 + 1: return chunk_form<T, 16, 1, FLOW>(win, heun, corr, alt);
        case 16 * 16 + 2: return chunk_form<T, 16, 2, FLOW>(win, heun, corr, alt);
        case 16 * 16 + 3: return chunk_form<T, 16, 3, FLOW>(win, heun, corr, alt);
        case 16 * 16 + 4: return chunk_form<T, 16, 4, FLOW>(win, heun, corr, alt);
        case 32 * 16 + 3: return chunk_form<T, 32, 3, FLOW>(win, heun, corr, alt);
        case 32 * 16 + 4: return chunk_form<T, 32, 4, FLOW>(win, heun, corr, alt);
        default: return nullptr;
    }
}

}  // namespace
}  // namespace ssk
