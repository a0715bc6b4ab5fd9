// The chain kernel in FP64, with the flow terms.
#include "ss_chunk.inl"

const void* ssk::chunk_fn_f64_flow(int W, int B, int win, bool heun, bool corr, bool alt) {
    return chunk_fn<double, true>(W, B, win, heun, corr, alt);
}
