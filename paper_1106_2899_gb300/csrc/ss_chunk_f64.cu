// The chain kernel in FP64, without the flow terms.
#include "ss_chunk.inl"

const void* ssk::chunk_fn_f64(int W, int B, int win, bool heun, bool corr, bool alt) {
    return chunk_fn<double, false>(W, B, win, heun, corr, alt);
}
