// The chain kernel in FP32, without the flow terms.
#include "ss_chunk.inl"

const void* ssk::chunk_fn_f32(int W, int B, int win, bool heun, bool corr, bool alt) {
    return chunk_fn<float, false>(W, B, win, heun, corr, alt);
}
