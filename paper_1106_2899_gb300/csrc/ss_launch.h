// ss_launch.h -- the chain kernels by lane layout, for the host runtime.
//
// The instantiations live in translation units of their own (ss_chunk_*.cu,
// ss_batched.cu, ss_adjoint.cu), so that they compile in parallel; each hands out
// its kernels as cudaLaunchKernel takes them.
#pragma once

namespace ssk {

// chunk_kernel<T, W, B, win, FLOW, heun, corr, alt>, launched with (ChunkArgs,
// StepConst<T>); null for a layout that is not compiled, the first form where there is
// no second.  Windows (win != kWinOff)
// run the Euler-Maruyama step without flow.
const void* chunk_fn_f32(int W, int B, int win, bool heun, bool corr, bool alt);
const void* chunk_fn_f32_flow(int W, int B, int win, bool heun, bool corr, bool alt);
const void* chunk_fn_f64(int W, int B, int win, bool heun, bool corr, bool alt);
const void* chunk_fn_f64_flow(int W, int B, int win, bool heun, bool corr, bool alt);
// batched_kernel<T, W, B>
const void* batched_fn_f32(int W, int B);
const void* batched_fn_f64(int W, int B);
// adjoint_kernel<T, W, B>, launched with (AdjArgs, StepConst<T>)
const void* adjoint_fn_f32(int W, int B);
const void* adjoint_fn_f64(int W, int B);

}  // namespace ssk
