// Programmatic dependent launch of the step kernels.
//
// A step of a small grid lasts 4 to 6 us, of which 1 to 2.5 us pass between the end of one kernel and the
// first instruction of the next: its launch waits until the writes of the kernel before it are flushed.
// Kernels launched with launch_pdl are set up while the last CTAs of the kernel before them in the stream
// end, and run up to pdl_wait, which returns when that kernel has ended and its writes are visible.  Before
// it a kernel touches only what no kernel writes after set-up (tile flags, work records, node types) and its
// own shared memory; every read of a state, every global write and every counter comes after.  Nothing else
// in a stream changes: a copy or a kernel launched the usual way still waits for the end of these.
//
// Measured with the plain launch on the same box (us per step in 16-step graphs, per step launched one by
// one, per fields pass): D2Q9 FP32 300 x 350 6.04 -> 5.53, 8.23 -> 5.67, 6.21 -> 4.31; 600 x 400 6.80 -> 6.42,
// 8.24 -> 6.46, 8.22 -> 5.03; D2Q9 FP64 100 x 100 11.0 -> 10.8, 12.3 -> 10.8, 10.3 -> 8.1; 96 FP32 grids of
// 128^2 to 512^2: the fields of all 800 -> 584.  No kernel lets the next one start earlier than its end
// (griddepcontrol.launch_dependents): at its beginning that costs more than it gives, since the CTAs that
// wait take the place of CTAs that work (300 x 350: 6.32 us, 600 x 400: 6.96 us).
#pragma once

#include <utility>

#include <cuda_runtime.h>

namespace lbmwet {

#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
#endif

template <class... P, class... A>
cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = s;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &attr;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kernel, P(std::forward<A>(args))...);
}

}  // namespace lbmwet
