// Kernel launches of libqamw: every kernel may start while the one before it on the stream drains.
#ifndef QAMW_LAUNCH_H_
#define QAMW_LAUNCH_H_

#include <cuda_runtime.h>

#include <utility>

namespace qamw {

// Launch with programmatic stream serialisation.  The kernel must call chain_wait() (qamw_device.cuh) before it
// touches anything an earlier kernel of the stream may write or still read; what it does before that -- tables
// of a codebook, which never change -- overlaps the end of its predecessor.  Measured on a B200 with kernels that
// only spin: ordinary launches on a stream complete on a grid of 2.05 us (a 3 us kernel costs 4.1 us, one of
// 1 us 2.6 us), chained ones take their own time and at least 2.0 us.
template <class... P, class... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = st;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &attr;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kernel, P(std::forward<A>(args))...);
}

}  // namespace qamw

#endif  // QAMW_LAUNCH_H_
