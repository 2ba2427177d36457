// The fp32 product kernel with the convolution's addressing modes, in a translation unit of its own.
#include "pf_tc.h"

#include "pf_tc_f32_kernel.cuh"
#include "pf_tc_host.h"

namespace pf {
namespace tc {

cudaError_t launch_f32_conv(int blocks, size_t smem, cudaStream_t stream, const F32Launch& a) {
    const cudaError_t e = allow_smem(tc_f32_kernel<true>, 227 * 1024);
    if (e != cudaSuccess) return e;
    return launch_overlapped(tc_f32_kernel<true>, dim3(static_cast<unsigned>(blocks)), dim3(kF32Threads), smem, stream, a);
}

}  // namespace tc
}  // namespace pf
