// The shared launch of pf_tc_gemm_kernel.cuh as the convolution's backward needs it (implicit-GEMM operands), in a
// translation unit of its own so that the plain kernels keep a module without it.
#include "pf_tc.h"

#include "pf_tc_gemm_kernel.cuh"
#include "pf_tc_host.h"

namespace pf {
namespace tc {

cudaError_t launch_gemm3_conv(int blocks, size_t smem, cudaStream_t stream, const Gemm3Args& a) {
    const cudaError_t e = allow_smem(tc_gemm3_kernel<true, false>, 227 * 1024);
    if (e != cudaSuccess) return e;
    return launch_overlapped(tc_gemm3_kernel<true, false>, dim3(static_cast<unsigned>(blocks)), dim3(kGemmThreads), smem, stream, a.ta[0], a.tb[0],
                             a.ta[1], a.tb[1], a.ta[2], a.tb[2], a.p[0], a.p[1], a.p[2], a.end0, a.end1, a.tiles[0], a.tiles[1], a.tiles[2]);
}

}  // namespace tc
}  // namespace pf
