// The fused chain kernels with a convolution as first product, in a translation unit of their own: with the
// convolution's addressing behind a run-time test in the shared kernels, both they and it ran 3-4 % slower.
#include <cuda.h>

#include "pf_tc.h"
#include "pf_tc_host.h"
#include "pf_tc_chain_pipe.cuh"

namespace pf {
namespace tc {

int chain_launch_conv(bool pipe, bool ragged, dim3 grid, size_t smem, cudaStream_t stream, const CUtensorMap& ta, const CUtensorMap& tb1,
                      const CUtensorMap& tb2, const CUtensorMap& to, const CUtensorMap& tt, const ChainParams& p) {
    auto* kernel = pipe ? (ragged ? tc_chain_pipe_kernel<2> : tc_chain_pipe_kernel<1>)
                        : (ragged ? tc_chain_kernel<false, false, 2> : tc_chain_kernel<false, false, 1>);
    if (allow_smem(kernel, 227 * 1024) != cudaSuccess ||
        launch_overlapped(kernel, grid, dim3(kChainThreads), smem, stream, ta, tb1, tb2, to, tt, p) != cudaSuccess)
        return PF_ERR_CUDA;
    count_launch();
    return PF_OK;
}

}  // namespace tc
}  // namespace pf
