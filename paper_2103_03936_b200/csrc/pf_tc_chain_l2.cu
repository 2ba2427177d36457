// The fused chain kernel with hints to L2, for launches that stream more than it holds, in a translation unit of its own (see
// pf_tc_chain_multi.cu).
#include <cuda.h>

#include "pf_tc.h"
#include "pf_tc_host.h"
#include "pf_tc_chain_kernel.cuh"

namespace pf {
namespace tc {

int chain_launch_hints(dim3 grid, size_t smem, cudaStream_t stream, const CUtensorMap& ta, const CUtensorMap& tb1, const CUtensorMap& tb2,
                       const CUtensorMap& to, const CUtensorMap& tt, const ChainParams& p) {
    auto* kernel = p.bias || p.act ? tc_chain_kernel<false, true, 4> : tc_chain_kernel<false, false, 4>;
    if (allow_smem(kernel, 227 * 1024) != cudaSuccess ||
        launch_overlapped(kernel, grid, dim3(kChainThreads), smem, stream, ta, tb1, tb2, to, tt, p) != cudaSuccess)
        return PF_ERR_CUDA;
    count_launch();
    return PF_OK;
}

}  // namespace tc
}  // namespace pf
