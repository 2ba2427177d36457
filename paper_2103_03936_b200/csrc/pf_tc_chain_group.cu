// The fused chain kernel over several groups of one shape, in a translation unit of its own (see pf_tc_chain_multi.cu).
#include <cuda.h>

#include "pf_tc.h"
#include "pf_tc_host.h"
#include "pf_tc_chain_kernel.cuh"

namespace pf {
namespace tc {

int chain_launch_groups(dim3 grid, size_t smem, cudaStream_t stream, const CUtensorMap& ta, const CUtensorMap& tb1, const CUtensorMap& tb2,
                        const CUtensorMap& to, const CUtensorMap& tt, const ChainParams& p) {
    if (allow_smem(tc_chain_kernel<false, false, 3>, 227 * 1024) != cudaSuccess ||
        launch_overlapped(tc_chain_kernel<false, false, 3>, grid, dim3(kChainThreads), smem, stream, ta, tb1, tb2, to, tt, p) != cudaSuccess)
        return PF_ERR_CUDA;
    count_launch();
    return PF_OK;
}

}  // namespace tc
}  // namespace pf
