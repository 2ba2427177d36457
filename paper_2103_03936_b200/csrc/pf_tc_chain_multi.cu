// The software-pipelined persistent form of the fused chain (pf_tc_chain_pipe.cuh, r <= 128), compiled in a translation
// unit of its own: with both forms in one module the single-tile form, which the one-wave layers run,
// measurably slowed down inside a training step although the persistent form was never launched there.
#include <cuda.h>

#include "pf_tc.h"
#include "pf_tc_host.h"
#include "pf_tc_chain_pipe.cuh"

namespace pf {
namespace tc {

int chain_launch_pipe(dim3 grid, size_t smem, cudaStream_t stream, const CUtensorMap& ta, const CUtensorMap& tb1,
                      const CUtensorMap& tb2, const CUtensorMap& to, const CUtensorMap& tt, const ChainParams& p) {
    if (allow_smem(tc_chain_pipe_kernel<0>, 227 * 1024) != cudaSuccess ||
        launch_overlapped(tc_chain_pipe_kernel<0>, grid, dim3(kChainThreads), smem, stream, ta, tb1, tb2, to, tt, p) != cudaSuccess)
        return PF_ERR_CUDA;
    count_launch();
    return PF_OK;
}

}  // namespace tc
}  // namespace pf
