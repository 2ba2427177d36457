// Plain products with several output tiles per block (run_tiles of pf_tc_gemm_kernel.cuh), in a translation unit of their
// own: compiled beside the convolution's products they changed those kernels' code and slowed them by 3 %.
#include "pf_tc.h"

#include "pf_tc_gemm_kernel.cuh"
#include "pf_tc_host.h"

namespace pf {
namespace tc {

namespace {
template <int BN>
cudaError_t launch_one(dim3 grid, size_t smem, cudaStream_t stream, const CUtensorMap& ta, const CUtensorMap& tb, const GemmParams& p) {
    const cudaError_t e = allow_smem(tc_gemm_kernel<BN, true, false>, 227 * 1024);
    return e != cudaSuccess ? e : launch_overlapped(tc_gemm_kernel<BN, true, false>, grid, dim3(kGemmThreads), smem, stream, ta, tb, p);
}
}  // namespace

cudaError_t launch_gemm_runs(int bn, dim3 grid, size_t smem, cudaStream_t stream, const CUtensorMap& ta, const CUtensorMap& tb,
                             const GemmParams& p) {
    if (bn > 128) return cudaErrorInvalidValue;
    return bn == 64 ? launch_one<64>(grid, smem, stream, ta, tb, p) : launch_one<128>(grid, smem, stream, ta, tb, p);
}

}  // namespace tc
}  // namespace pf
