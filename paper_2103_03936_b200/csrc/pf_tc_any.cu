// The product kernels of pf_tc_gemm_kernel.cuh compiled for any form of output (see gemm_tile), in a translation unit of
// their own so that the others keep a module without them.
#include "pf_tc.h"

#include "pf_tc_gemm_kernel.cuh"
#include "pf_tc_host.h"

namespace pf {
namespace tc {

namespace {
template <int BN>
cudaError_t launch_one(dim3 grid, size_t smem, cudaStream_t stream, const CUtensorMap& ta, const CUtensorMap& tb, const GemmParams& p) {
    const cudaError_t e = allow_smem(tc_gemm_kernel<BN, false, true>, 227 * 1024);
    return e != cudaSuccess ? e : launch_overlapped(tc_gemm_kernel<BN, false, true>, grid, dim3(kGemmThreads), smem, stream, ta, tb, p);
}
template <bool kConv>
cudaError_t launch_three(int blocks, size_t smem, cudaStream_t stream, const Gemm3Args& a) {
    const cudaError_t e = allow_smem(tc_gemm3_kernel<kConv, true>, 227 * 1024);
    if (e != cudaSuccess) return e;
    return launch_overlapped(tc_gemm3_kernel<kConv, true>, dim3(static_cast<unsigned>(blocks)), dim3(kGemmThreads), smem, stream, a.ta[0], a.tb[0],
                             a.ta[1], a.tb[1], a.ta[2], a.tb[2], a.p[0], a.p[1], a.p[2], a.end0, a.end1, a.tiles[0], a.tiles[1], a.tiles[2]);
}
}  // namespace

cudaError_t launch_gemm_any(int bn, dim3 grid, size_t smem, cudaStream_t stream, const CUtensorMap& ta, const CUtensorMap& tb, const GemmParams& p) {
    return bn == 64 ? launch_one<64>(grid, smem, stream, ta, tb, p) : launch_one<128>(grid, smem, stream, ta, tb, p);
}
cudaError_t launch_gemm3_any(bool conv, int blocks, size_t smem, cudaStream_t stream, const Gemm3Args& a) {
    return conv ? launch_three<true>(blocks, smem, stream, a) : launch_three<false>(blocks, smem, stream, a);
}

}  // namespace tc
}  // namespace pf
