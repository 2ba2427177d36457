// Tensor-core (tcgen05 / TMEM / TMA) path for bf16 storage.  Each entry either handles the
// call (*handled = 1) or declines it (*handled = 0, nothing launched) when the shape lies
// outside its envelope; the caller then uses the FMA kernels.
#ifndef PF_TC_H_
#define PF_TC_H_

#include <functional>

#include "pf_internal.h"

namespace pf {

unsigned int* device_status_ptr();  // per-device address of the bounded-wait status word

namespace tc {

struct LinearArgs {
    const void *x = nullptr, *U = nullptr, *V = nullptr, *dY = nullptr;
    void *y = nullptr, *T = nullptr, *dX = nullptr, *dU = nullptr, *dV = nullptr;
    int64_t ldx = 0, ldu = 0, ldv = 0, ldy = 0, ldt = 0, lddy = 0, lddx = 0, lddu = 0, lddv = 0;
    int64_t m = 0, k = 0, n = 0, r = 0;
    char *ws = nullptr, *ws_T = nullptr, *ws_G = nullptr;
    cudaStream_t stream = nullptr;
    const void* bias = nullptr;   // forward: y = act((x U) V^T + bias)
    int act = 0;
    bool tight = false;           // forward: the leaner plan, for a workspace of a given size that the faster one does not fit
    bool whole = false;           // forward: no slices of the first product, which take room
    bool group_member = false;    // one of several calls that make up a grouped one (two launches each, as documented)
    // backward: where the fp32 slices of dU / dV were left in the workspace (partial null: nowhere), for callers that want
    // the unrounded sums; a product that is one slice leaves only that
    struct Slices {
        const float* partial = nullptr;
        int splits = 0, bn = 0, tiles_x = 0, tiles_y = 0;
        int conv_c = 0;     // > 0: tiles are pairs of 64-channel blocks of a [taps][conv_c] row index
    };
    Slices* du_slices = nullptr;
    Slices* dv_slices = nullptr;
};

struct ConvArgs {
    const void *x, *U, *V, *dY;
    void *y, *T, *dX, *dU, *dV;
    int N, H, W, C, R, O, kh, kw, stride, pad, Ho, Wo;
    char *ws, *ws_T, *ws_G;
    cudaStream_t stream;
    // backward: where the fp32 slices of dU / dV were left (see LinearArgs::Slices); may be null
    LinearArgs::Slices *du_slices, *dv_slices;
    struct Gradients {            // the caller's matrices, of a call that wants them in fp32 or accumulated
        void *dU, *dV;
        bool f32, accumulate, written;      // written: by the launches themselves
    } * gradients;                // null: dU and dV are the caller's
    bool lean;      // backward, bf16: ws and ws_G have room for the products that fetch pixels per tap only, ws_G with R elements per pixel
};

// Launches that what follows reads: made once a call is accepted, i.e. when nothing can decline it any more.
using Before = std::function<int()>;

// Fused chain kernel (pf_tc_chain.cu): out = (A * B1) * B2^T with the intermediate on chip.
struct ChainPlan {
    int r_pad, num_stages, stage_bytes, nsplit, tiles_per_split, row_tiles, boxes_per_stage, staging_off;
    size_t smem;
};
// `max_split` caps the number of column ranges the output is split into (0 = no cap); `groups` problems share the launch.
bool chain_plan(int64_t M, int64_t K1, int64_t N2, int64_t r, bool has_out, ChainPlan* plan, int rows_tile = 128,
                int max_split = 0, int groups = 1);
// Blocks of output pixels of a convolution (see conv_tiling): bh full-width rows of nb images, tpi blocks per
// image (nb > 1 only with whole images).
struct ConvTiling {
    int nb = 1, bh = 1, tpi = 1, pixels = 0;
    int64_t blocks = 0;
};
ConvTiling conv_tiling(int N, int Ho, int Wo, int limit);
// When `conv` is given, A is an NHWC image and phase 1 is the implicit GEMM of a kh x kw convolution: B1 = U
// as [kh*kw][C][r] (M and K1 are derived from it).  stride applies to the k x k convolution: the image tile of
// a tap is fetched with that step between pixels (a tensor map with element strides).
struct ChainConv {
    int N, H, W, C, kh, kw, pad, stride;
};
int chain(const void* A, int64_t lda, int64_t M, int64_t K1, const void* B1, int64_t ldb1, int64_t r,
          const void* B2, int64_t ldb2, int64_t N2, void* out, int64_t ldo, void* T, int64_t ldt,
          cudaStream_t stream, const ChainConv* conv = nullptr, int max_split = 0, const void* bias = nullptr,
          int act = 0,    // bias [N2] (bf16) and act (0 identity, 1 max(0, .)) apply to `out`
          float keep_a = 0.f, float keep_out = 0.f,       // how L2 treats A and `out` (l2_policy in pf_tc_prims.cuh)
          const Before& before = {});

int chain_groups(int groups, int all, const void* A, int64_t lda, int64_t sA, int64_t M, int64_t K1, const void* B1, int64_t ldb1, int64_t sB1, int64_t r,
                 const void* B2, int64_t ldb2, int64_t sB2, int64_t N2, void* out, int64_t ldo, int64_t sO, void* T, int64_t ldt, int64_t sT,
                 bool late_wait, cudaStream_t stream);

// Products on CTA pairs (pf_tc_pair.cu): C[M,N] = act(A * B + bias) for `groups` problems of one shape, matrices *_gs
// elements apart (0 = one operand shared by all groups); sum_groups: the groups are summed into one C.
struct PairJob {
    const void* A;
    int64_t lda;
    bool a_mn;
    int64_t a_gs;
    const void* B;
    int64_t ldb;
    bool b_mn;
    int64_t b_gs;
    int64_t M, N, K;
    void* C;
    int64_t ldc;
    int64_t c_gs = 0;
    int groups = 1;
    bool sum_groups = false;
    const void* bias = nullptr;
    int act = 0;
    bool a_early = false, b_early = false;      // see kEarlyA in pf_tc_prims.cuh
};
int gemm_pairs(const PairJob* jobs, int count, int first, cudaStream_t stream);

// Grouped factorized linear layer: `groups` problems of one shape (several factor pairs applied to the
// same or to different inputs) in two launches forward and two backward, whatever the group count.
// Strides s* are in elements between consecutive groups; sx == 0 means one x shared by all groups,
// in which case dX is ONE matrix, the sum over the groups.
struct GroupedArgs {
    int groups = 1;
    const void *x = nullptr, *U = nullptr, *V = nullptr, *dY = nullptr;
    void *y = nullptr, *T = nullptr, *dX = nullptr, *dU = nullptr, *dV = nullptr;
    int64_t ldx = 0, ldu = 0, ldv = 0, ldy = 0, ldt = 0, lddy = 0, lddx = 0, lddu = 0, lddv = 0;
    int64_t sx = 0, su = 0, sv = 0, sy = 0, st = 0, sdy = 0, sdx = 0, sdu = 0, sdv = 0;
    int64_t m = 0, k = 0, n = 0, r = 0;
    char* ws = nullptr;
    cudaStream_t stream = nullptr;
};
size_t grouped_workspace(int groups, int64_t m, int64_t k, int64_t n, int64_t r, bool bwd);
int linear_grouped_fwd(const GroupedArgs& a, int* handled);
int linear_grouped_bwd(const GroupedArgs& a, int* handled);

size_t linear_extra_workspace(int64_t m, int64_t k, int64_t n, int64_t r, bool bwd);
size_t conv_extra_workspace(int N, int H, int W, int C, int R, int O, int kh, int kw, int stride,
                            int pad, bool bwd, bool lean = false);
void reset_fix_counters();  // clears the slice-sum counters (after PF_ERR_TIMEOUT)
size_t linear_fwd_need(const LinearArgs& a, bool* handles);   // bytes of a.ws the forward really touches
int64_t linear_fwd_rows(const LinearArgs& a, size_t room, LinearArgs* b);   // rows at a time in so much room, 0: not by rows
int linear_fwd(const LinearArgs& a, int* handled);
bool few_rows_fused(const LinearArgs& a);     // a forward that small::linear_fwd fits, but the fused kernel takes
int linear_bwd(const LinearArgs& a, int* handled);

// fp32 storage (pf_tc_f32.cu).  `room`: bytes available at a.ws (a call that does not fit is declined).
size_t f32_linear_workspace(int64_t m, int64_t k, int64_t n, int64_t r, bool bwd, bool tight = false);
int f32_linear_fwd(const LinearArgs& a, int* handled, size_t room);
int f32_linear_bwd(const LinearArgs& a, int* handled);
size_t f32_conv_workspace(const ConvArgs& a, bool bwd);      // a: sizes only
int f32_conv_fwd(const ConvArgs& a, int* handled);
int f32_conv_bwd(const ConvArgs& a, int* handled);
// Device counters for one product whose contraction is split (null on error).
unsigned int* split_counters();
// 3 x 3, stride-1 convolutions on resident image windows (pf_tc_conv_res.cu); PF_ERR_UNSUPPORTED outside their envelope.
int conv_res_fwd(const ConvArgs& a, int64_t ldf, const Before& before);      // ldf: pitch of the factors
// Their backward (pf_tc_conv_bwd.cu), where `conv_flat_bwd_pays`; T is x U, a.ws_G takes dT.  PF_ERR_UNSUPPORTED: nothing has been launched.
bool conv_flat_bwd_pays(const ConvArgs& a, bool dX);      // a: sizes only
size_t conv_flat_bwd_workspace(const ConvArgs& a);      // a: sizes only; 0 where it does not pay
int conv_flat_bwd(const ConvArgs& a, const void* T, const void* U, int64_t ldu, char* ws, bool early,     // early: the launch before copies U, nothing else
                  const Before& before);
int conv_fwd(const ConvArgs& a, int* handled);
int conv_bwd(const ConvArgs& a, int* handled);      // a.ws_G: conv_dt_pitch(R) elements per pixel, unless lean
int64_t conv_dt_pitch(int64_t R);

}  // namespace tc

// Few rows, bf16, any layout (pf_small.cu).
namespace small {
bool linear_fwd_fits(int64_t m, int64_t k, int64_t n, int64_t r);
int linear_fwd(const tc::LinearArgs& a, void* T, int64_t ldt);
// The smallest layers, any layout: the whole backward in one launch (needs T; a.dU and a.dV are the caller's).
bool tiny_fits(int64_t m, int64_t k, int64_t n, int64_t r, int dtype);
int tiny_bwd(const tc::LinearArgs& a, int dtype, bool grads_f32, bool accumulate);
// fp32, small products, any layout.
bool f32_fits(int64_t m, int64_t k, int64_t n, int64_t r, bool bwd);
int f32_linear_fwd(const tc::LinearArgs& a, void* T, int64_t ldt);
int f32_linear_bwd(const tc::LinearArgs& a);
}  // namespace small
}  // namespace pf
#endif
