// Tensor-core path (bf16 storage) for sm_100a: host planning of every product (tensor maps, tiles, slices of split
// contractions, which products share a launch) and the plain product kernels of pf_tc_gemm_kernel.cuh.
#include "pf_tc.h"

#include <cuda.h>

#include <algorithm>
#include <atomic>
#include <cmath>

#include "pf_tc_gemm_kernel.cuh"
#include "pf_tc_host.h"

namespace pf {
namespace tc {
namespace {

constexpr int kFixSlots = 32;  // counter sets handed out round-robin to launches that split a contraction
constexpr int kFixTiles = 160; // output tiles of one split product (tiles * slices never exceeds the SM count)

// Arrival / departure counters of the in-kernel slice sum, two per output tile.  They are zero
// between launches: the last CTA to leave a tile clears its pair.
__device__ unsigned int g_fix_counters[kFixSlots][kFixTiles * 2];

// ------------------------------------------------------------------------------ host side
// One operand of C = A * B.  `mn_major == false`: stored [MN, K] row-major (contraction index
// contiguous).  `mn_major == true`: stored [K, MN] row-major (M or N index contiguous).
struct Operand {
    const void* p;
    int64_t ld;
    bool mn_major;
    int64_t gs = 0;     // grouped products: elements between the matrices of consecutive groups (0 = one matrix shared by all)
    bool warm = false;  // written by the launch before: in L2 if it fits
    bool early = false; // neither written by the launch before nor by anything that may still run when that one has started (kEarlyA)
};

// Several problems of one shape in one product.  sum_groups: the groups are summed into ONE output (the
// group index is part of the contraction; both operands K-major), otherwise every group has its own
// output, c_gs elements apart.
struct Grouping {
    int groups = 1;
    int64_t c_gs = 0;
    bool sum_groups = false;
};

size_t gemm_smem(int bn, int stages, bool dx = false) {
    return 1024 + 1024 + static_cast<size_t>(stages) * (kBM * kBK * 2 + bn * kBK * 2) + (dx ? 4 * kDxPanel : 0);
}
// Pipeline depth: a grid that fits one wave gets every stage shared memory has room for; a
// larger grid gets stages small enough for two CTAs per SM, so that the prologue and epilogue of
// one CTA overlap the main loop of the other.
int pick_stages(int bn, int64_t ctas, bool dx = false) {
    const size_t stage = static_cast<size_t>(kBM * kBK * 2 + bn * kBK * 2);
    const size_t room = (ctas > num_sms() ? (113 * 1024 - 2048) : (200 * 1024 - 2048)) - (dx ? 4 * kDxPanel : 0);
    int ns = static_cast<int>(room / stage);
    if (ns > kMaxStages) ns = kMaxStages;
    if (ns < 2) ns = 2;
    return ns;
}

// Blocks that share the tiles of a convolution's dX: runs of about 16 k-blocks hide the start of a block (2 tiles of a
// stride-1 layer, 8 of a strided one, whose tiles are short), longer ones make the blocks of the launch unequal
// (backward of 32 x 56 x 56, 64 -> 16 -> 64 with 6 tiles per block: 61 us instead of 56, cold L2); every SM gets a
// block first.
// The tiles of a block are that many blocks apart: no multiple of the stride's factors, so that it gets every class.
unsigned run_blocks(int64_t tiles, int64_t kblocks_per_tile, int stride) {
    const int64_t want = std::min<int64_t>(8, std::max<int64_t>(2, ceil_div(16, std::max<int64_t>(1, kblocks_per_tile))));
    int64_t blocks = ceil_div(tiles, std::min(want, ceil_div(tiles, num_sms())));
    while (stride > 1 && blocks < tiles && (blocks % 2 == 0 || blocks % stride == 0)) ++blocks;      // (strides up to 4)
    return static_cast<unsigned>(blocks);
}

bool vector_rows(const void* C, int64_t ldc, int64_t gs) { return ldc % 8 == 0 && gs % 8 == 0 && (reinterpret_cast<uintptr_t>(C) & 15) == 0; }
// A product that needs the kernels compiled for any form (see gemm_tile).
bool any_form(const GemmParams& p) { return p.bias || p.act || p.C2 || (p.partial && p.splits <= 1) || !vector_rows(p.C, p.ldc, p.c_gstride); }

template <int BN>
cudaError_t launch_gemm(const CUtensorMap& ta, const CUtensorMap& tb, const GemmParams& p, dim3 grid,
                        cudaStream_t stream) {
    cudaError_t e = cudaSuccess;
    if (any_form(p)) {
        e = launch_gemm_any(BN, grid, gemm_smem(BN, p.num_stages), stream, ta, tb, p);
    } else {
        e = allow_smem(tc_gemm_kernel<BN, false, false>, gemm_smem(BN, kMaxStages));
        if (e == cudaSuccess)
            e = launch_overlapped(tc_gemm_kernel<BN, false, false>, grid, dim3(kGemmThreads), gemm_smem(BN, p.num_stages), stream, ta, tb, p);
    }
    if (e == cudaSuccess) count_launch();
    return e;
}

// Workspace floats of a product's slices: one 128 x bn block per (tile, slice).
size_t slice_bytes(int64_t M, int64_t N, int splits) {
    const int bn = N <= 64 ? 64 : 128;
    return static_cast<size_t>(ceil_div(M, kBM) * ceil_div(N, bn)) * std::max(1, splits) * kBM * bn * 4;
}
size_t partial_bytes(int64_t M, int64_t N, int splits) { return splits <= 1 ? 0 : slice_bytes(M, N, splits); }      // a split product
// Where a product may leave its slices, and how many bytes it may use there.
struct SliceRoom {
    float* p = nullptr;
    size_t bytes = 0;
};

// What a block that is alone on its SM spends on kb k-blocks of a contraction cut into s slices, beyond its start and
// end: 0.16 us per k-block on warm caches, 0.3 on cold ones, and for the sum of the slices 5 us at two slices, 4.2 at
// four, 3.8 at eight (the fewer slices, the larger the share that a block sums).  So short contractions stay whole:
// 1024 x 256 over 512: 9.3 us in two slices, 4.8 whole; over 1024: 8.4 in four, 6.0 whole; over 2048: 8.4 in eight, 8.4
// whole; over 4096: 9.3 in eight, 13.0 whole.  (dU of 26 x 7 x 7, 160 -> 40 -> 160 over 26 blocks of 49 pixels: backward 13.8 us
// split, 16.0 whole; of 16 x 14 x 14, stride 2, over 16: 12.8 and 9.8.)
// What a whole contraction costs is exactness of the sum, which tensor memory truncates: dV = dY^T T of 512 -> 128 -> 512 in fp32
// against 64 bits, 1000 rows: relative error 9.7e-7 whole, 1.0e-7 in sixteen slices; 512 rows 4.7e-7 and 0.9e-7 (8192 rows of 1024 ->
// 256 -> 4096, two slices: 4.4e-6).  It does not show in the gradients of the layer, whose T and G are rounded to bf16: 1000
// rows, fp32 dU and dV are off by 1.6625e-3 and 1.6439e-3 whole, 1.6625e-3 and 1.6442e-3 in slices; stored in bf16 by 2.34e-3.
constexpr double kBlockUs = 0.23;
double slice_us(int64_t nkb, int64_t s) {
    return kBlockUs * static_cast<double>(ceil_div(nkb, s)) + (s > 1 ? 3.4 + 3.4 / static_cast<double>(s) : 0.0);
}
// Slices of a contraction that is alone in its launch.
int slices_of(int64_t tiles, int64_t nkb) {
    if (tiles < 1 || nkb < 1) return 1;
    const int64_t s = std::min<int64_t>(64, std::min(num_sms() / tiles, nkb / 4));     // at least 4 k-blocks per slice
    return s > 1 && slice_us(nkb, s) < slice_us(nkb, 1) ? static_cast<int>(s) : 1;
}
int pick_splits(int64_t M, int64_t N, int bn, int64_t K) { return slices_of(ceil_div(M, kBM) * ceil_div(N, bn), ceil_div(K, kBK)); }
int pick_bn(int64_t N) { return N <= 64 ? 64 : 128; }

// Slice counts for two products that share one launch (dU: Mu x N over nkb_u k-blocks, dV: Mv x N over nkb_v):
// all CTAs should fit one wave and finish together, so the time of the longest CTA is
// minimised subject to tiles_u * su + tiles_v * sv <= SM count.
void pick_pair_splits(int64_t Mu, int64_t Mv, int64_t N, int64_t nkb_u, int64_t nkb_v, int* su, int* sv, int groups = 1) {
    const int bn = pick_bn(N);
    const int64_t tu = ceil_div(Mu, kBM) * ceil_div(N, bn) * groups, tv = ceil_div(Mv, kBM) * ceil_div(N, bn) * groups;
    *su = 1; *sv = 1;
    if (tu < 1 || tv < 1 || nkb_u < 1 || nkb_v < 1 || tu + tv > num_sms()) return;
    double best = std::max(slice_us(nkb_u, 1), slice_us(nkb_v, 1));
    if (best < slice_us(1, 64)) return;      // shorter than any sum of slices
    auto consider = [&](int64_t a) {         // a slices of dU, and what is left of the machine to dV; true: dU is not the longer one
        const double u = slice_us(nkb_u, a);
        const int64_t most = std::min(std::min<int64_t>(64, nkb_v), (num_sms() - tu * a) / tv);
        const double whole = slice_us(nkb_v, 1), cut = slice_us(nkb_v, most), v = std::min(whole, cut);
        if (std::max(u, v) < best) {
            best = std::max(u, v);
            *su = static_cast<int>(a);
            *sv = static_cast<int>(cut < whole ? most : 1);
        }
        return u <= v;
    };
    consider(1);
    // from two slices on, more slices shorten dU and lengthen dV: the best count is where the two meet
    int64_t lo = 2, hi = std::min(std::min<int64_t>(64, nkb_u), (num_sms() - tv) / tu);
    if (lo > hi) return;
    while (lo < hi) {
        const int64_t mid = (lo + hi) / 2;
        if (consider(mid)) hi = mid; else lo = mid + 1;
    }
    consider(lo);
    if (lo > 2) consider(lo - 1);
}

// Slices of dU (k x r) and dV (n x r) in the backward of the linear layer, and whether dV runs BESIDE
// the fused dX kernel instead of after it.  dV = dY^T T needs nothing that kernel writes.  When the
// contraction of the fused kernel's first product is long against its output (n >= 2k), that kernel is
// left unsplit (one block per 128-row tile, no block repeats another's first product), which leaves
// SMs free; the dV blocks are sized to exactly those SMs, come first in their launch and do not wait
// for the fused kernel, and the dU blocks (which need G) follow on the other SMs once that kernel's
// blocks retire.  (Measured on the Transformer-FFN shapes: doing the same for n < 2k, where only the
// 20 SMs the split fused kernel leaves idle are free, loses more through the long dV blocks than the
// overlap gains.)
void bwd_split_plan(int64_t m, int64_t k, int64_t n, int64_t r, bool fused_dx, int* su, int* sv, bool* beside) {
    // Unfused, each shares a launch with a product that waits for nothing (see linear_bwd), so each may fill the machine by
    // itself, also where the tiles of both do not fit it together.  Backward with both whole there / split: 8192 x 1504 -> 376 ->
    // 6016: 161 / 146 us, 8192 x 768 -> 768 -> 3072: 106 / 86, 11209 x 3072 -> 768 -> 768: 139 / 114, 4096 x 1024 -> 1024 -> 4096:
    // 75.5 / 74.1.
    if (!fused_dx) {
        *su = pick_splits(k, r, pick_bn(r), m);
        *sv = pick_splits(n, r, pick_bn(r), m);
        *beside = false;
        return;
    }
    pick_pair_splits(k, n, r, ceil_div(m, kBK), ceil_div(m, kBK), su, sv);
    *beside = false;
    if (n < 2 * k) return;
    const int bn = pick_bn(r);
    const int64_t row_tiles = ceil_div(m, kBM), nkb = ceil_div(m, kBK);
    const int64_t tu = ceil_div(k, kBM) * ceil_div(r, bn), tv = ceil_div(n, kBM) * ceil_div(r, bn);
    const int64_t free_sms = num_sms() - row_tiles;
    const int64_t smax = std::max<int64_t>(1, std::min<int64_t>(64, nkb / 4));
    if (free_sms < tv || tu > kFixTiles || tv > kFixTiles) return;
    const int64_t b = std::min(free_sms / tv, smax);
    // dU gets the SMs that dV does not hold: dV may still be running when the fused kernel retires
    const int64_t a = std::min((num_sms() - tv * b) / tu, smax);
    if (a < 1 || b < 1) return;
    // ... unless too few SMs are left: dV has to be done with about when the fused kernel is (16384 rows, 512 -> 128 -> 2048, 16
    // of the 20 free SMs: 84 us beside, 38.5 behind; 256 -> 32 -> 1024: 32.1 and 23.7)
    const double chain_us = 3.8 + 0.31 * static_cast<double>(ceil_div(n, kBK)) + 0.65 * static_cast<double>(ceil_div(k, 128));
    if (slice_us(nkb, b) > 1.5 * chain_us) return;
    *su = static_cast<int>(a);
    *sv = static_cast<int>(b);
    *beside = true;
}

struct ConvA {
    int mode;                   // 1: dX (A = dT image), 2: dU (A = x image)
    int N, H, W, C, R, Ho, Wo, kh, kw, pad, stride;     // the layer
};
// Blocks of output pixels that the contraction of dU runs over, and of the pixels of one class that dX covers.
ConvTiling conv_k_tiling(const ConvA& c) { return conv_tiling(c.N, c.Ho, c.Wo, kBK); }
ConvTiling conv_dx_tiling(const ConvA& c) {
    return conv_tiling(c.N, static_cast<int>(ceil_div(c.H, c.stride)), static_cast<int>(ceil_div(c.W, c.stride)), kBM);
}
// Row tiles of dU: pairs of 64-channel blocks of the unrolled factor.
int64_t conv_du_tiles(int kh, int kw, int C) { return ceil_div(static_cast<int64_t>(kh) * kw * ceil_div(C, 64), 2); }

struct GemmLaunch {
    CUtensorMap ta, tb;
    GemmParams p;
    dim3 grid;
    int bn;
    bool runs = false;       // several tiles per block (plain product, K-major A and MN-major B)
    bool straddles = false, warm = false;     // A's rows do not start on 128-byte lines; see Operand
};

// Bytes of the slices of a prepared product.
size_t slices_of_launch(const GemmParams& p) {
    return static_cast<size_t>(p.tiles_x) * p.tiles_y * std::max(1, p.groups) * std::max(1, p.splits) * kBM * p.bn * 4;
}

// Encodes the tensor maps and launch geometry of C[M,N] = A * B without launching.  A contraction whose slices do not fit `room`
// is refused.
int gemm_prepare(const Operand& A, const Operand& B, int64_t M, int64_t N, int64_t K, void* C, int64_t ldc,
                 int splits, SliceRoom room, const ConvA* cv, GemmLaunch* out, const Grouping* gr = nullptr) {
    if (M > 0x7fffffff || N > 0x7fffffff || K > 0x7fffffff) return PF_ERR_UNSUPPORTED;
    const int groups = gr ? gr->groups : 1;
    const bool sum_groups = gr && gr->sum_groups;
    if (gr && (cv || groups < 1 || groups > 1024 || (sum_groups && (A.mn_major || B.mn_major)))) return PF_ERR_UNSUPPORTED;
    const int bn = pick_bn(N);
    CUtensorMap& ta = out->ta;
    CUtensorMap& tb = out->tb;
    bool oka, okb;
    ConvTiling ct;
    if (cv && cv->mode == 1) {
        ct = conv_dx_tiling(*cv);
        oka = cached_map_nhwc(&ta, A.p, cv->N, cv->Ho, cv->Wo, cv->R, static_cast<int>(ceil_div(cv->W, cv->stride)), ct.bh, ct.nb, 1, A.ld);
        okb = cached_map_2d(&tb, B.p, static_cast<int64_t>(cv->kh) * cv->kw * cv->C, cv->R, B.ld, bn);   // rows past a tap's C: columns past N
    } else if (cv && cv->mode == 2) {
        ct = conv_k_tiling(*cv);
        oka = cached_map_nhwc(&ta, A.p, cv->N, cv->H, cv->W, cv->C, cv->Wo, ct.bh, ct.nb, cv->stride, A.ld);
        okb = cached_map_nhwc(&tb, B.p, cv->N, cv->Ho, cv->Wo, cv->R, cv->Wo, ct.bh, ct.nb, 1, B.ld);
    } else if (gr) {
        const int64_t ga = A.gs == 0 ? 1 : groups, gb = B.gs == 0 ? 1 : groups;
        oka = A.mn_major ? cached_map_3d(&ta, A.p, ga, K, M, A.ld, A.gs, 64) : cached_map_3d(&ta, A.p, ga, M, K, A.ld, A.gs, kBM);
        okb = B.mn_major ? cached_map_3d(&tb, B.p, gb, K, N, B.ld, B.gs, 64) : cached_map_3d(&tb, B.p, gb, N, K, B.ld, B.gs, bn);
    } else {
        oka = A.mn_major ? cached_map_2d(&ta, A.p, K, M, A.ld, 64) : cached_map_2d(&ta, A.p, M, K, A.ld, kBM);
        okb = B.mn_major ? cached_map_2d(&tb, B.p, K, N, B.ld, 64) : cached_map_2d(&tb, B.p, N, K, B.ld, bn);
    }
    if (!oka || !okb) return PF_ERR_CUDA;
    GemmParams& p = out->p;
    p.M = static_cast<int>(M); p.N = static_cast<int>(N); p.K = static_cast<int>(K);
    p.a_mn = A.mn_major; p.b_mn = B.mn_major;
    p.C = C; p.ldc = ldc;
    p.C2 = nullptr; p.ldc2 = 0; p.c2_gstride = 0;
    p.bias = nullptr; p.act = 0;
    p.conv_mode = 0; p.cv_blks = 1; p.cv_kw = 1; p.cv_kh = 1; p.cv_pad = 0; p.cv_stride = 1; p.cv_C = 1; p.cv_bh = 1; p.cv_nb = 1;
    p.cv_tpi = 1; p.cv_N = p.cv_H = p.cv_W = p.cv_bw = p.cv_inv_bw = p.cv_inv_bh = p.cv_tiles_class = 1; p.cv_blocks = 0;
    p.rows_tile = kBM; p.kpix = kBK; p.ksteps = kBK / 16;
    int64_t row_tiles = ceil_div(M, kBM);
    if (cv) {
        p.conv_mode = cv->mode; p.cv_kw = cv->kw; p.cv_kh = cv->kh; p.cv_pad = cv->pad; p.cv_stride = cv->stride; p.cv_C = cv->C;
        p.cv_bh = ct.bh; p.cv_nb = ct.nb; p.cv_tpi = ct.tpi; p.cv_N = cv->N; p.cv_H = cv->H; p.cv_W = cv->W;
        if (cv->mode == 1) {
            p.cv_blks = static_cast<int>(ceil_div(cv->R, 64));
            p.cv_bw = static_cast<int>(ceil_div(cv->W, cv->stride));
            p.cv_inv_bw = 65535 / p.cv_bw + 1;
            p.cv_inv_bh = 65535 / p.cv_bh + 1;
            p.cv_tiles_class = static_cast<int>(ct.blocks);
            p.rows_tile = ct.pixels;
            if (cv->R < kBK) p.ksteps = static_cast<int>(ceil_div(cv->R, 16));
            row_tiles = ct.blocks * cv->stride * cv->stride;
        } else {
            p.cv_blks = static_cast<int>(ceil_div(cv->C, 64));
            p.cv_blocks = cv->kh * cv->kw * p.cv_blks;
            p.kpix = ct.pixels;
            p.ksteps = static_cast<int>(ceil_div(ct.pixels, 16));
            row_tiles = conv_du_tiles(cv->kh, cv->kw, cv->C);
        }
    }
    p.groups = gr ? groups : 1;
    p.a_shared = gr && A.gs == 0; p.b_shared = gr && B.gs == 0;
    p.c_gstride = gr ? gr->c_gs : 0;
    p.kb_per_group = 0;
    int64_t nkb = ceil_div(K, kBK);
    if (cv) nkb = cv->mode == 2 ? ct.blocks : static_cast<int64_t>(cv->kh) * cv->kw * p.cv_blks;   // (dX: at most, the kernel counts per class)
    if (sum_groups) {                       // the groups are part of the contraction: one output
        p.kb_per_group = static_cast<int>(nkb);
        nkb *= groups;
        p.groups = 1;
    }
    const int out_groups = sum_groups ? 1 : groups;
    p.nkb_total = static_cast<int>(nkb);
    p.kb_per_split = static_cast<int>(ceil_div(nkb, splits < 1 ? 1 : splits));
    p.splits = static_cast<int>(ceil_div(nkb, p.kb_per_split));   // every slice gets >= 1 k-block
    p.status = device_status_ptr();
    dim3 grid(static_cast<unsigned>(row_tiles), static_cast<unsigned>(ceil_div(N, bn)),
              static_cast<unsigned>(p.splits * out_groups));
    if (grid.y > 65535 || grid.z > 65535) return PF_ERR_UNSUPPORTED;
    p.tiles_x = static_cast<int>(grid.x);
    p.tiles_y = static_cast<int>(grid.y);
    p.bn = bn;
    const bool dx = p.conv_mode == 1;
    if (dx) grid = dim3(run_blocks(static_cast<int64_t>(p.tiles_x) * p.tiles_y, nkb / (cv->stride * cv->stride), cv->stride));
    p.num_stages = pick_stages(bn, static_cast<int64_t>(grid.x) * grid.y * grid.z, dx);
    p.counters = nullptr;
    p.partial = p.splits > 1 ? room.p : nullptr;
    p.independent = 0;
    p.early = (A.early ? kEarlyA : 0) | (B.early ? kEarlyB : 0);
    p.keep_a = 0.f;
    if (p.splits > 1) {
        // the CTAs of a tile wait for one another, so all of them must be resident at once
        if (static_cast<int64_t>(grid.x) * grid.y * out_groups > kFixTiles || static_cast<int64_t>(grid.x) * grid.y * grid.z > num_sms() ||
            room.p == nullptr || slices_of_launch(p) > room.bytes)
            return PF_ERR_UNSUPPORTED;
        p.counters = split_counters();
        if (!p.counters) return PF_ERR_CUDA;
    }
    out->grid = grid;
    out->bn = bn;
    out->straddles = A.ld % 64 != 0;
    out->warm = A.warm;
    return PF_OK;
}

// Launches one prepared product on its own.
int launch_prepared(const GemmLaunch& g, cudaStream_t stream) {
    if (g.runs) {
        if (launch_gemm_runs(g.bn, g.grid, gemm_smem(g.bn, g.p.num_stages, true), stream, g.ta, g.tb, g.p) != cudaSuccess) return PF_ERR_CUDA;
        count_launch();
        return PF_OK;
    }
    const cudaError_t e = g.bn == 64 ? launch_gemm<64>(g.ta, g.tb, g.p, g.grid, stream) : launch_gemm<128>(g.ta, g.tb, g.p, g.grid, stream);
    return e == cudaSuccess ? PF_OK : PF_ERR_CUDA;
}

// One launch for up to three prepared products.  Products whose contraction is split must come
// first and fit the machine together (their CTAs wait for one another); tiles are 64 or 128 wide.
int gemm_multi(const GemmLaunch* const* g, int count, cudaStream_t stream) {
    if (count < 1 || count > 3) return PF_ERR_UNSUPPORTED;
    int ctas[3] = {0, 0, 0};
    int total = 0, split_ctas = 0;
    bool seen_plain = false;
    for (int i = 0; i < count; ++i) {
        ctas[i] = static_cast<int>(g[i]->grid.x * g[i]->grid.y * g[i]->grid.z);
        total += ctas[i];
        if (g[i]->p.splits > 1) {
            if (seen_plain) return PF_ERR_UNSUPPORTED;
            split_ctas += ctas[i];
        } else {
            seen_plain = true;
        }
    }
    // The blocks of a split product wait for one another and must be resident together.  A first
    // product marked independent never waits for anything later in the launch and is dispatched
    // first, so it only has to fit by itself, and the products behind it by themselves.
    const bool lead = count > 1 && g[0]->p.independent && g[0]->p.splits > 1;
    const int resident = lead ? std::max(ctas[0], split_ctas - ctas[0]) : split_ctas;
    if (resident > num_sms()) return PF_ERR_UNSUPPORTED;
    const int wave = lead ? std::max(ctas[0], total - ctas[0]) : total;
    GemmParams prm[3];
    size_t smem = 0;
    for (int i = 0; i < 3; ++i) {
        const GemmLaunch* src = g[i < count ? i : 0];
        prm[i] = src->p;
        const bool dx = src->p.conv_mode == 1;
        const int stages = pick_stages(src->bn, wave, dx);
        prm[i].num_stages = stages;
        if (i < count) smem = std::max(smem, gemm_smem(src->bn, stages, dx));
    }
    Gemm3Args k;
    bool conv = false, any = false;
    for (int i = 0; i < 3; ++i) {
        const GemmLaunch* src = g[i < count ? i : 0];
        any = any || any_form(src->p);
        k.ta[i] = src->ta; k.tb[i] = src->tb; k.p[i] = prm[i];
        k.tiles[i] = make_int2(src->grid.x, src->grid.y);
        conv = conv || src->p.conv_mode != 0;
    }
    k.end0 = ctas[0]; k.end1 = ctas[0] + ctas[1];
    cudaError_t e;
    if (any) {
        e = launch_gemm3_any(conv, total, smem, stream, k);
    } else if (conv) {
        e = launch_gemm3_conv(total, smem, stream, k);
    } else {
        e = allow_smem(tc_gemm3_kernel<false, false>, gemm_smem(128, kMaxStages));
        if (e == cudaSuccess)
            e = launch_overlapped(tc_gemm3_kernel<false, false>, dim3(static_cast<unsigned>(total)), dim3(kGemmThreads), smem, stream, k.ta[0], k.tb[0],
                                  k.ta[1], k.tb[1], k.ta[2], k.tb[2], k.p[0], k.p[1], k.p[2], k.end0, k.end1, k.tiles[0], k.tiles[1], k.tiles[2]);
    }
    if (e != cudaSuccess) return PF_ERR_CUDA;
    count_launch();
    return PF_OK;
}

// What the expected time of a product depends on.
struct Work {
    double M, N, kb, blocks;      // kb: k-blocks of a thread block, all of the contraction's where there are no slices
    double alone, beside;         // microseconds per k-block by itself on its SM, and beside another block
    double a_bytes, cold, end;    // end: the sum of slices, rows that take no 16-byte stores
    bool vec;
};
// groups: problems of one shape that the product covers (1 where they are part of the contraction).
Work work_of(int64_t M, int64_t N, int64_t nkb, int splits, int64_t groups, bool a_mn, bool straddles, bool warm, bool vec) {
    Work w;
    const int bn = pick_bn(N);
    const int64_t per = ceil_div(nkb, std::max(1, splits)), s = ceil_div(nkb, std::max<int64_t>(1, per));
    w.M = static_cast<double>(M); w.N = static_cast<double>(N); w.kb = static_cast<double>(per);
    w.blocks = static_cast<double>(ceil_div(M, kBM) * ceil_div(N, bn) * s * groups);
    w.a_bytes = static_cast<double>(M) * static_cast<double>(nkb) * 128.0 * static_cast<double>(groups);
    w.cold = warm && w.a_bytes < 6e7 ? 0.0 : std::min(1.0, w.a_bytes / 16e6);
    const double lines = !straddles ? 1.0 : a_mn ? 1.55 : 1.15;
    w.alone = (0.15 + 0.12 * w.cold) * lines;
    w.beside = (0.33 + 0.28 * w.cold) * lines;
    w.vec = vec;
    w.end = s > 1 ? 3.6 + 3.6 / static_cast<double>(s) : vec ? 0.0 : 3.3;
    return w;
}
// Expected microseconds of one launch of products on single CTAs, and of one product on CTA pairs, fitted to forwards of 559
// shapes on three forms each and backwards of 774 in two or three orders of launches (64 to 32768 rows, widths of 64 to 6912, ranks
// of 8 to 1024), most within 15 %.  A single CTA's 128 x 128 tile alone on its SM: 3.7 us of start and end, 0.15 us per k-block from
// L2 and 0.27 from memory; beside another 4.5 and 0.33 to 0.61, and whole rounds of two blocks per SM where the launch
// is one product.  Rows of A that straddle 128-byte lines are two requests each: 1.55 times that where the contraction runs
// down the rows.  A pair's 256 x 256 tile: 0.27 to 0.32 us per k-block, and 2.3 us of every tile do not hide.  An A that does
// not stay in L2 is read from memory once per column of tiles.
double singles_us(const Work* w, int count) {
    const double sms = num_sms();
    double blocks = 0, load = 0, alone = 0, beside = 0, memory = 0, shortest = 1e30;
    for (int i = 0; i < count; ++i) shortest = std::min(shortest, w[i].kb);
    for (int i = 0; i < count; ++i) {
        blocks += w[i].blocks;
        load += w[i].blocks * (w[i].beside * w[i].kb + 4.5 + w[i].end);
        alone = std::max(alone, w[i].alone * w[i].kb + w[i].end);
        beside = std::max(beside, w[i].beside * shortest + w[i].alone * (w[i].kb - shortest) + w[i].end);
        if (w[i].a_bytes > 6e7) memory += w[i].a_bytes * std::ceil(w[i].N / pick_bn(static_cast<int64_t>(w[i].N))) / 6.7e6;
    }
    double us = 3.7 + alone;
    if (blocks > sms) {
        us = load / (2.0 * sms);
        const int rounds = static_cast<int>(std::ceil(blocks / sms));
        us = std::max(us, count == 1 ? (rounds / 2) * (w[0].beside * w[0].kb + 4.5) + (rounds % 2) * (w[0].alone * w[0].kb + 3.7) : beside + 4.5);
    }
    return std::max(us, memory + 3.7);
}
double pairs_us(const Work* w, int count) {      // unsplit products
    const int pairs = num_sms() / 2;
    double load = 0, longest = 0, tiles = 0, memory = 0;
    for (int i = 0; i < count; ++i) {
        const double per_group = std::ceil(w[i].M / kBM) * std::ceil(w[i].N / pick_bn(static_cast<int64_t>(w[i].N)));
        const double n = std::ceil(w[i].M / 256) * std::ceil(w[i].N / 256) * (w[i].blocks / per_group);
        const double us = (0.265 + 0.055 * w[i].cold) * w[i].kb + (w[i].vec ? 2.25 : 4.9);
        tiles += n;
        load += n * us;
        longest = std::max(longest, us);
        if (w[i].a_bytes > 6e7) memory += w[i].a_bytes * std::ceil(w[i].N / 256) / 6.7e6;
    }
    const double total = count == 1 ? longest * std::ceil(tiles / pairs) : std::max(longest, load / pairs);
    return std::max(total, memory) + 3.85;
}
Work work_of(const GemmLaunch& g) {
    return work_of(g.p.M, g.p.N, g.p.nkb_total, g.p.splits, std::max(1, g.p.groups), g.p.a_mn != 0, g.straddles, g.warm, vector_rows(g.p.C, g.p.ldc, g.p.c_gstride));
}
double single_us(const GemmLaunch* const* g, int count) {
    Work w[3];
    for (int i = 0; i < count; ++i) w[i] = work_of(*g[i]);
    return singles_us(w, count);
}
// The same products on pairs: whole, whatever the slices of the launches on single CTAs.
double pairs_us(const GemmLaunch* const* g, int count) {
    Work w[3];
    for (int i = 0; i < count; ++i)
        w[i] = work_of(g[i]->p.M, g[i]->p.N, g[i]->p.nkb_total, 1, std::max(1, g[i]->p.groups), g[i]->p.a_mn != 0, g[i]->straddles, g[i]->warm,
                       vector_rows(g[i]->p.C, g[i]->p.ldc, g[i]->p.c_gstride));
    return pairs_us(w, count);
}
// One launch of up to three products on single CTAs (one launch each where they cannot share it).
int launch_singles(const GemmLaunch* const* g, int count, cudaStream_t stream) {
    if (count == 1) return launch_prepared(*g[0], stream);
    const GemmLaunch* list[3];
    int n = 0;
    for (int i = 0; i < count; ++i) list[n++] = g[i];
    // split products first, then the longest tiles (backward of 1000 x 512 -> 128 -> 512, dX of 2 k-blocks in
    // front of dU of 16: 12.5 us, behind it 11.8)
    std::stable_sort(list, list + n, [](const GemmLaunch* x, const GemmLaunch* y) {
        return (x->p.splits > 1) != (y->p.splits > 1) ? x->p.splits > 1 : x->p.kb_per_split > y->p.kb_per_split;
    });
    int st = gemm_multi(list, count, stream);
    for (int i = 0; st == PF_ERR_UNSUPPORTED && i < count; ++i) {
        const int one = launch_prepared(*list[i], stream);
        if (one != PF_OK) return one;
        if (i + 1 == count) return PF_OK;
    }
    return st;
}
constexpr double kPairMargin = 0.9;      // pairs have to be expected so much faster (the expectation is off by up to 15 %)
// One launch of one or two products, on whichever form is expected to be faster.  The products are independent of
// each other; jobs[i] describes the same product as *g[i].  pair_extra: microseconds that the caller has to spend after
// pairs only; *pairs tells which form it was.
int launch_faster(const GemmLaunch* const* g, const PairJob* jobs, int count, cudaStream_t stream, double pair_extra = 0.0,
                  bool* pairs = nullptr) {
    if (pairs_us(g, count) + pair_extra < kPairMargin * single_us(g, count)) {
        PairJob order[2] = {jobs[0], jobs[count > 1 ? 1 : 0]};
        auto kb = [](const PairJob& j) { return ceil_div(j.K, 64) * (j.sum_groups ? j.groups : 1); };
        if (count > 1 && kb(order[1]) > kb(order[0])) std::swap(order[0], order[1]);     // long tiles first
        const int st = gemm_pairs(order, count, 1, stream);
        if (st != PF_ERR_UNSUPPORTED) {
            if (pairs) *pairs = true;
            return st;
        }
    }
    return launch_singles(g, count, stream);
}
// One launch of up to three products on single CTAs, or the first of them on CTA pairs by itself and then the others.
int launch_with(const GemmLaunch* const* g, const PairJob* first, int count, cudaStream_t stream) {
    if (pairs_us(g, 1) + single_us(g + 1, count - 1) < kPairMargin * single_us(g, count)) {
        const int st = gemm_pairs(first, 1, 1, stream);
        if (st == PF_OK) return launch_singles(g + 1, count - 1, stream);
        if (st != PF_ERR_UNSUPPORTED) return st;
    }
    return launch_singles(g, count, stream);
}

// Prepares a product, unsplit where its slices do not fit their room, the counters or the machine.
int gemm_prepare_any(const Operand& A, const Operand& B, int64_t M, int64_t N, int64_t K, void* C, int64_t ldc, int splits, SliceRoom room,
                     const ConvA* cv, GemmLaunch* out) {
    const int st = gemm_prepare(A, B, M, N, K, C, ldc, splits, room, cv, out);
    return st == PF_ERR_UNSUPPORTED && splits > 1 ? gemm_prepare(A, B, M, N, K, C, ldc, 1, {}, cv, out) : st;
}
// One product in a launch of its own.  `copy2` (optional): asks for a second copy of C at pitch ldc2; *copy2_done tells
// whether the launch wrote it (the CTA-pair kernel cannot), else the caller copies C itself.
int gemm(const Operand& A, const Operand& B, int64_t M, int64_t N, int64_t K, void* C, int64_t ldc,
         int splits, SliceRoom room, cudaStream_t stream, void* copy2 = nullptr, int64_t ldc2 = 0, bool* copy2_done = nullptr,
         const void* bias = nullptr, int act = 0) {
    GemmLaunch g;
    const int st = gemm_prepare_any(A, B, M, N, K, C, ldc, splits, room, nullptr, &g);
    if (st != PF_OK) return st;
    if (copy2) {
        g.p.C2 = copy2; g.p.ldc2 = ldc2;
    }
    g.p.bias = bias; g.p.act = act;               // (given for unsplit products only)
    PairJob j{A.p, A.ld, A.mn_major, 0, B.p, B.ld, B.mn_major, 0, M, N, K, C, ldc};
    j.bias = bias;
    j.act = act;
    j.a_early = A.early;
    j.b_early = B.early;
    const GemmLaunch* const list[1] = {&g};
    bool pairs = false;
    const int rc = launch_faster(list, &j, 1, stream, copy2 ? 6.0 : 0.0, &pairs);
    if (copy2_done) *copy2_done = copy2 != nullptr && !pairs;
    return rc;
}

// A row-major bf16 matrix that TMA must read: used as is when 16-byte aligned with a pitch that is
// a multiple of 8 elements, otherwise copied to `scratch` with the pitch rounded up.
struct Staged {
    const void* p;
    int64_t ld;
    bool copied = false;
};
// Pitch of a matrix in the workspace: whole 128-byte lines, so that no 128-byte row of a TMA box touches two of them (narrow
// rows: whole 16-byte pieces).  8 x (700 x 1500 -> 1500), r 375: forward 43.7 -> 37.5 us, backward 81.0 -> 62.5, against
// pitches of 376 and 1504 elements; 3000 x 2000 -> 500 -> 500: 28.7 -> 24.4 and 48.8 -> 39.7.
int64_t row_pitch(int64_t v, bool tight = false) { return v > 32 && !tight ? (v + 63) / 64 * 64 : (v + 7) / 8 * 8; }

// The re-pitch copies of one call are collected and issued as one launch.
struct RepackList {
    RepackJob jobs[6];
    int count = 0;
    int flush(cudaStream_t stream) {
        const cudaError_t e = count > 0 ? repack_rows_bf16_multi(jobs, count, stream) : cudaSuccess;
        count = 0;
        return e == cudaSuccess ? PF_OK : PF_ERR_CUDA;
    }
};

// returns 0 = usable, 1 = needs repack but no room reserved (decline), <0 never
int stage_operand(const void* p, int64_t ld, int64_t rows, int64_t cols, char*& scratch, Staged* out, RepackList* list, bool tight = false) {
    if (tma_ok(p, ld)) { out->p = p; out->ld = ld; return 0; }
    if (cols % 8 == 0) return 1;   // the workspace query reserves repack room only for ragged widths
    const int64_t ldp = row_pitch(cols, tight);
    list->jobs[list->count++] = RepackJob{p, ld, scratch, ldp, rows, cols};
    out->p = scratch; out->ld = ldp; out->copied = true;
    scratch += align_up(static_cast<size_t>(rows) * ldp * 2, 256);
    return 0;
}
// The backward's fused chain pays off once there are enough 128-row tiles to fill the machine, and while the
// rank is small enough for the layer to be bound by memory traffic: from r = 256 up the two
// products are tensor-bound and run faster unfused on CTA pairs (the intermediate is only m x r).
bool use_chain(int64_t m, int64_t r) { return m >= 2048 && r <= 192; }
// Batches that just fill a few SMs per row tile, with the longer contraction in the fused kernel's first product, which a block
// contracts alone: 2048 x 512 -> 128 -> 2048: 22.0 us fused, 18.3 unfused; 3000: 22.3 and 19.8; 4096: 23.2 and 22.2; 2048 x 1024 ->
// 64 -> 1024: 15.9 and 14.9; but 2048 x 2048 -> 128 -> 512: 17.6 and 19.4, 2048 x 768 -> 192 -> 768: 18.9 and 20.5.
bool unfused_backward(int64_t m, int64_t k, int64_t n, int64_t r) { return m < 3500 && n >= k && n >= 1024 && r <= 128; }
// The forward's fused kernel is one launch instead of two, so it takes smaller batches too, while its first product, which
// one block contracts alone where the unfused one is split over the SMs, is short.  Fused against unfused, caches warm:
// 300 x 512 -> 128 -> 2048: 6.4 against 8.7 us; 1000 x 1536 -> 128 -> 1536: 10.5 / 11.7; 500 x 2048 -> 128 -> 2048: 11.7 / 11.7;
// 1024 x 4096 -> 128 -> 1024: 18.6 / 12.1; r 256, 1024 x 1024 -> 1024: 11.8 / 10.3.  Up to 32 rows against the kernels of
// pf_small.cu: 20 x 512 -> 128 -> 2048: 5.9 / 6.8; 8 x 1024 -> 64 -> 1024: 6.5 / 5.4.  A stash that TMA cannot write would take
// a launch of its own again.  Rows that do not start on 128-byte lines cost two lines per row of a box: 500 x 1480 -> 120 ->
// 1480: 14.5 / 12.4; 400 x 1096 -> 136 -> 4384: 16.9 / 14.5; 1000 x 1336 -> 80 -> 344: 11.4 / 14.1.
bool short_first_product(int64_t k, int64_t r, int64_t ldx, int64_t ldu, int64_t most) {
    const int64_t lines = 128 * (ldx % 64 ? 2 : 1) + ceil_div(r, 64) * 64 * (ldu % 64 ? 2 : 1);      // of a k-block
    return k <= most && ceil_div(k, kBK) * lines <= 11000;
}
double streamed_bytes(int64_t m, int64_t k, int64_t n) { return static_cast<double>(m) * static_cast<double>(k + n) * 2.0; }
// Whether a fused launch streams more than L2 holds: its output is then the first to leave L2, and so is an operand's row once
// read.  (An output that fits stays, for whoever reads it next.)
bool beyond_l2(int64_t m, int64_t k, int64_t n) { return streamed_bytes(m, k, n) > kL2Bytes; }
bool use_chain_fwd(const LinearArgs& a) {
    if (a.r > 192 || !tma_out(a.y, a.ldy, a.n)) return false;
    // (rows of 16 bytes, eight to a line that every block asks for: 2000 x 1024 -> 8 -> 1024: 17.9 us, unfused 13.5; of 32 bytes: 12.0 and 12.3;
    // 2000 x 512 -> 8 -> 512: 9.0 and 12.7; 1400 x 512 -> 8 -> 2048: 12.3 and 13.6)
    if (!a.tight && a.r <= 8 && a.n >= 1024 && a.n < 2048 && a.m > 1024 && a.m < 2048) return false;
    // (operands that are copied first arrive on whole lines)
    return a.m >= 2048 || (short_first_product(a.k, a.r, tma_ok(a.x, a.ldx) ? a.ldx : 0, tma_ok(a.U, a.ldu) ? a.ldu : 0, 1536) && (!a.T || tma_out(a.T, a.ldt, a.r)));
}

size_t repack_room(int64_t rows, int64_t cols, bool tight = false) {
    return cols % 8 == 0 ? 0 : align_up(static_cast<size_t>(rows) * row_pitch(cols, tight) * 2, 256);
}

// Whether the tiles of dU (rows_u x r) and dV (rows_v x r) fit the machine together.  Such reductions run on single CTAs,
// split or whole, and can leave their fp32 slices to a call that wants unrounded gradients.
bool narrow_reductions(int64_t rows_u, int64_t rows_v, int64_t r) {
    return (ceil_div(rows_u, kBM) + ceil_div(rows_v, kBM)) * ceil_div(r, pick_bn(r)) <= num_sms();
}
// Room for the fp32 slices of dU and dV under either backward structure (which one a call takes depends on pointers the
// workspace query does not see).  Reductions that do not fit the machine together may each be split by themselves (they
// share their launches with other products); only narrow ones leave one slice.
void bwd_partial_bytes(int64_t m, int64_t k, int64_t n, int64_t r, size_t* bytes_u, size_t* bytes_v) {
    int su, sv, su2, sv2;
    bool beside;
    bwd_split_plan(m, k, n, r, false, &su, &sv, &beside);
    bwd_split_plan(m, k, n, r, true, &su2, &sv2, &beside);
    su = std::max(su, su2);
    sv = std::max(sv, sv2);
    pick_pair_splits(k, n, r, ceil_div(m, kBK), ceil_div(m, kBK), &su2, &sv2);
    const auto bytes = narrow_reductions(k, n, r) ? slice_bytes : partial_bytes;
    *bytes_u = align_up(bytes(k, r, std::max(su, su2)), 256);
    *bytes_v = align_up(bytes(n, r, std::max(sv, sv2)), 256);
}
// ... and for those of the m x r products (x U and, backward, dY V), one after the other.
size_t first_partial_bytes(int64_t m, int64_t k, int64_t n, int64_t r, bool bwd) {
    const int s = std::max(pick_splits(m, r, pick_bn(r), k), bwd ? pick_splits(m, r, pick_bn(r), n) : 1);
    return align_up(partial_bytes(m, r, s), 256);
}
// Where a prepared reduction leaves its fp32 slices; an unsplit one is told to leave its one slice.
void keep_slices(LinearArgs::Slices* out, GemmLaunch* g, SliceRoom room, int conv_c = 0) {
    if (!out) return;
    *out = LinearArgs::Slices();
    if (!room.p || slices_of_launch(g->p) > room.bytes) return;
    g->p.partial = room.p;
    out->partial = room.p; out->splits = g->p.splits; out->bn = g->bn;
    out->tiles_x = static_cast<int>(g->grid.x); out->tiles_y = static_cast<int>(g->grid.y); out->conv_c = conv_c;
}

}  // namespace

// Device address of the counter set a launch may use (sets rotate, so that launches in flight on
// different streams do not share counters unless more than kFixSlots of them overlap).
unsigned int* split_counters() {
    static unsigned int* base[64] = {};
    static std::atomic<unsigned int> next{0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    if (!base[dev]) {
        void* ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_fix_counters) != cudaSuccess) return nullptr;
        base[dev] = static_cast<unsigned int*>(ptr);
    }
    return base[dev] + static_cast<size_t>(next.fetch_add(1) % kFixSlots) * (kFixTiles * 2);
}

// Extra workspace of the tensor-core linear path: repack buffers for operands whose width is not a
// multiple of 8 elements (TMA needs 16-byte row pitches), the two m x r intermediates at a padded
// pitch, and split partials of dU / dV.
size_t linear_extra_workspace(int64_t m, int64_t k, int64_t n, int64_t r, bool bwd) {
    size_t b = 0;
    b += repack_room(m, k) + repack_room(k, r) + repack_room(n, r);        // x, U, V
    b += align_up(static_cast<size_t>(m) * row_pitch(r) * 2, 256);               // T at padded pitch
    if (bwd) {
        b += repack_room(m, n);                                             // dY
        b += align_up(static_cast<size_t>(m) * row_pitch(r) * 2, 256);           // G at padded pitch
        // slices for either backward structure (the choice depends on pointers the query does not see)
        size_t bu, bv;
        bwd_partial_bytes(m, k, n, r, &bu, &bv);
        b += bu + bv;
    }
    // skinny batches: the m x r products (x U, dY V) are split over their contraction to fill the SMs
    return b + first_partial_bytes(m, k, n, r, bwd);
}

// Bytes of `a.ws` that linear_fwd(a) will really touch for these pointers and sizes (it takes the
// same decisions in the same order), and whether it will handle the call at all.  The public
// workspace query cannot see pointers and pitches and therefore reserves for every path.
size_t linear_fwd_need(const LinearArgs& a, bool* handles) {
    *handles = false;
    if (encode_fn() == nullptr) return 0;
    if (a.k > (1 << 22) || a.n > (1 << 22) || a.r > (1 << 22)) return 0;
    size_t room = 0;
    const struct { const void* p; int64_t ld, rows, cols; } ops[3] = {
        {a.x, a.ldx, a.m, a.k}, {a.U, a.ldu, a.k, a.r}, {a.V, a.ldv, a.n, a.r}};
    for (const auto& o : ops) {
        if (tma_ok(o.p, o.ld)) continue;
        if (o.cols % 8 == 0) return 0;               // declined: FMA kernels
        room += repack_room(o.rows, o.cols, a.tight);
    }
    *handles = true;
    const size_t t_bytes = align_up(static_cast<size_t>(a.m) * row_pitch(a.r, a.tight) * 2, 256);
    ChainPlan plan;
    if (use_chain_fwd(a) && chain_plan(a.m, a.k, a.n, a.r, true, &plan))
        return room + (a.T && !tma_out(a.T, a.ldt, a.r) ? t_bytes : 0);
    return room + t_bytes + (a.whole ? 0 : first_partial_bytes(a.m, a.k, a.n, a.r, false));
}

// The fused kernel needs no room for x U, however many rows there are, and only its stores keep rows that end inside a 16-byte piece
// from it.  In a workspace of a given size such a call runs on the products that take them, so many rows at a time as fit:
// how many (0: it is no such call), where *b is how each of these calls is made.
int64_t linear_fwd_rows(const LinearArgs& a, size_t room, LinearArgs* b) {
    ChainPlan plan;
    if (a.r > 192 || !tma_ok(a.y, a.ldy) || (a.n % 8 == 0 && (!a.T || !tma_ok(a.T, a.ldt) || a.r % 8 == 0))) return 0;
    if (a.m < 2048 && !(short_first_product(a.k, a.r, tma_ok(a.x, a.ldx) ? a.ldx : 0, tma_ok(a.U, a.ldu) ? a.ldu : 0, 1536) && (!a.T || tma_ok(a.T, a.ldt)))) return 0;
    if (!chain_plan(a.m, a.k, a.n, a.r, true, &plan)) return 0;
    *b = a;
    b->tight = b->whole = true;
    for (int64_t rows = a.m;; rows = ceil_div(ceil_div(rows, 2), kBM) * kBM) {      // (whole tiles: blocks start where TMA takes them)
        bool handles = false;
        b->m = rows;
        const size_t need = linear_fwd_need(*b, &handles);
        if (!handles) return 0;
        if (rows == a.m && !tma_ok(a.x, a.ldx)) {      // what the fused kernel would need, the copies of all rows, has to fit behind x U
            const size_t t_bytes = align_up(static_cast<size_t>(a.m) * row_pitch(a.r, true) * 2, 256), fused = need - (a.T && !tma_ok(a.T, a.ldt) ? 0 : t_bytes);
            if (fused > 0 && align_up(static_cast<size_t>(a.m) * a.r * 2, 256) + fused > room) return 0;
        }
        if (need <= room) return rows;
        if (rows <= kBM) return 0;
    }
}

// Whether a forward of few rows runs on the fused kernel, which takes its operands as they are, instead of pf_small.cu.  Those kernels
// take as long for 1 row as for 8 and more from there on, the fused one the same for all 32: 570 shapes, fused against pf_small.cu
// in the mean 1.04 times up to 8 rows, 0.94 for 12 and 16, 0.92 for 20 and 24, 0.77 beyond.  Up to 8 rows the fused kernel is
// faster where its first product is one k-block or pf_small.cu's would be cut finely, at small ranks (8 x 384 -> 32 -> 1536: 0.91; 8 x
// 256 -> 192 -> 256: 1.21); a wide output of a small rank is many rows of V in few lines (20 x 512 -> 8 -> 6000: 1.18).
bool few_rows_fused(const LinearArgs& a) {
    const bool faster = a.m <= 8 ? a.r <= 64 && a.n <= 2048 && (a.k <= 64 || a.k > 256) : !(a.n > 4096 && a.m <= 24 && a.r < 64);
    return faster && encode_fn() != nullptr && a.k <= 512 && a.n <= (1 << 22) && use_chain_fwd(a) && tma_ok(a.x, a.ldx) && tma_ok(a.U, a.ldu) && tma_ok(a.V, a.ldv);
}

int linear_fwd(const LinearArgs& a, int* handled) {
    *handled = 0;
    if (encode_fn() == nullptr) return PF_OK;
    // the grids below index column tiles with 16 bits: absurdly wide layers take the FMA kernels
    if (a.k > (1 << 22) || a.n > (1 << 22) || a.r > (1 << 22)) return PF_OK;
    int st = PF_OK;
    char* scratch = a.ws;
    Staged x, U, V;
    RepackList repacks;
    if (stage_operand(a.x, a.ldx, a.m, a.k, scratch, &x, &repacks, a.tight)) return PF_OK;
    if (stage_operand(a.U, a.ldu, a.k, a.r, scratch, &U, &repacks, a.tight)) return PF_OK;
    if (stage_operand(a.V, a.ldv, a.n, a.r, scratch, &V, &repacks, a.tight)) return PF_OK;
    const bool copies = repacks.count > 0;
    st = repacks.flush(a.stream);
    if (st != PF_OK) return st;
    *handled = 1;
    // T: written straight into the stash when TMA can store it (fused) or read it back, else into padded scratch
    void* T = scratch;
    int64_t ldT = row_pitch(a.r, a.tight);
    ChainPlan plan;
    const bool fused = use_chain_fwd(a) && chain_plan(a.m, a.k, a.n, a.r, true, &plan);
    const bool stash_direct = a.T && (fused ? tma_out(a.T, a.ldt, a.r) : tma_ok(a.T, a.ldt));
    if (stash_direct) { T = a.T; ldT = a.ldt; }
    bool stash_written = false;   // the stash at its own (TMA-unreadable) pitch came out of the first product
    if (fused) {
        // one fused kernel; the intermediate leaves the chip only if a stash was asked for
        st = chain(x.p, x.ld, a.m, a.k, U.p, U.ld, a.r, V.p, V.ld, a.n, a.y, a.ldy, a.T ? T : nullptr, ldT,
                   a.stream, nullptr, 0, a.bias, a.act, beyond_l2(a.m, a.k, a.n) ? kL2Stream : 0.f, beyond_l2(a.m, a.k, a.n) ? kL2Stream : 0.f);
    } else {
        const SliceRoom p1{reinterpret_cast<float*>(scratch + align_up(static_cast<size_t>(a.m) * row_pitch(a.r, a.tight) * 2, 256)),
                           first_partial_bytes(a.m, a.k, a.n, a.r, false)};
        // (V, and beside copies what was not copied, need not wait for the launch before)
        st = gemm({x.p, x.ld, false, 0, false, copies && !x.copied}, {U.p, U.ld, true, 0, false, copies && !U.copied}, a.m, a.r, a.k, T, ldT,
                  a.whole ? 1 : pick_splits(a.m, a.r, pick_bn(a.r), a.k), a.whole ? SliceRoom() : p1, a.stream,
                  (a.T && !stash_direct) ? a.T : nullptr, a.ldt, &stash_written);
        if (st != PF_OK) return st;
        st = gemm({T, ldT, false, 0, true}, {V.p, V.ld, false, 0, false, true}, a.m, a.n, a.r, a.y, a.ldy, 1, {}, a.stream, nullptr, 0, nullptr,
                  a.bias, a.act);
    }
    if (st != PF_OK) return st;
    if (a.T && !stash_direct && !stash_written &&
        repack_rows_bf16(T, ldT, a.T, a.ldt, a.m, a.r, a.r, a.stream) != cudaSuccess)
        return PF_ERR_CUDA;
    return PF_OK;
}

int linear_bwd(const LinearArgs& a, int* handled) {
    *handled = 0;
    if (encode_fn() == nullptr) return PF_OK;
    // the grids below index column tiles with 16 bits: absurdly wide layers take the FMA kernels
    if (a.k > (1 << 22) || a.n > (1 << 22) || a.r > (1 << 22)) return PF_OK;
    int st = PF_OK;
    char* scratch = a.ws;
    Staged x, U, V, dY, T;
    RepackList repacks;
    if (stage_operand(a.x, a.ldx, a.m, a.k, scratch, &x, &repacks)) return PF_OK;
    if (stage_operand(a.U, a.ldu, a.k, a.r, scratch, &U, &repacks)) return PF_OK;
    if (stage_operand(a.V, a.ldv, a.n, a.r, scratch, &V, &repacks)) return PF_OK;
    if (stage_operand(a.dY, a.lddy, a.m, a.n, scratch, &dY, &repacks)) return PF_OK;
    char* Tbuf = scratch;
    scratch += align_up(static_cast<size_t>(a.m) * row_pitch(a.r) * 2, 256);
    if (a.T) {
        if (tma_ok(a.T, a.ldt)) { T.p = a.T; T.ld = a.ldt; }
        else if (a.r % 8 == 0) return PF_OK;   // odd pitch on an even width: FMA path
        else {
            repacks.jobs[repacks.count++] = RepackJob{a.T, a.ldt, Tbuf, row_pitch(a.r), a.m, a.r};
            T.p = Tbuf; T.ld = row_pitch(a.r); T.copied = true;
        }
    }
    const bool copies = repacks.count > 0;
    st = repacks.flush(a.stream);
    if (st != PF_OK) return st;
    *handled = 1;
    bool need_T = false;
    if (!a.T) {
        need_T = true;
        T.p = Tbuf; T.ld = row_pitch(a.r);
    }
    char* G = scratch;
    const int64_t ldG = row_pitch(a.r);
    scratch += align_up(static_cast<size_t>(a.m) * ldG * 2, 256);
    size_t pu_bytes = 0, pv_bytes = 0;
    ChainPlan plan;
    const bool fused_dx = use_chain(a.m, a.r) && !unfused_backward(a.m, a.k, a.n, a.r) && (!a.dX || tma_out(a.dX, a.lddx, a.k)) &&
                          chain_plan(a.m, a.n, a.k, a.r, a.dX != nullptr, &plan);
    int su, sv;
    bool dv_beside;
    bwd_split_plan(a.m, a.k, a.n, a.r, fused_dx, &su, &sv, &dv_beside);
    bwd_partial_bytes(a.m, a.k, a.n, a.r, &pu_bytes, &pv_bytes);
    const SliceRoom pu{reinterpret_cast<float*>(scratch), pu_bytes};
    scratch += pu_bytes;
    const SliceRoom pv{reinterpret_cast<float*>(scratch), pv_bytes};
    scratch += pv_bytes;
    const SliceRoom p1{reinterpret_cast<float*>(scratch), first_partial_bytes(a.m, a.k, a.n, a.r, true)};
    const bool narrow = narrow_reductions(a.k, a.n, a.r);
    // G = dY V ; dX = G U^T ; dU = x^T G ; dV = dY^T T
    if (need_T) {   // no stash: recompute T = x U
        st = gemm({x.p, x.ld, false, 0, false, copies && !x.copied}, {U.p, U.ld, true, 0, false, copies && !U.copied}, a.m, a.r, a.k, Tbuf, row_pitch(a.r),
                  pick_splits(a.m, a.r, pick_bn(a.r), a.k), p1, a.stream);
        if (st != PF_OK) return st;
    }
    if (fused_dx) {
        const bool big = beyond_l2(a.m, a.k, a.n);
        st = chain(dY.p, dY.ld, a.m, a.n, V.p, V.ld, a.r, U.p, U.ld, a.k, a.dX, a.lddx, G, ldG, a.stream, nullptr,
                   dv_beside ? 1 : 0, nullptr, 0, big ? 0.2f : 0.f, big ? kL2Stream : 0.f);
        if (st != PF_OK) return st;
    } else {
        // G = dY V, then dU = x^T G and dX = G U^T, which need it; dV = dY^T T needs nothing.  Where the tiles of dU and dV fit the machine
        // they run on single CTAs, split or whole, and the launches are ordered as is expected to be fastest:
        //   two      {G, dV}, {dU, dX}: each reduction fills the machine, two sums of slices; few rows, or many columns of y
        //   three    {G}, {dU, dV, dX}: one sum, and the long contraction behind one start only; 512 -> 128 -> 512: 1000 rows 10.8 us
        //            against 12.3, 4096 x 1500 -> 256 -> 1500: 40.1 against 47.3; 8192 x 1024 -> 256 -> 4096: 78 against 61
        //   pairs    G and dX on CTA pairs by themselves, {dU, dV}: 16384 x 768 -> 512 -> 3072: 123 us, two 144, three 150
        // (G and dX run on pairs by themselves in the first two where that is faster.)  Larger reductions run on whichever form is faster.
        GemmLaunch gg, gv, gu, gx;
        const int bn = pick_bn(a.r);
        const int64_t tr = ceil_div(a.r, bn), tg = ceil_div(a.m, kBM) * tr, tv = ceil_div(a.n, kBM) * tr, kb_n = ceil_div(a.n, kBK), kb_m = ceil_div(a.m, kBK);
        const int sg_alone = pick_splits(a.m, a.r, bn, a.n);
        int sg = sg_alone;
        if (sg > 1 && sv > 1 && tg * sg + tv * sv > num_sms()) {        // both sums in one launch: their blocks must fit together
            int sg2 = 1, sv2 = 1;
            pick_pair_splits(a.m, a.n, a.r, kb_n, kb_m, &sg2, &sv2);
            sg = std::min(sg, sg2);                                      // (no more slices than the workspace holds)
            sv = std::min(sv, sv2);
        }
        enum { kTwo, kThree, kPairs } order = kTwo;
        if (narrow) {
            int su3, sv3;
            pick_pair_splits(a.k, a.n, a.r, kb_m, kb_m, &su3, &sv3);
            const bool sx = x.ld % 64 != 0, sy = dY.ld % 64 != 0, vu = vector_rows(a.dU, a.lddu, 0), vv = vector_rows(a.dV, a.lddv, 0);
            const Work x_work = work_of(a.m, a.k, ceil_div(a.r, kBK), 1, 1, false, false, true, vector_rows(a.dX, a.lddx, 0));
            const Work g_work = work_of(a.m, a.r, kb_n, sg_alone, 1, false, sy, false, true), g_whole = work_of(a.m, a.r, kb_n, 1, 1, false, sy, false, true);
            const Work two1[2] = {work_of(a.m, a.r, kb_n, sg, 1, false, sy, false, true), work_of(a.n, a.r, kb_m, sv, 1, true, sy, false, vv)};
            const Work two2[2] = {x_work, work_of(a.k, a.r, kb_m, su, 1, true, sx, false, vu)};
            const Work all[3] = {work_of(a.k, a.r, kb_m, su3, 1, true, sx, false, vu), work_of(a.n, a.r, kb_m, sv3, 1, true, sy, false, vv), x_work};
            const double pair_g = pairs_us(&g_whole, 1), pair_x = pairs_us(&x_work, 1);
            const double two = std::min(singles_us(two1, 2), (pair_g + singles_us(two1 + 1, 1)) / kPairMargin) +
                               (a.dX ? std::min(singles_us(two2, 2), (pair_x + singles_us(two2 + 1, 1)) / kPairMargin) : singles_us(two2 + 1, 1));
            const double three = std::min(singles_us(&g_work, 1), pair_g / kPairMargin) + singles_us(all, a.dX ? 3 : 2);
            const double pairs = a.dX ? pair_g + pair_x + singles_us(all, 2) : 1e30;
            // (The expectation is too good for long reductions beside many tiles of dX.  Of 774 shapes 6 take more than 3 % longer than
            // in two launches, 1 more than 8 %; all of them together 5.6 % less, 0.9 % more than the best order of each.)
            const bool short_ones = std::max(all[0].kb, all[1].kb) <= 64 && (a.n < 2 * a.k || a.m < 2048);
            if (short_ones && 1.08 * three < std::min(two, 1.1 * pairs)) order = kThree;
            else if (1.1 * pairs < two) order = kPairs;
            if (order != kTwo) { sg = sg_alone; su = su3; sv = sv3; }
        }
        // What need not wait for the launch before: behind copies what was not copied, behind the recomputed T all but T, and behind
        // G all but G.
        const bool e_dy = need_T || (copies && !dY.copied), e_v = need_T || (copies && !V.copied);
        const bool e_t = order == kThree || order == kPairs || (!need_T && copies && !T.copied);
        const Operand op_dy{dY.p, dY.ld, false, 0, false, e_dy}, op_v{V.p, V.ld, true, 0, false, e_v};
        const Operand op_dyt{dY.p, dY.ld, true, 0, false, order == kTwo ? e_dy : true}, op_t{T.p, T.ld, true, 0, false, e_t};
        st = gemm_prepare_any(op_dy, op_v, a.m, a.r, a.n, G, ldG, sg, p1, nullptr, &gg);
        if (st == PF_OK) st = gemm_prepare_any(op_dyt, op_t, a.n, a.r, a.m, a.dV, a.lddv, sv, pv, nullptr, &gv);
        if (st == PF_OK) st = gemm_prepare_any({x.p, x.ld, true, 0, false, true}, {G, ldG, true}, a.k, a.r, a.m, a.dU, a.lddu, su, pu, nullptr, &gu);
        if (st == PF_OK && a.dX) st = gemm_prepare({G, ldG, false, 0, true}, {U.p, U.ld, false, 0, false, true}, a.m, a.k, a.r, a.dX, a.lddx, 1, {}, nullptr, &gx);
        if (st != PF_OK) return st;
        PairJob j1[2] = {{dY.p, dY.ld, false, 0, V.p, V.ld, true, 0, a.m, a.r, a.n, G, ldG},
                         {dY.p, dY.ld, true, 0, T.p, T.ld, true, 0, a.n, a.r, a.m, a.dV, a.lddv}};
        PairJob j2[2] = {{G, ldG, false, 0, U.p, U.ld, false, 0, a.m, a.k, a.r, a.dX, a.lddx},
                         {x.p, x.ld, true, 0, G, ldG, true, 0, a.k, a.r, a.m, a.dU, a.lddu}};
        j1[0].a_early = j1[1].a_early = e_dy; j1[0].b_early = e_v; j1[1].b_early = op_t.early;
        j2[0].b_early = j2[1].a_early = true;
        const GemmLaunch* const l1[2] = {&gg, &gv};
        const GemmLaunch* const l2[2] = {&gx, &gu};
        if (!narrow) {
            bool pairs_v = false, pairs_u = false;
            st = launch_faster(l1, j1, 2, a.stream, 0.0, &pairs_v);
            if (st == PF_OK) st = a.dX ? launch_faster(l2, j2, 2, a.stream, 0.0, &pairs_u) : launch_faster(l2 + 1, j2 + 1, 1, a.stream, 0.0, &pairs_u);
            keep_slices(a.du_slices, &gu, gu.p.splits > 1 && !pairs_u ? pu : SliceRoom());      // (split ones leave them anyway)
            keep_slices(a.dv_slices, &gv, gv.p.splits > 1 && !pairs_v ? pv : SliceRoom());
            return st;
        }
        keep_slices(a.du_slices, &gu, pu);
        keep_slices(a.dv_slices, &gv, pv);
        if (order == kTwo) {
            st = launch_with(l1, j1, 2, a.stream);
            if (st != PF_OK) return st;
            return a.dX ? launch_with(l2, j2, 2, a.stream) : launch_singles(l2 + 1, 1, a.stream);
        }
        const GemmLaunch* const l3[3] = {&gu, &gv, &gx};
        if (order == kPairs) {
            st = gemm_pairs(j1, 1, 1, a.stream);
            if (st == PF_ERR_UNSUPPORTED) st = launch_prepared(gg, a.stream);
            if (st == PF_OK) st = gemm_pairs(j2, 1, 1, a.stream);
            if (st == PF_ERR_UNSUPPORTED) st = launch_prepared(gx, a.stream);
            return st == PF_OK ? launch_singles(l3, 2, a.stream) : st;
        }
        st = launch_faster(l1, j1, 1, a.stream);
        return st == PF_OK ? launch_singles(l3, a.dX ? 3 : 2, a.stream) : st;
    }
    // dU = x^T G, dV = dY^T T: one launch when their tiles allow
    GemmLaunch gu, gv;
    st = gemm_prepare_any({x.p, x.ld, true, 0, false, true}, {G, ldG, true}, a.k, a.r, a.m, a.dU, a.lddu, su, pu, nullptr, &gu);
    if (st == PF_OK) st = gemm_prepare_any({dY.p, dY.ld, true, 0, false, true}, {T.p, T.ld, true, 0, false, true}, a.n, a.r, a.m, a.dV, a.lddv, sv, pv, nullptr, &gv);
    if (st != PF_OK) return st;
    keep_slices(a.du_slices, &gu, narrow ? pu : SliceRoom());
    keep_slices(a.dv_slices, &gv, narrow ? pv : SliceRoom());
    // dY is read for the last time and makes room.  So does x, but it is the output of the layer below, whose activation's backward
    // reads it next: in a step that streams less than a quarter of L2 it stays.  Blocks of two layers with their activations, six in
    // a row, x first to go / as ever: 4096 x 512 -> 128 -> 2048 and back (21 MB a layer): 89.7 / 87.2 us a block, 6000: 98.9 / 97.1, 8192:
    // 108.8 / 108.3, 12000: 141.4 / 143.9, 16384: 176.0 / 179.7; backward of one layer of 8192 x 2048 -> 128 -> 512: 27.0 / 28.3, of 12000 x
    // 2048 -> 96 -> 2048: 51.8 / 56.0.  In a step that streams more than L2 holds a fifth of dY is kept for this launch, and
    // everything else passes through: 16384 x 4096 -> 64 -> 4096: 161 -> 149 us, 8192 x 4096 -> 64 -> 4096: 101 -> 88, 16384 x 2048 -> 64 ->
    // 2048: 91 -> 81.
    gu.p.keep_a = streamed_bytes(a.m, a.k, a.n) > kL2Bytes / 4 ? kL2Stream : 0.f;
    gv.p.keep_a = kL2Stream;
    const GemmLaunch* list[2] = {&gu, &gv};
    if (gu.p.splits <= 1 && gv.p.splits > 1) std::swap(list[0], list[1]);       // a split product has to come before the plain ones
    if (dv_beside) {
        // dV first (its blocks are dispatched first, onto the SMs the fused kernel left free) and
        // without waiting for the fused kernel; dU follows as that kernel's blocks retire
        gv.p.independent = 1;
        list[0] = &gv; list[1] = &gu;
    }
    st = gemm_multi(list, 2, a.stream);
    if (st != PF_ERR_UNSUPPORTED) return st;
    gv.p.independent = 0;
    st = launch_prepared(gu, a.stream);      // tile widths that cannot share a launch: one launch each
    return st == PF_OK ? launch_prepared(gv, a.stream) : st;
}

// ------------------------------------------------------------------------------ grouped linear layer
namespace {
struct GroupedPlan {
    int bn;                       // tile width of the m x r and (k|n) x r products
    int s1, sg, su, sv;           // slices of x U, dY V, dU, dV
    size_t t_bytes, p1_bytes, pu_bytes, pv_bytes;
};
GroupedPlan grouped_plan(int groups, int64_t m, int64_t k, int64_t n, int64_t r) {
    GroupedPlan g;
    g.bn = pick_bn(r);
    const int64_t tr = ceil_div(r, g.bn);
    const int64_t tm = ceil_div(m, kBM) * tr * groups, tk = ceil_div(k, kBM) * tr * groups, tn = ceil_div(n, kBM) * tr * groups;
    g.s1 = slices_of(tm, ceil_div(k, kBK));
    g.sg = slices_of(tm, ceil_div(n, kBK));
    g.su = slices_of(tk, ceil_div(m, kBK));
    g.sv = slices_of(tn, ceil_div(m, kBK));
    if (tm > kFixTiles) g.s1 = g.sg = 1;
    if (tk > kFixTiles) g.su = 1;
    if (tn > kFixTiles) g.sv = 1;
    g.t_bytes = align_up(static_cast<size_t>(groups) * m * row_pitch(r) * 2, 256);
    g.p1_bytes = align_up(static_cast<size_t>(groups) * std::max(partial_bytes(m, r, g.s1), partial_bytes(m, r, g.sg)), 256);
    g.pu_bytes = align_up(static_cast<size_t>(groups) * partial_bytes(k, r, g.su), 256);
    g.pv_bytes = align_up(static_cast<size_t>(groups) * partial_bytes(n, r, g.sv), 256);
    return g;
}
bool grouped_ok(const void* p, int64_t ld, int64_t gs) { return tma_ok(p, ld) && gs % 8 == 0; }

// A grouped operand that TMA must read: as it is, or (ragged widths) all its groups copied to `scratch` at a
// padded pitch.  A shared operand is one matrix.
struct StagedGroups {
    const void* p;
    int64_t ld, gs;
    bool copied = false;
};
int stage_groups(const void* p, int64_t ld, int64_t gs, int groups, bool shared, int64_t rows, int64_t cols, char*& scratch,
                 StagedGroups* out, RepackList* list) {
    *out = StagedGroups{p, ld, gs};
    if (grouped_ok(p, ld, gs)) return 0;
    if (cols % 8 == 0) return 1;          // the workspace query reserves repack room only for ragged widths
    const int64_t ldp = row_pitch(cols), n = shared ? 1 : groups;
    list->jobs[list->count++] = RepackJob{p, ld, scratch, ldp, rows, cols, n, gs};
    *out = StagedGroups{scratch, ldp, shared ? 0 : rows * ldp, true};
    scratch += align_up(static_cast<size_t>(n) * rows * ldp * 2, 256);
    return 0;
}
size_t groups_room(int groups, int64_t rows, int64_t cols) {
    return cols % 8 == 0 ? 0 : align_up(static_cast<size_t>(groups) * rows * row_pitch(cols) * 2, 256);
}
}  // namespace

size_t grouped_workspace(int groups, int64_t m, int64_t k, int64_t n, int64_t r, bool bwd) {
    const GroupedPlan g = grouped_plan(groups, m, k, n, r);
    size_t b = g.t_bytes + g.p1_bytes + (bwd ? g.t_bytes + g.pu_bytes + g.pv_bytes : 0);
    b += groups_room(groups, m, k) + groups_room(groups, k, r) + groups_room(groups, n, r);      // x, U, V
    if (bwd) b += groups_room(groups, m, n) + groups_room(groups, m, r);                          // dY, T
    return b;
}

int linear_grouped_fwd(const GroupedArgs& a, int* handled) {
    *handled = 0;
    if (a.groups == 1) return PF_OK;      // one group is the ungrouped layer, whose kernels take 2-D maps
    if (encode_fn() == nullptr || a.groups > 1024 || a.k > (1 << 22) || a.n > (1 << 22) || a.r > (1 << 22)) return PF_OK;
    const GroupedPlan gp = grouped_plan(a.groups, a.m, a.k, a.n, a.r);
    const bool shared_x = a.sx == 0 && a.groups > 1;
    char* ws = a.ws;
    char* Tbuf = ws; ws += gp.t_bytes;
    const SliceRoom p1{reinterpret_cast<float*>(ws), gp.p1_bytes}; ws += gp.p1_bytes;
    StagedGroups x, U, V;
    RepackList repacks;
    if (stage_groups(a.x, a.ldx, a.sx, a.groups, shared_x, a.m, a.k, ws, &x, &repacks) ||
        stage_groups(a.U, a.ldu, a.su, a.groups, false, a.k, a.r, ws, &U, &repacks) ||
        stage_groups(a.V, a.ldv, a.sv, a.groups, false, a.n, a.r, ws, &V, &repacks))
        return PF_OK;
    // T: the stash itself when TMA can read it back, else scratch at a padded pitch; the first product then
    // writes the stash beside it
    const bool stash_direct = a.T && grouped_ok(a.T, a.ldt, a.st);
    void* T = stash_direct ? a.T : static_cast<void*>(Tbuf);
    const int64_t ldT = stash_direct ? a.ldt : row_pitch(a.r), sT = stash_direct ? a.st : a.m * row_pitch(a.r);
    // The fused kernel where it pays for one group (see use_chain_fwd; k up to 1024, as the groups share the SMs), in two
    // launches of half of the groups each (the call's launches are documented as two) that run side by side.  Not where the
    // tiles are small and more than a wave or two, whose starts the two products hide better: 4 x (8000 x 256 -> 32 -> 64): 10.7 us
    // unfused, 13.8 fused; 4 x (8000 x 64 -> 32 -> 256): 12.5 and 11.3.  Against two products one after the
    // other: 4 x (1024 x 512 -> 128 -> 512): 13.0 -> 8.3 us, 4 x (8192 x 512 -> 128 -> 512): 26.7 -> 19.3, 2 x (7666 x 1976 ->
    // 120 -> 1976): 51 -> 42; 4 x (185 x 1536 -> 192 -> 1536): 12.1 -> 12.8; 8 x (4789 x 72 -> 8 -> 72): 18.3 -> 18.8.
    ChainPlan plan;
    if (a.r <= 192 && (a.m >= 2048 || short_first_product(a.k, a.r, x.ld, U.ld, 1024)) && (a.k + a.n >= 512 || ceil_div(a.m, kBM) * a.groups <= (a.n >= 256 ? 2 : 1) * num_sms()) && grouped_ok(a.y, a.ldy, a.sy) && a.n % 8 == 0 && (!a.T || (stash_direct && a.r % 8 == 0)) &&
        chain_plan(a.m, a.k, a.n, a.r, true, &plan, 128, 0, a.groups)) {
        *handled = 1;
        int st = repacks.flush(a.stream);
        const int half[3] = {0, a.groups / 2, a.groups};
        auto at = [](const void* p, int64_t gs, int g) { return const_cast<char*>(static_cast<const char*>(p)) + static_cast<size_t>(g) * gs * 2; };
        for (int h = 0; h < 2 && st == PF_OK; ++h) {
            const int g = half[h];
            st = chain_groups(half[h + 1] - g, a.groups, at(x.p, x.gs, g), x.ld, x.gs, a.m, a.k, at(U.p, U.gs, g), U.ld, U.gs, a.r, at(V.p, V.gs, g), V.ld, V.gs, a.n,
                              at(a.y, a.sy, g), a.ldy, a.sy, a.T ? at(a.T, a.st, g) : nullptr, a.ldt, a.st, h == 1, a.stream);
        }
        return st;
    }
    GemmLaunch g1, g2;
    const Grouping gt{a.groups, sT, false}, gy{a.groups, a.sy, false};
    const bool copies = repacks.count > 0;      // (what need not wait for the launch before: as in linear_fwd)
    int st = gemm_prepare({x.p, x.ld, false, x.gs, false, copies && !x.copied}, {U.p, U.ld, true, U.gs, false, copies && !U.copied}, a.m, a.r, a.k, T, ldT, gp.s1,
                          p1, nullptr, &g1, &gt);
    if (st == PF_OK)
        st = gemm_prepare({T, ldT, false, sT, true}, {V.p, V.ld, false, V.gs, false, true}, a.m, a.n, a.r, a.y, a.ldy, 1, {}, nullptr, &g2, &gy);
    if (st == PF_ERR_UNSUPPORTED) return PF_OK;
    if (st != PF_OK) return st;
    if (a.T && !stash_direct) {
        g1.p.C2 = a.T; g1.p.ldc2 = a.ldt; g1.p.c2_gstride = a.st;
    }
    *handled = 1;
    st = repacks.flush(a.stream);
    if (st == PF_OK) st = launch_prepared(g1, a.stream);
    if (st != PF_OK) return st;
    PairJob jy{T, ldT, false, sT, V.p, V.ld, false, V.gs, a.m, a.n, a.r, a.y, a.ldy, a.sy, a.groups};
    jy.b_early = true;
    const GemmLaunch* const ly[1] = {&g2};
    return launch_faster(ly, &jy, 1, a.stream);
}

int linear_grouped_bwd(const GroupedArgs& a, int* handled) {
    *handled = 0;
    if (a.groups == 1) return PF_OK;      // one group is the ungrouped layer, whose kernels take 2-D maps
    if (encode_fn() == nullptr || a.groups > 1024 || a.k > (1 << 22) || a.n > (1 << 22) || a.r > (1 << 22)) return PF_OK;
    const GroupedPlan gp = grouped_plan(a.groups, a.m, a.k, a.n, a.r);
    const bool shared_x = a.sx == 0 && a.groups > 1;
    char* ws = a.ws;
    void* Tbuf = ws; ws += gp.t_bytes;
    const SliceRoom p1{reinterpret_cast<float*>(ws), gp.p1_bytes}; ws += gp.p1_bytes;
    void* Gbuf = ws; ws += gp.t_bytes;
    const SliceRoom pu{reinterpret_cast<float*>(ws), gp.pu_bytes}; ws += gp.pu_bytes;
    const SliceRoom pv{reinterpret_cast<float*>(ws), gp.pv_bytes}; ws += gp.pv_bytes;
    const int64_t ldW = row_pitch(a.r), sW = a.m * row_pitch(a.r);
    StagedGroups x, U, V, dY, T{Tbuf, ldW, sW};
    RepackList repacks;
    if (stage_groups(a.x, a.ldx, a.sx, a.groups, shared_x, a.m, a.k, ws, &x, &repacks) ||
        stage_groups(a.U, a.ldu, a.su, a.groups, false, a.k, a.r, ws, &U, &repacks) ||
        stage_groups(a.V, a.ldv, a.sv, a.groups, false, a.n, a.r, ws, &V, &repacks) ||
        stage_groups(a.dY, a.lddy, a.sdy, a.groups, false, a.m, a.n, ws, &dY, &repacks) ||
        (a.T && stage_groups(a.T, a.ldt, a.st, a.groups, false, a.m, a.r, ws, &T, &repacks)))
        return PF_OK;
    // The fused kernel for G and dX as in linear_bwd, then dU and dV, whose slices have to fit the machine together:
    // 2 x (8000 x 1024 -> 64 -> 256): 44.6 -> 23.4 us, 4 x (8192 x 512 -> 128 -> 512): 48.8 -> 42.1, 2 x (7666 x 1976 -> 120 -> 1976):
    // 104 -> 78.  Narrow dX only while its tiles are one wave: 8 x (8000 x 64 -> 32 -> 256): 30.5 us unfused, 35.3 fused; 8 x (4000 x 256 ->
    // 64 -> 64): 0.84 times.
    ChainPlan plan;
    const bool fused = !shared_x && a.dX && use_chain(a.m, a.r) && grouped_ok(a.dX, a.lddx, a.sdx) && a.k % 8 == 0 && (a.k >= 256 || ceil_div(a.m, kBM) * a.groups <= num_sms()) && chain_plan(a.m, a.n, a.k, a.r, true, &plan, 128, 0, a.groups);
    int su = gp.su, sv = gp.sv;
    if (fused) {
        const int64_t nkb = ceil_div(a.m, kBK);
        int su2, sv2;
        pick_pair_splits(a.k, a.n, a.r, nkb, nkb, &su2, &sv2, a.groups);
        su = std::min(su, su2);
        sv = std::min(sv, sv2);
    }
    GemmLaunch gT, gG, gV, gU, gX;
    const Grouping gw{a.groups, sW, false}, gdv{a.groups, a.sdv, false}, gdu{a.groups, a.sdu, false};
    const Grouping gdx{a.groups, shared_x ? 0 : a.sdx, shared_x};
    int st = PF_OK;
    // What need not wait for the launch before: as in linear_bwd (behind the fused kernel everything but G).
    const bool copies = repacks.count > 0, e_dy = !a.T || (copies && !dY.copied), e_v = !a.T || (copies && !V.copied), e_t = a.T && copies && !T.copied;
    if (!a.T) st = gemm_prepare({x.p, x.ld, false, x.gs, false, copies && !x.copied}, {U.p, U.ld, true, U.gs, false, copies && !U.copied}, a.m, a.r, a.k, Tbuf, ldW,
                                gp.s1, p1, nullptr, &gT, &gw);
    // the recomputed T and G share the slice buffer p1: they are separate launches, one after the other
    if (st == PF_OK) st = gemm_prepare({dY.p, dY.ld, false, dY.gs, false, e_dy}, {V.p, V.ld, true, V.gs, false, e_v}, a.m, a.r, a.n, Gbuf, ldW, gp.sg, p1, nullptr, &gG, &gw);
    if (st == PF_OK) st = gemm_prepare({dY.p, dY.ld, true, dY.gs, false, fused || e_dy}, {T.p, T.ld, true, T.gs, false, fused || e_t}, a.n, a.r, a.m, a.dV, a.lddv, sv, pv, nullptr, &gV, &gdv);
    if (st == PF_OK) st = gemm_prepare({x.p, x.ld, true, x.gs, false, true}, {Gbuf, ldW, true, sW}, a.k, a.r, a.m, a.dU, a.lddu, su, pu, nullptr, &gU, &gdu);
    if (st == PF_OK && a.dX)
        st = gemm_prepare({Gbuf, ldW, false, sW, true}, {U.p, U.ld, false, U.gs, false, true}, a.m, a.k, a.r, a.dX, a.lddx, 1, {}, nullptr, &gX, &gdx);
    if (st == PF_ERR_UNSUPPORTED) return PF_OK;
    if (st != PF_OK) return st;
    *handled = 1;
    st = repacks.flush(a.stream);
    if (st != PF_OK) return st;
    if (!a.T) {
        st = launch_prepared(gT, a.stream);
        if (st != PF_OK) return st;
    }
    if (fused) {
        st = chain_groups(a.groups, a.groups, dY.p, dY.ld, dY.gs, a.m, a.n, V.p, V.ld, V.gs, a.r, U.p, U.ld, U.gs, a.k, a.dX, a.lddx, a.sdx, Gbuf, ldW, sW,
                          false, a.stream);
        if (st != PF_OK) return st;
        PairJob jf[2] = {{x.p, x.ld, true, x.gs, Gbuf, ldW, true, sW, a.k, a.r, a.m, a.dU, a.lddu, a.sdu, a.groups},
                               {dY.p, dY.ld, true, dY.gs, T.p, T.ld, true, T.gs, a.n, a.r, a.m, a.dV, a.lddv, a.sdv, a.groups}};
        jf[0].a_early = jf[1].a_early = jf[1].b_early = true;
        const GemmLaunch* const lf[2] = {&gU, &gV};
        return launch_faster(lf, jf, 2, a.stream);
    }
    // launch A: G = dY V and dV = dY^T T (independent of each other); launch B: dU = x^T G and dX = G U^T
    PairJob ja[2] = {{dY.p, dY.ld, false, dY.gs, V.p, V.ld, true, V.gs, a.m, a.r, a.n, Gbuf, ldW, sW, a.groups},
                           {dY.p, dY.ld, true, dY.gs, T.p, T.ld, true, T.gs, a.n, a.r, a.m, a.dV, a.lddv, a.sdv, a.groups}};
    PairJob jb[2] = {{x.p, x.ld, true, x.gs, Gbuf, ldW, true, sW, a.k, a.r, a.m, a.dU, a.lddu, a.sdu, a.groups},
                           {Gbuf, ldW, false, sW, U.p, U.ld, false, U.gs, a.m, a.k, a.r, a.dX, a.lddx, shared_x ? 0 : a.sdx, a.groups, shared_x}};
    ja[0].a_early = ja[1].a_early = e_dy; ja[0].b_early = e_v; ja[1].b_early = e_t;
    jb[0].a_early = jb[1].b_early = true;
    const GemmLaunch* const la[2] = {&gG, &gV};
    const GemmLaunch* const lb[2] = {&gU, &gX};
    st = launch_faster(la, ja, 2, a.stream);
    if (st != PF_OK) return st;
    return launch_faster(lb, jb, a.dX ? 2 : 1, a.stream);
}

// After a bounded wait has expired some CTAs may have left their tile counters non-zero.
void reset_fix_counters() {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_fix_counters) == cudaSuccess) cudaMemset(ptr, 0, sizeof(unsigned int) * kFixSlots * kFixTiles * 2);
}

// Tensor-core envelope of the factorized convolution: channel counts that are multiples of 8 (TMA pitches; a
// ragged 64-channel block is zero-filled), output rows that fit the tiles (128 pixels forward and dX, 64 for
// the contraction of dU), and for a strided backward at least one tap per pixel class (kernel >= stride).
constexpr int kConvMaxRank = 384;
static bool conv_tc_ok(const ConvArgs& a, bool fwd) {
    if (a.kh != a.kw || a.C % 8 != 0 || a.R % 8 != 0 || a.O % 8 != 0 || a.R > kConvMaxRank) return false;
    if (a.stride > 4 || a.Wo > (fwd ? 128 : 64) || a.stride * a.Wo > 256) return false;
    if (!fwd && (a.kh < a.stride || ceil_div(a.W, a.stride) > 128)) return false;
    if (static_cast<int64_t>(a.N) * a.H * a.W > 0x7fffffff || static_cast<int64_t>(a.kh) * a.kw * a.C > 0x7fffffff) return false;
    return encode_fn() != nullptr;
}
static bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

namespace {
// Slices of dU and dV of a convolution: both reductions share one launch.
void conv_splits(const ConvA& c, int O, int* su, int* sv) {
    pick_pair_splits(conv_du_tiles(c.kh, c.kw, c.C) * kBM, O, c.R, conv_k_tiling(c).blocks,
                     ceil_div(static_cast<int64_t>(c.N) * c.Ho * c.Wo, kBK), su, sv);
}
// Room for the slices of dU and dV ((kh*kw*C) x R and O x R), as bwd_partial_bytes.
void conv_partial_bytes(const ConvA& c, int O, int su, int sv, size_t* bytes_u, size_t* bytes_v) {
    const int64_t rows = conv_du_tiles(c.kh, c.kw, c.C) * kBM;
    const bool narrow = narrow_reductions(rows, O, c.R);
    *bytes_u = narrow ? align_up(slice_bytes(rows, c.R, su), 256) : 0;
    *bytes_v = narrow ? align_up(slice_bytes(O, c.R, sv), 256) : 0;
}
}  // namespace

// Elements from one pixel of dT to the next: rows of 24, 40, 48, 56 or 80 ranks would straddle 128-byte lines, and the products that
// read them once per tap take two requests for most.  (Ranks whose rows divide a line, or are made of lines, lie as they are.)  Backward of
// 16 x 14 x 14, 160 -> 40 -> 160 18.9 -> 16.6 us, of 8 x 28 x 28, 192 -> 48 -> 192 18.9 -> 16.6, stride 2 of 64 x 14 x 14, 256 -> 72 -> 256 22.0 -> 19.9.
// (Ranks that only the FMA kernels take have no such rows.)
int64_t conv_dt_pitch(int64_t R) { return R % 64 == 0 || 64 % R == 0 || R % 8 != 0 || R > kConvMaxRank ? R : (R + 63) / 64 * 64; }
// dX reads U once per tile, so for many pixels it too is copied to that pitch, beside the launch that makes dT; the forward copies both
// factors, and from fewer pixels on: every block reads all of U, a box of 64 ranks' rows in up to twice the requests.  What that
// saves depends on how the rows lie, what it costs is a launch, so the lines are measured (passes over buffers that do not fit L2, without
// and with copies; C is 2 or 4 ranks wide, square y):
//   rows at an odd multiple of 16 bytes.  Above 64 ranks they gain most: forward 3 x 3, 12544 pixels: 72 26 -> 22 us, 120 35 -> 28, 136 45 -> 34, 184
//     56 -> 46; one tap gains later (72: 12544 pixels 9.0 -> 9.4, 25088 13 -> 11; 136: 12544 16.2 -> 15.6).  24 and 40 ranks: 3 x 3 of 12544 15.0 -> 13.7 and 17.5
//     -> 16.9, of 25088 21 -> 18 and 19.2 -> 18.2; one tap of 12544 8.7 -> 8.8 and 8.6 -> 9.5, of 25088 13 -> 11 and 13 -> 12; 5 x 5 of
//     40 12544 31.7 -> 32.4, 25088 60 -> 57, but 96 -> 24 -> 96 of 100352 129 -> 136 (3 x 3: 32.7 -> 29.3).  56 ranks are
//     nearly a line: 5 x 5 of 25088 43 -> 41, else 3 x 3 of 12544 13.8 -> 14.5, of 25088 17.0 -> 17.6, one tap 11.1 -> 11.6.
//   rows at an odd multiple of 32 bytes, above 64 ranks: 3 x 3 of 25088: 80 37 -> 34, 112 47 -> 45, 144 62 -> 61, 176 84 -> 79; of 12544 within 2 %, one tap
//     slower (80: 9.5 -> 10.7).  (48 ranks: 3 x 3 of 100352 34.9 -> 35.9.)
//   rows at a multiple of 64 bytes: 96 13.9 -> 15.5 (12544), 39.0 -> 39.4 (25088); 160 73.0 -> 72.8.
// Backward, stride 1 and more taps than one: 80 of 25088 51 -> 44, 120 70 -> 59, 184 222 -> 207, 24 45 -> 41, 40 43 -> 41, 96 46 -> 44; 56 36 -> 37, of 50176
// 53 -> 52.  Stride 2 gains above 64 ranks with rows at odd multiples of 16 bytes (72 101 -> 94; 24 44 -> 44, 80 57 -> 58, 96 58 -> 60); one tap
// does not (40 26 -> 28, 56 36 -> 39, 120 30 -> 30, 144 46 -> 48), nor 5 x 5 of many pixels (80 -> 40 -> 80 of 100352 262 -> 279).
static size_t conv_factor_copy(int64_t pixels, int kernel, int64_t C, int64_t R, int stride, bool fwd) {
    if (conv_dt_pitch(R) == R || (R < 64 && R % 16 == 0)) return 0;
    const bool odd16 = R % 16 != 0, wide = R > 64;
    int64_t least;
    if (!fwd) {
        if (kernel == 1 || (stride > 1 && !(odd16 && wide)) || (kernel > 3 && !wide && pixels > 80000)) return 0;
        least = R == 56 ? 40000 : 20000;
    } else if (!odd16) {
        if (R % 32 == 0 || kernel == 1) return 0;
        least = 20000;
    } else if (wide) {
        least = kernel == 1 && R < 128 ? 20000 : 12000;
    } else {
        if (R == 56 && kernel < 5) return 0;
        if (kernel > 3 && C < 128 && pixels > 80000) return 0;
        least = R == 24 && kernel > 1 ? 12000 : 20000;
    }
    return pixels < least ? 0 : align_up(static_cast<size_t>(kernel) * kernel * C * conv_dt_pitch(R) * 2, 256);
}

size_t conv_extra_workspace(int N, int H, int W, int C, int R, int O, int kh, int kw, int stride, int pad,
                            bool bwd, bool lean) {
    const int Ho = (H + 2 * pad - kh) / stride + 1, Wo = (W + 2 * pad - kw) / stride + 1;
    if (N < 1 || Ho < 1 || Wo < 1) return 0;
    const size_t copy = lean ? 0 : conv_factor_copy(static_cast<int64_t>(N) * Ho * Wo, kh, C, R, stride, !bwd);
    if (!bwd) return copy > 0 ? copy + align_up(static_cast<size_t>(O) * conv_dt_pitch(R) * 2, 256) : 0;
    const ConvA c{2, N, H, W, C, R, Ho, Wo, kh, kw, pad, stride};
    int su, sv;
    size_t bu, bv;
    conv_splits(c, O, &su, &sv);
    conv_partial_bytes(c, O, su, sv, &bu, &bv);
    ConvArgs a = {};
    a.N = N; a.H = H; a.W = W; a.C = C; a.R = R; a.O = O; a.kh = kh; a.kw = kw; a.stride = stride; a.pad = pad; a.Ho = Ho; a.Wo = Wo;
    return lean ? bu + bv : copy + std::max(bu + bv, conv_flat_bwd_workspace(a));
}

int conv_fwd(const ConvArgs& a, int* handled) {
    *handled = 0;
    if (!conv_tc_ok(a, true) || !aligned16(a.x) || !aligned16(a.U) || !aligned16(a.V) || !aligned16(a.y) ||
        (a.T && !aligned16(a.T)))
        return PF_OK;
    const ChainConv cv{a.N, a.H, a.W, a.C, a.kh, a.kw, a.pad, a.stride};
    // the factors at a pitch of whole lines, where the caller's scratch holds the copies
    const int64_t Keff = static_cast<int64_t>(a.kh) * a.kw * a.C;
    const size_t copy = a.ws ? conv_factor_copy(static_cast<int64_t>(a.N) * a.Ho * a.Wo, a.kh, a.C, a.R, a.stride, true) : 0;
    ConvArgs b = a;
    int64_t ldf = a.R;
    if (copy > 0) {
        ldf = conv_dt_pitch(a.R);
        b.U = a.ws;
        b.V = a.ws + copy;
    }
    const Before copies = [&] {
        const RepackJob jobs[2] = {RepackJob{a.U, a.R, a.ws, ldf, Keff, a.R}, RepackJob{a.V, a.R, a.ws + copy, ldf, a.O, a.R}};
        return copy == 0 || repack_rows_bf16_multi(jobs, 2, a.stream) == cudaSuccess ? PF_OK : PF_ERR_CUDA;
    };
    int st = conv_res_fwd(b, ldf, copies);
    if (st == PF_ERR_UNSUPPORTED) st = chain(b.x, b.C, 0, 0, b.U, ldf, b.R, b.V, ldf, b.O, b.y, b.O, b.T, b.R, b.stream, &cv, 0, nullptr, 0, 0.f, 0.f, copies);
    if (st == PF_ERR_UNSUPPORTED) return PF_OK;      // declined: nothing has been launched
    *handled = 1;
    return st;
}

int conv_bwd(const ConvArgs& a, int* handled) {
    *handled = 0;
    if (!conv_tc_ok(a, false) || !aligned16(a.x) || !aligned16(a.U) || !aligned16(a.V) || !aligned16(a.dY) ||
        (a.T && !aligned16(a.T)) || (a.dX && !aligned16(a.dX)))
        return PF_OK;
    const int64_t P = static_cast<int64_t>(a.N) * a.Ho * a.Wo, Keff = static_cast<int64_t>(a.kh) * a.kw * a.C;
    int st;
    const void* T = a.T ? a.T : a.ws_T;
    void* dT = a.ws_G;
    auto recompute = [&] {   // the thin convolution (phase 1 of the forward only)
        const ChainConv cv{a.N, a.H, a.W, a.C, a.kh, a.kw, a.pad, a.stride};
        return chain(a.x, a.C, 0, 0, a.U, a.R, a.R, a.V, a.R, a.O, nullptr, a.O, a.ws_T, a.R, a.stream, &cv);
    };
    const bool flat = !a.lean && conv_flat_bwd_pays(a, a.dX != nullptr) && aligned16(a.dU) && aligned16(a.dV);
    // (Narrow rows that are read once or by dU alone lie as they are: without dX 64 -> 24 -> 64 of 25088 pixels 20.4 us, 20.9 at the pitch; one
    // tap, 160 -> 40 -> 160 of 50176 37.5 / 38.5, 64 -> 24 -> 64 of 100352 45.0 / 46.1.)
    const int64_t ldt = a.lean || (a.R < 64 && a.kh == 1) || (!a.dX && !flat && a.R < 32) ? a.R : conv_dt_pitch(a.R);
    const size_t copy_bytes = a.lean ? 0 : conv_factor_copy(P, a.kh, a.C, a.R, a.stride, false);
    const bool copy = a.dX && copy_bytes > 0;      // of U for dX; the launch that makes dT runs beside it
    char* const ws = a.ws + copy_bytes;
    const Operand U{copy ? a.ws : a.U, copy ? ldt : a.R, false, 0, false, true};
    const Before first = [&] {          // x U where there is no stash, and the copy of U
        const int rc = a.T ? PF_OK : recompute();
        const RepackJob job{a.U, a.R, a.ws, ldt, Keff, a.R};
        return rc != PF_OK || !copy || repack_rows_bf16_multi(&job, 1, a.stream) == cudaSuccess ? rc : PF_ERR_CUDA;
    };
    if (flat) {
        st = conv_flat_bwd(a, T, U.p, U.ld, ws, copy, first);
        *handled = st != PF_ERR_UNSUPPORTED;
        if (*handled) return st;
    }
    // Every product is prepared (tensor maps, geometry; nothing launched) before the call is
    // accepted, so a shape that one of them cannot take still reaches the FMA kernels.
    // dU[tap] = shifted x^T dT ; dV = dY^T T   (reductions over all output pixels, split across CTAs)
    // dX = sum over taps of shifted dT times U[tap]^T  (implicit GEMM over (tap, rank))
    const ConvA cu{2, a.N, a.H, a.W, a.C, a.R, a.Ho, a.Wo, a.kh, a.kw, a.pad, a.stride};
    ConvA cx = cu;
    cx.mode = 1;
    int su, sv;
    conv_splits(cu, a.O, &su, &sv);
    size_t bu, bv;
    conv_partial_bytes(cu, a.O, su, sv, &bu, &bv);
    const SliceRoom pu{reinterpret_cast<float*>(ws), bu}, pv{reinterpret_cast<float*>(ws + bu), bv};
    GemmLaunch gt, gu, gv, gx;
    st = gemm_prepare_any({a.dY, a.O, false, 0, false, copy}, {a.V, a.R, true, 0, false, copy}, P, a.R, a.O, dT, ldt, 1, {}, nullptr, &gt);
    // (the launch before these three writes dT only)
    if (st == PF_OK) st = gemm_prepare_any({a.x, a.C, true, 0, false, true}, {dT, ldt, true}, Keff, a.R, P, a.dU, a.R, su, pu, &cu, &gu);
    if (st == PF_OK) st = gemm_prepare_any({a.dY, a.O, true, 0, false, true}, {T, a.R, true, 0, false, true}, a.O, a.R, P, a.dV, a.R, sv, pv, nullptr, &gv);
    if (st == PF_OK && a.dX)
        st = gemm_prepare_any({dT, ldt, false}, U, static_cast<int64_t>(a.N) * a.H * a.W, a.C,
                     static_cast<int64_t>(a.kh) * a.kw * a.R, a.dX, a.C, 1, {}, &cx, &gx);
    if (st == PF_ERR_UNSUPPORTED) return PF_OK;      // declined: nothing has been launched
    if (st != PF_OK) return st;
    // dT: more tiles than two per SM, of few k-blocks each, go up to four to a block
    const int64_t gt_tiles = static_cast<int64_t>(gt.grid.x) * gt.grid.y;
    if (gt.p.nkb_total <= 8 && gt_tiles > 2 * num_sms()) {
        gt.runs = true;
        gt.grid = dim3(static_cast<unsigned>(ceil_div(gt_tiles, std::min<int64_t>(4, ceil_div(gt_tiles, 2 * num_sms())))));
        gt.p.num_stages = pick_stages(gt.bn, gt.grid.x, true);
    }
    st = first();
    if (st == PF_ERR_UNSUPPORTED) return PF_OK;
    *handled = 1;
    if (st != PF_OK) return st;
    const bool narrow = narrow_reductions(conv_du_tiles(a.kh, a.kw, a.C) * kBM, a.O, a.R);
    keep_slices(a.du_slices, &gu, narrow ? pu : SliceRoom(), a.C);
    keep_slices(a.dv_slices, &gv, narrow ? pv : SliceRoom());
    // dT = dY V  (per pixel)
    st = launch_prepared(gt, a.stream);
    if (st != PF_OK) return st;
    // dU, dV and dX depend on dT only and share one launch: the few long CTAs of the split reductions
    // start first and the many short dX tiles fill the second CTA slot of every SM beside them.
    const GemmLaunch* list[3] = {&gu, &gv, &gx};
    if (gu.p.splits <= 1 && gv.p.splits > 1) { list[0] = &gv; list[1] = &gu; }
    // (never declined: R <= 384 keeps the tiles at most 128 columns wide, and conv_splits fits the slices of both.)
    return gemm_multi(list, a.dX ? 3 : 2, a.stream);
}

}  // namespace tc
}  // namespace pf
