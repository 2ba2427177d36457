// Host side of the fused two-GEMM chain (kernel: pf_tc_chain_kernel.cuh): shape envelope, launch
// geometry, tensor maps, and the launch of the single-tile form.
#include <cuda.h>

#include <algorithm>

#include "pf_tc.h"
#include "pf_tc_host.h"
#include "pf_tc_chain_kernel.cuh"

namespace pf {
namespace tc {

// How the output pixels of a convolution are cut into blocks of at most `limit`: full-width rows of one
// image, as many as fit and about equally many per block, or several whole images when at least two fit.
ConvTiling conv_tiling(int N, int Ho, int Wo, int limit) {
    ConvTiling t;
    const int whole = static_cast<int>(std::min<int64_t>(N, limit / (static_cast<int64_t>(Ho) * Wo)));
    if (whole >= 2) {
        t.nb = whole; t.bh = Ho; t.tpi = 1;
    } else {
        t.nb = 1;
        t.tpi = static_cast<int>(ceil_div(Ho, std::max(1, limit / Wo)));
        t.bh = static_cast<int>(ceil_div(Ho, t.tpi));
    }
    t.pixels = t.nb * t.bh * Wo;
    t.blocks = ceil_div(N, t.nb) * t.tpi;
    return t;
}

// Shape envelope of the fused kernel and its launch geometry.
bool chain_plan(int64_t M, int64_t K1, int64_t N2, int64_t r, bool has_out, ChainPlan* plan, int rows_tile, int max_split, int groups) {
    const int64_t r_pad = (r + 63) / 64 * 64;
    if (r_pad > 384 || M > 0x7fffffff || K1 > 0x7fffffff || N2 > 0x7fffffff) return false;
    const int64_t stage = kTileBytes + r_pad * 128;
    // Small ranks: dedicated 32 KB store staging, and a whole B2 tile (r_pad / 64 boxes) per stage
    // in phase 2.  Larger ranks: staging lives in the idle B1 part of the stages, one box per stage.
    const bool dedicated = r_pad <= 128;
    const int64_t budget = 227 * 1024 - 2048 - r_pad * 256 - (dedicated ? 32768 : 0);
    int64_t ns = budget / stage;
    if (ns > kMaxStages) ns = kMaxStages;
    if (ns < 2 || (!dedicated && ns * (r_pad / 32) < 8)) return false;
    const int64_t row_tiles = ceil_div(M, rows_tile), all_tiles = row_tiles * groups, nt = ceil_div(N2, 128);
    // Split N2 over blockIdx.y while that shortens the critical path of a CTA (each split repeats
    // phase 1, cost ~ K1; phase 2 costs ~ N2 / split) and the grid still fits one wave.
    int64_t best = 1;
    if (has_out) {
        double best_cost = 1e30;
        for (int64_t s = 1; s <= nt && (s == 1 || all_tiles * s <= num_sms()) && (max_split <= 0 || s <= max_split); ++s) {
            const double waves = static_cast<double>(ceil_div(all_tiles * s, num_sms()));
            const double cost = waves * (static_cast<double>(K1) + 128.0 * ceil_div(nt, s));
            if (cost < best_cost * 0.97) { best_cost = cost; best = s; }
        }
    }
    plan->r_pad = static_cast<int>(r_pad);
    plan->num_stages = static_cast<int>(ns);
    plan->stage_bytes = static_cast<int>(stage);
    plan->nsplit = static_cast<int>(has_out ? best : 1);
    plan->tiles_per_split = has_out ? static_cast<int>(ceil_div(nt, best)) : 0;
    plan->nsplit = has_out ? static_cast<int>(ceil_div(nt, plan->tiles_per_split)) : 1;
    plan->smem = static_cast<size_t>(2048 + r_pad * 256 + ns * stage + (dedicated ? 32768 : 0));
    plan->boxes_per_stage = dedicated ? static_cast<int>(r_pad / 64) : 1;
    plan->staging_off = dedicated ? static_cast<int>(1024 + r_pad * 256 + ns * stage) : 0;
    plan->row_tiles = static_cast<int>(row_tiles);
    return true;
}

// out may be null (phase 1 only: T is written and nothing else).  All pointers must satisfy tma_ok, those of the caller's
// matrices that are written tma_out.
int chain(const void* A, int64_t lda, int64_t M, int64_t K1, const void* B1, int64_t ldb1, int64_t r,
          const void* B2, int64_t ldb2, int64_t N2, void* out, int64_t ldo, void* T, int64_t ldt,
          cudaStream_t stream, const ChainConv* conv, int max_split, const void* bias, int act, float keep_a, float keep_out, const Before& before) {
    ChainPlan plan;
    const int cs = conv ? conv->stride : 1;
    const int Ho = conv ? (conv->H + 2 * conv->pad - conv->kh) / cs + 1 : 1;
    const int Wo = conv ? (conv->W + 2 * conv->pad - conv->kw) / cs + 1 : 1;
    ConvTiling ct;
    if (conv) {
        if (Wo > 128) return PF_ERR_UNSUPPORTED;
        ct = conv_tiling(conv->N, Ho, Wo, 128);
        if (cs * Wo > 256 || cs * ct.bh > 256 || ct.nb > 256) return PF_ERR_UNSUPPORTED;
        M = ct.blocks * ct.pixels;                                  // rows of whole tiles
        K1 = static_cast<int64_t>(conv->kh) * conv->kw * ceil_div(conv->C, 64) * 64;
    }
    int rows_tile = conv ? ct.pixels : 128;
    if (!chain_plan(M, K1, N2, r, out != nullptr, &plan, rows_tile, max_split)) return PF_ERR_UNSUPPORTED;
    // Row tiles of 96 rows where they fit one wave: a block's time is that of its own rows through its SM's load and store
    // path, so SMs that 128-row tiles leave idle take some of them (the idle MMA rows cost nothing).  Not where the output
    // columns are split (148 instead of 128 blocks of an FFN layer delay the next launch's start: training step 1-3 %
    // slower), and not where another launch counts on the idle SMs (max_split).  Forward, 12000 rows, 768 -> 96 -> 3072:
    // 29.2 -> 25.1 us (125 blocks instead of 94; caches warm, 30.7 with a cold L2).  112 rows would help 16384-row layers by 1-2 % (147 blocks instead of 128),
    // but need output boxes of 16 rows, which slowed the 128-row tiles as much.
    if (!conv && out && max_split <= 0 && plan.nsplit == 1 && ceil_div(M, 96) <= num_sms()) rows_tile = 96;
    if (!conv) plan.row_tiles = static_cast<int>(ceil_div(M, rows_tile));
    CUtensorMap ta, tb1, tb2, to, tt;
    const bool ragged = conv && conv->C % 64 != 0;
    bool ok = conv ? cached_map_nhwc(&ta, A, conv->N, conv->H, conv->W, conv->C, Wo, ct.bh, ct.nb, cs) : cached_map_2d(&ta, A, M, K1, lda, rows_tile);
    ok = ok && (ragged ? cached_map_planes(&tb1, B1, static_cast<int64_t>(conv->kh) * conv->kw, conv->C, r, conv->C, 64, ldb1)
                       : cached_map_2d(&tb1, B1, K1, r, ldb1, 64));
    ok = ok && cached_map_2d(&tb2, B2, N2, r, ldb2, 128);
    if (conv) {   // outputs as windows of one tile's rows that start at any image row and end with the tile
        const int64_t starts = static_cast<int64_t>(conv->N) * Ho - static_cast<int64_t>(ct.nb) * ct.bh + 1;
        ok = ok && (out ? cached_map_planes(&to, out, starts, rows_tile, N2, Wo, 32) : cached_map_2d(&to, B2, N2, r, ldb2, 32));
        ok = ok && (T ? cached_map_planes(&tt, T, starts, rows_tile, r, Wo, rows_tile) : cached_map_2d(&tt, B2, N2, r, ldb2, 128));
    } else {
        ok = ok && (out ? cached_map_2d(&to, out, M, N2, ldo, 32) : cached_map_2d(&to, B2, N2, r, ldb2, 32));
        ok = ok && (T ? cached_map_2d(&tt, T, M, r, ldt, rows_tile) : cached_map_2d(&tt, B2, N2, r, ldb2, 128));
    }
    if (!ok) return PF_ERR_CUDA;
    const int st = before ? before() : PF_OK;
    if (st != PF_OK) return st;
    ChainParams p;
    p.M = static_cast<int>(M); p.K1 = static_cast<int>(K1); p.N2 = static_cast<int>(N2);
    // Zeros behind the rank for any number of rows, as the unfused products have them: 0.1 us where the rank is no multiple of
    // 64 (2641 x 768 -> 80 -> 768: 9.9 -> 10.0; 9000 x 512 -> 100 -> 512: 12.2 -> 12.4; 19500 x 512 -> 96 -> 512, pipelined: 15.4 both).
    p.r = conv ? plan.r_pad : static_cast<int>(r);
    p.r_pad = plan.r_pad; p.num_stages = plan.num_stages; p.stage_bytes = plan.stage_bytes;
    p.tiles_per_split = plan.tiles_per_split; p.store_T = T != nullptr;
    p.boxes_per_stage = plan.boxes_per_stage; p.staging_off = plan.staging_off;
    p.conv_cblks = 0; p.conv_kw = 1; p.conv_pad = 0; p.conv_stride = 1; p.conv_bh = 1; p.conv_nb = 1; p.conv_tpi = 1;
    p.conv_Ho = 1; p.conv_N = 1;
    if (conv) {
        p.conv_cblks = static_cast<int>(ceil_div(conv->C, 64)); p.conv_kw = conv->kw; p.conv_pad = conv->pad; p.conv_stride = cs;
        p.conv_bh = ct.bh; p.conv_nb = ct.nb; p.conv_tpi = ct.tpi; p.conv_Ho = Ho; p.conv_N = conv->N;
    }
    p.rows_tile = rows_tile;
    p.row_tiles = plan.row_tiles;
    // More row tiles than SMs: a persistent grid of equally loaded CTAs whose tiles overlap (phase 1 of
    // the next under the stores of the current), with the output accumulators behind T's in TMEM.
    int grid_x = plan.row_tiles;
    p.acc_base = 0; p.acc_bufs = kAccBufs;
    const bool persistent = plan.r_pad <= 128 && plan.nsplit == 1 && plan.row_tiles > num_sms();
    if (persistent) {
        const int per_cta = static_cast<int>(ceil_div(plan.row_tiles, num_sms()));
        grid_x = static_cast<int>(ceil_div(plan.row_tiles, per_cta));
        p.acc_base = 128; p.acc_bufs = 3;
    }
    p.bias = bias; p.act = act;
    p.status = device_status_ptr();
    p.keep[0] = keep_a; p.keep[1] = keep_out;
    dim3 grid(static_cast<unsigned>(grid_x), static_cast<unsigned>(plan.nsplit), 1);
    // (The persistent forms, which take over from 148 row tiles on, have no hints; with them they have not been measured.)
    if (!conv && !persistent && (keep_a != 0.f || keep_out != 0.f)) return chain_launch_hints(grid, plan.smem, stream, ta, tb1, tb2, to, tt, p);
    if (out && (bias || act)) return chain_launch_act(persistent, grid, plan.smem, stream, ta, tb1, tb2, to, tt, p);
    if (persistent) {
        // software-pipelined form: two T accumulators and two T buffers, the ring (four stages or more) behind them,
        // then the 32 KB of store staging; output accumulators in what tensor memory the T accumulators leave
        const int64_t stage = plan.stage_bytes, t2 = 2 * static_cast<int64_t>(plan.r_pad) * 256;
        int64_t ns = (227 * 1024 - 2048 - t2 - 32768) / stage;
        if (ns > kMaxStages) ns = kMaxStages;
        p.num_stages = static_cast<int>(ns);
        p.staging_off = static_cast<int>(1024 + t2 + ns * stage);
        p.boxes_per_stage = plan.r_pad / 64;
        p.acc_base = 2 * plan.r_pad;
        p.acc_bufs = (512 - 2 * plan.r_pad) / 128;
        const size_t smem = static_cast<size_t>(2048 + t2 + ns * stage + 32768);
        return conv ? chain_launch_conv(true, ragged, grid, smem, stream, ta, tb1, tb2, to, tt, p)
                    : chain_launch_pipe(grid, smem, stream, ta, tb1, tb2, to, tt, p);
    }
    if (conv) return chain_launch_conv(false, ragged, grid, plan.smem, stream, ta, tb1, tb2, to, tt, p);
    if (allow_smem(tc_chain_kernel<false, false, 0>, 227 * 1024) != cudaSuccess ||
        launch_overlapped(tc_chain_kernel<false, false, 0>, grid, dim3(kChainThreads), plan.smem, stream, ta, tb1, tb2, to, tt, p) !=
            cudaSuccess)
        return PF_ERR_CUDA;
    count_launch();
    return PF_OK;
}

// The chain for several groups of one shape, sA (0: one A read by all) ... sT elements apart; T may be null.
// The launch shares the machine with those of the other groups of `all`; late_wait: the launch before in the stream is one of them.
int chain_groups(int groups, int all, const void* A, int64_t lda, int64_t sA, int64_t M, int64_t K1, const void* B1, int64_t ldb1, int64_t sB1, int64_t r,
                 const void* B2, int64_t ldb2, int64_t sB2, int64_t N2, void* out, int64_t ldo, int64_t sO, void* T, int64_t ldt, int64_t sT,
                 bool late_wait, cudaStream_t stream) {
    ChainPlan plan;
    if (groups > 65535 || !chain_plan(M, K1, N2, r, true, &plan, 128, 0, all)) return PF_ERR_UNSUPPORTED;
    // (row tiles of 96 rows: see chain)
    const int rows_tile = plan.nsplit == 1 && ceil_div(M, 96) * all <= num_sms() ? 96 : 128;
    CUtensorMap ta, tb1, tb2, to, tt;
    const bool ok = cached_map_3d(&ta, A, sA == 0 ? 1 : groups, M, K1, lda, sA, rows_tile) && cached_map_3d(&tb1, B1, groups, K1, r, ldb1, sB1, 64) &&
                    cached_map_3d(&tb2, B2, groups, N2, r, ldb2, sB2, 128) &&
                    cached_map_3d(&to, out, groups, M, N2, ldo, sO, 32) &&
                    (T ? cached_map_3d(&tt, T, groups, M, r, ldt, sT, rows_tile) : cached_map_3d(&tt, B2, groups, N2, r, ldb2, sB2, 128));
    if (!ok) return PF_ERR_CUDA;
    ChainParams p = {};
    p.M = static_cast<int>(M); p.K1 = static_cast<int>(K1); p.N2 = static_cast<int>(N2);
    p.r = static_cast<int>(r); p.r_pad = plan.r_pad; p.num_stages = plan.num_stages; p.stage_bytes = plan.stage_bytes;
    p.tiles_per_split = plan.tiles_per_split; p.store_T = T != nullptr;
    p.boxes_per_stage = plan.boxes_per_stage; p.staging_off = plan.staging_off;
    p.conv_kw = p.conv_stride = p.conv_bh = p.conv_nb = p.conv_tpi = p.conv_Ho = p.conv_N = 1;
    p.rows_tile = rows_tile;
    p.row_tiles = static_cast<int>(ceil_div(M, rows_tile));
    p.acc_bufs = kAccBufs;
    p.status = device_status_ptr();
    p.group_flags[0] = sA == 0;
    p.group_flags[1] = late_wait;
    const dim3 grid(static_cast<unsigned>(p.row_tiles), static_cast<unsigned>(plan.nsplit), static_cast<unsigned>(groups));
    return chain_launch_groups(grid, plan.smem, stream, ta, tb1, tb2, to, tt, p);
}

}  // namespace tc
}  // namespace pf
