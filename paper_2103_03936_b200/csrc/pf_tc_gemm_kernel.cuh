// Product kernels of the tensor-core path (templates; host side in pf_tc.cu):
//   tc_gemm_kernel<BN>  C[M,N] = A * B for every operand orientation the factorized layers need
//                       (row-major operands read either along or across the contraction index,
//                       i.e. K-major or MN-major shared-memory descriptors), with an optional
//                       reduction split whose fp32 partials are summed in a fixed order.
//   tc_gemm3_kernel     up to three such products in one launch.
// Warp roles: warp 0 = TMA producer of operand A, warp 1 = TMEM allocation + MMA issue, warps 2..5 =
// epilogue (each owns the 32 TMEM lanes of its warp-id quadrant), warp 6 = TMA producer of operand B.
// The plain products are instantiated in pf_tc.cu, several tiles per block in pf_tc_runs.cu, the convolution's in
// pf_tc_conv.cu.
#ifndef PF_TC_GEMM_KERNEL_CUH_
#define PF_TC_GEMM_KERNEL_CUH_

#include <cuda.h>

#include "pf_tc_prims.cuh"

namespace pf {
namespace tc {

struct GemmParams {
    int M, N, K;
    int a_mn, b_mn;          // 1 = operand stored with the M/N index contiguous
    int kb_per_split;        // k-blocks handled by one z-slice
    int splits;
    int num_stages;
    int bn;                  // columns of an output tile (the kernel's template value; 64 or 128 in a shared launch)
    int tiles_x;             // row tiles of this product (tile id = column tile * tiles_x + row tile)
    void* C;                 // bf16 [M, ldc]
    long long ldc;
    void* C2;                // optional second copy of the result at another pitch, groups c2_gstride elements apart
    long long ldc2, c2_gstride;
    const void* bias;        // unsplit plain products: C = act(A B + bias), bias [N] in bf16 or null
    int act;
    float* partial;          // fp32 slices, one 128 x BN block per (tile, slice); an unsplit product that has it leaves its one slice there instead of writing C
    unsigned int* counters;  // splits > 1: two counters per tile
    unsigned int* status;
    // Implicit-GEMM convolution (conv_mode 0 = plain product); blocks of pixels are cv_bh full-width rows of cv_nb
    // images, cv_tpi blocks per image:
    //   conv_mode 1 (dX): A K-major = the image dT [N, Ho, Wo, R], B K-major = U as (taps * C) x R.  With stride s the
    //                     pixels of x fall into s x s classes by (row mod s, column mod s); the pixels of a class
    //                     see dT through the same few taps, at consecutive positions of dT.  A row tile is a
    //                     block of one class (cv_tiles_class blocks per class), a k-block is (tap of the class,
    //                     64-rank block); the output rows of a tile are s pixels apart.
    //   conv_mode 2 (dU): A MN-major = the image x, B MN-major = the image dT.  A row tile is two 64-channel blocks
    //                     of the unrolled factor (block = (tap, channel block), cv_blocks in all); a k-block is one
    //                     block of at most 64 output pixels, x read s pixels apart.
    int conv_mode, cv_blks, cv_kw, cv_kh, cv_pad, cv_stride, cv_C, cv_bh, cv_nb, cv_tpi;
    int cv_N, cv_H, cv_W, cv_bw, cv_inv_bw, cv_inv_bh, cv_tiles_class;   // dX: the image x and the width of a class's block
    int cv_blocks;           // dU
    int rows_tile;           // output rows per CTA: 128, or the pixels of a block for conv_mode 1
    int kpix;                // conv_mode 2: pixels per k-block (<= 64), else 64
    int ksteps;              // 16-element steps of a k-block that can be non-zero (1..4)
    int nkb_total;           // k-blocks of the whole contraction
    float keep_a;            // plain products: how L2 treats A (see l2_policy)
    int independent;         // 1: reads nothing the preceding kernel of the stream writes (see gemm_tile)
    int early;               // kEarlyA | kEarlyB: the operands of which that is true
    // Grouped products (several problems of one shape in a launch): tmA / tmB are 3-D maps whose outermost
    // coordinate is the group (a shared operand has one group only), outputs of group g start g * c_gstride
    // elements after C.  kb_per_group > 0 instead makes the group part of the CONTRACTION: k-block kb reads
    // group kb / kb_per_group, 64-element block kb % kb_per_group of both operands (the sum over groups of
    // A_g B_g^T, i.e. dX of several factor pairs that share one input).
    int groups, a_shared, b_shared, kb_per_group, tiles_y;
    long long c_gstride;
};

// Launches of the instantiations that have translation units of their own (pf_tc_runs.cu, pf_tc_conv.cu).
cudaError_t launch_gemm_runs(int bn, dim3 grid, size_t smem, cudaStream_t stream, const CUtensorMap& ta, const CUtensorMap& tb,
                             const GemmParams& p);
struct Gemm3Args {
    CUtensorMap ta[3], tb[3];
    GemmParams p[3];
    int end0, end1;
    int2 tiles[3];
};
cudaError_t launch_gemm3_conv(int blocks, size_t smem, cudaStream_t stream, const Gemm3Args& a);
// ... with products of any form (pf_tc_any.cu; see gemm_tile).
cudaError_t launch_gemm_any(int bn, dim3 grid, size_t smem, cudaStream_t stream, const CUtensorMap& ta, const CUtensorMap& tb, const GemmParams& p);
cudaError_t launch_gemm3_any(bool conv, int blocks, size_t smem, cudaStream_t stream, const Gemm3Args& a);

namespace {

constexpr int kBM = 128;       // rows of the output tile = TMEM lanes
constexpr int kBK = 64;        // contraction elements per pipeline stage (128 bytes of bf16)
constexpr int kMaxStages = 6;
constexpr uint32_t kDxPanel = 2048;      // staging of one epilogue warp of run_tiles, behind the stages
constexpr int kGemmThreads = 224;   // A producer, MMA issue, 4 epilogue warps, B producer

struct GemmCtl {
    uint64_t full[kMaxStages];
    uint64_t empty[kMaxStages];
    uint64_t tmem_full;
    uint64_t acc_full[2], acc_empty[2];      // run_tiles
    uint32_t tmem_base;
    uint32_t abort;
    uint32_t fix_ok;
};

// What a row tile covers: the first image, row and class of a convolution's block (unused otherwise).
struct TileOrigin {
    int img, row, ph, pw, na, nb, a0, b0;
};
template <int kMode>
__device__ __forceinline__ TileOrigin tile_origin(const GemmParams& p, int bx) {
    TileOrigin o = {};
    if constexpr (kMode == 1) {
        int t = bx;
        o.na = p.cv_kh;
        o.nb = p.cv_kw;
        if (p.cv_stride > 1) {       // (a handful of integer divisions, kept off the stride-1 tiles: these are short)
            const int s = p.cv_stride, cls = bx / p.cv_tiles_class;
            t = bx - cls * p.cv_tiles_class;
            o.ph = cls / s;
            o.pw = cls - o.ph * s;
            o.a0 = (o.ph + p.cv_pad) % s;            // first tap row / column of the class, and how many
            o.b0 = (o.pw + p.cv_pad) % s;
            o.na = (p.cv_kh - o.a0 + s - 1) / s;
            o.nb = (p.cv_kw - o.b0 + s - 1) / s;
        }
        const int g = p.cv_tpi > 1 ? t / p.cv_tpi : t;
        o.img = g * p.cv_nb;
        o.row = (t - g * p.cv_tpi) * p.cv_bh;
    }
    return o;
}
// Row of the output matrix that row r of tile bx holds, -1 if none.
template <int kMode>
__device__ __forceinline__ int output_row(const GemmParams& p, const TileOrigin& o, int bx, int r) {
    if constexpr (kMode == 0) {
        const int row = bx * kBM + r;
        return row < p.M ? row : -1;
    } else if constexpr (kMode == 1) {
        // r < 128, so multiplying by the rounded-up 2^16 / d divides exactly by the block's width and height
        const int line = (r * p.cv_inv_bw) >> 16, w = (r - line * p.cv_bw) * p.cv_stride + o.pw;
        const int i = (line * p.cv_inv_bh) >> 16, img = o.img + i, h = (o.row + line - i * p.cv_bh) * p.cv_stride + o.ph;
        return (r < p.rows_tile && img < p.cv_N && h < p.cv_H && w < p.cv_W) ? (img * p.cv_H + h) * p.cv_W + w : -1;
    } else {
        const int blk = bx * 2 + (r >> 6), tap = blk / p.cv_blks, c = (blk - tap * p.cv_blks) * 64 + (r & 63);
        return (blk < p.cv_blocks && c < p.cv_C) ? tap * p.cv_C + c : -1;
    }
}

// Four columns of a row, of which `left` exist, in the widest stores that the address takes.
__device__ __forceinline__ void store_columns(__nv_bfloat16* dst, uint32_t lo, uint32_t hi, int left) {
    unsigned short* d = reinterpret_cast<unsigned short*>(dst);
    const uint32_t off = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(dst)) & 7u;
    if (left >= 4) {
        if (off == 0) {
            *reinterpret_cast<uint2*>(d) = make_uint2(lo, hi);
        } else if ((off & 2u) == 0) {
            *reinterpret_cast<uint32_t*>(d) = lo;
            *reinterpret_cast<uint32_t*>(d + 2) = hi;
        } else {
            d[0] = static_cast<unsigned short>(lo);
            *reinterpret_cast<uint32_t*>(d + 1) = __funnelshift_r(lo, hi, 16);
            d[3] = static_cast<unsigned short>(hi >> 16);
        }
        return;
    }
    if (left > 0) d[0] = static_cast<unsigned short>(lo);
    if (left > 1) d[1] = static_cast<unsigned short>(lo >> 16);
    if (left > 2) d[2] = static_cast<unsigned short>(hi);
}

// One output tile (128 rows x BN columns) of C = A * B, or one slice of its contraction.
//
// Epilogue.  Unsplit: each epilogue warp turns its 32 accumulator rows into bf16, transposes them
// through a padded shared-memory panel and writes whole 128-byte row segments (any pitch, any
// alignment, clipped at the matrix edge).  Split: the fp32 slice goes to the workspace in the
// order [32-row quadrant][4-column group][row][4], which makes every store instruction of a warp
// one contiguous 512-byte run; then the CTAs of a tile meet at a counter and each sums, in slice
// order, its share over all slices and writes bf16 (bit-reproducible, no second launch).
// kMode: 0 = plain (or grouped) product, 2 = dU of a convolution (dX: run_tiles), compiled apart so that the plain
// kernels carry none of its code (with all of them in one kernel the FFN backward ran 12 % slower).
// kAny: any output rows, second copies, bias and activation, one fp32 slice instead of C.  Without it: rows of whole 16-byte
// pieces and none of that; the code behind the main loop runs once, from a cold instruction cache, so what a product does
// not need is not compiled into its kernel (all of it in one kernel: backward of 8192 x 2048 -> 128 -> 512 30.0 us, apart 28.5; 64 x 512 ->
// 128 -> 512: 8.6 and 8.0).
template <int BN, int kMode, bool kAny>
__device__ __forceinline__ void gemm_tile(const CUtensorMap& tmA, const CUtensorMap& tmB, const GemmParams& p,
                                          const int bx, const int by, const int bz, const int bg) {
    constexpr uint32_t kABytes = kBM * kBK * 2;          // 16 KB
    constexpr uint32_t kBBytes = BN * kBK * 2;
    constexpr uint32_t kStageBytes = kABytes + kBBytes;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    uint8_t* smem = smem_raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);
    GemmCtl* ctl = reinterpret_cast<GemmCtl*>(smem);
    uint8_t* tiles = smem + 1024;
    volatile uint32_t* abort_flag = &ctl->abort;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = bx * kBM, n0 = by * BN;
    const TileOrigin org = tile_origin<kMode>(p, bx);
    const int kb_beg = bz * p.kb_per_split;
    const int kb_end = min(p.nkb_total, kb_beg + p.kb_per_split);
    const int nkb = kb_end - kb_beg;
    const uint32_t NS = static_cast<uint32_t>(p.num_stages);
    const int tile = (bg * p.tiles_y + by) * p.tiles_x + bx;
    const bool grouped = p.groups > 1 || p.kb_per_group > 0;

    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&ctl->full[s]), 2);     // one expect_tx arrival per producer thread
            mbar_init(smem_u32(&ctl->empty[s]), 1);
        }
        mbar_init(smem_u32(&ctl->tmem_full), 1);
        ctl->abort = 0;
        ctl->fix_ok = 0;
        fence_barrier_init();
        fence_proxy_async_smem();
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
    }
    if (kMode == 2 && (p.kpix & 15) != 0) {
        // k-blocks end inside a 16-pixel step: the unused contraction rows of that step must be zero in every
        // 64-column panel of both operands (TMA never writes them), so that they add nothing to the sum
        const int rows = 16 - (p.kpix & 15);
        const int pieces = rows * 8, panels = static_cast<int>(kStageBytes / 8192) * static_cast<int>(NS);
        for (int i = threadIdx.x; i < panels * pieces; i += blockDim.x) {
            const int panel = i / pieces, piece = i - panel * pieces;
            *reinterpret_cast<uint4*>(tiles + panel * 8192 + p.kpix * 128 + piece * 16) = make_uint4(0, 0, 0, 0);
        }
        fence_proxy_async_smem();
    }
    if (warp == 1) tmem_alloc(smem_u32(&ctl->tmem_base), BN);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // A product marked independent reads nothing that the kernel launched just before it writes, so
    // it does not wait for that kernel: its blocks run beside it on SMs that kernel leaves free.  (The kernels
    // of this library let their successors start only after their own wait has returned, i.e. once
    // everything older in the stream is complete, so older results are safe to read; the exceptions are named at kEarlyA.)
    // The same holds for a single operand (p.early): its producer fills the ring beside the previous kernel's tail.
    const bool ahead = p.independent || (warp == 0 && (p.early & kEarlyA)) || (warp == 6 && (p.early & kEarlyB));
    if (!ahead) pdl_wait();             // everything above overlapped the previous kernel's tail
    if (!ahead || p.independent) pdl_launch_dependents();
    const uint32_t tmem_base = ctl->tmem_base;

    // Producers and MMA issuer are each one thread chosen with elect.sync that runs its whole role
    // (a thread singled out by a lane-id test issues TMA / tcgen05 instructions several times slower).
    // Two producers, one per operand: a producer thread needs about 130 ns per stage for its loop,
    // barrier wait and expect_tx plus 40 ns per TMA instruction, which with four tile loads per
    // stage paced the whole pipeline when one thread issued both operands.
    if (warp == 0 || warp == 6) {
        if (elect_one()) {
            const bool do_a = warp == 0;
            const bool two = kMode != 2 || bx * 2 + 1 < p.cv_blocks;      // the tile's second channel block exists
            const uint32_t my_bytes = kMode == 2 ? static_cast<uint32_t>(p.kpix) * (do_a ? (two ? 256u : 128u) : BN * 2u)
                                                 : do_a ? kABytes : kBBytes;
            // One loop per addressing mode, its positions carried as counters in registers: whatever the thread
            // does per k-block beyond waiting and issuing paces the pipeline.
            const uint32_t base = smem_u32(tiles) + (do_a ? 0u : kABytes);
            const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
            auto produce = [&](auto&& issue) {
                uint32_t s = 0, ph = 1, dst = base;
                for (int i = 0; i < nkb; ++i) {
                    if (!mbar_wait(empty0 + 8 * s, ph, abort_flag, p.status)) break;
                    const uint32_t full = full0 + 8 * s;
                    mbar_expect_tx(full, my_bytes);
                    issue(dst, full);
                    dst += kStageBytes;
                    if (++s == NS) { s = 0; dst = base; ph ^= 1u; }
                }
            };
            int k0 = kb_beg * kBK;
            if constexpr (kMode == 2) {
                const int bh = p.cv_bh, nimg = p.cv_nb, tpi = p.cv_tpi;
                const int g = kb_beg / tpi;
                int t = kb_beg - g * tpi, img = g * nimg;
                if (do_a) {
                    const int blks = p.cv_blks, kw = p.cv_kw, step = bh * p.cv_stride;
                    const int tap0 = bx * 2 / blks, tap1 = (bx * 2 + 1) / blks, ta0 = tap0 / kw, ta1 = tap1 / kw;
                    const int c0 = (bx * 2 - tap0 * blks) * 64, c1 = (bx * 2 + 1 - tap1 * blks) * 64;
                    const int x0 = tap0 - ta0 * kw - p.cv_pad, x1 = tap1 - ta1 * kw - p.cv_pad;
                    int y = t * step + ta0 - p.cv_pad;
                    const int dy = ta1 - ta0, rewind = tpi * step;
                    produce([&](uint32_t dst, uint32_t full) {
                        tma_load_4d(dst, &tmA, full, c0, x0, y, img);
                        if (two) tma_load_4d(dst + 8192, &tmA, full, c1, x1, y + dy, img);
                        y += step;
                        if (++t == tpi) { t = 0; y -= rewind; img += nimg; }
                    });
                } else {
                    int row = t * bh;
                    produce([&](uint32_t dst, uint32_t full) {
#pragma unroll
                        for (int h = 0; h < BN / 64; ++h) tma_load_4d(dst + h * 8192, &tmB, full, n0 + 64 * h, 0, row, img);
                        row += bh;
                        if (++t == tpi) { t = 0; row = 0; img += nimg; }
                    });
                }
            } else if (grouped) {
                int g = bg, left = 0x7fffffff;            // k-blocks left of group g (groups inside the contraction)
                if (p.kb_per_group > 0) {
                    g = kb_beg / p.kb_per_group;
                    left = (g + 1) * p.kb_per_group - kb_beg;
                    k0 -= g * p.kb_per_group * kBK;
                }
                auto advance = [&] {
                    k0 += kBK;
                    if (--left == 0) { ++g; k0 = 0; left = p.kb_per_group; }
                };
                if (do_a && p.a_mn) {
                    produce([&](uint32_t dst, uint32_t full) {
                        tma_load_3d(dst, &tmA, full, m0, k0, p.a_shared ? 0 : g);
                        tma_load_3d(dst + 8192, &tmA, full, m0 + 64, k0, p.a_shared ? 0 : g);
                        advance();
                    });
                } else if (do_a) {
                    produce([&](uint32_t dst, uint32_t full) {
                        tma_load_3d(dst, &tmA, full, k0, m0, p.a_shared ? 0 : g);
                        advance();
                    });
                } else if (p.b_mn) {
                    produce([&](uint32_t dst, uint32_t full) {
#pragma unroll
                        for (int h = 0; h < BN / 64; ++h) tma_load_3d(dst + h * 8192, &tmB, full, n0 + 64 * h, k0, p.b_shared ? 0 : g);
                        advance();
                    });
                } else {
                    produce([&](uint32_t dst, uint32_t full) {
                        tma_load_3d(dst, &tmB, full, k0, n0, p.b_shared ? 0 : g);
                        advance();
                    });
                }
            } else if (do_a && p.a_mn) {
                const uint64_t policy = l2_policy(p.keep_a);
                produce([&](uint32_t dst, uint32_t full) {
                    tma_load_2d(dst, &tmA, full, m0, k0, policy);
                    tma_load_2d(dst + 8192, &tmA, full, m0 + 64, k0, policy);
                    k0 += kBK;
                });
            } else if (do_a) {
                produce([&](uint32_t dst, uint32_t full) { tma_load_2d(dst, &tmA, full, k0, m0); k0 += kBK; });
            } else if (p.b_mn) {
                produce([&](uint32_t dst, uint32_t full) {
#pragma unroll
                    for (int h = 0; h < BN / 64; ++h) tma_load_2d(dst + h * 8192, &tmB, full, n0 + 64 * h, k0);
                    k0 += kBK;
                });
            } else {
                produce([&](uint32_t dst, uint32_t full) { tma_load_2d(dst, &tmB, full, k0, n0); k0 += kBK; });
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            const uint32_t idesc = make_idesc_bf16(kBM, BN, p.a_mn, p.b_mn);
            // K-major: 8-row groups 1024 B apart, 16 contraction elements = 32 B along the row.
            // MN-major: 64-element M/N panels 8192 B apart (LBO), 8 contraction rows per
            // 1024 B group (SBO), 16 contraction rows = 2048 B.
            const uint32_t a_step = p.a_mn ? 128u : 2u, b_step = p.b_mn ? 128u : 2u;   // in 16-byte units
            const uint32_t a_addr = smem_u32(tiles), b_addr = a_addr + kABytes;
            const uint64_t a_desc0 = p.a_mn ? make_smem_desc(a_addr, 8192, 1024) : make_smem_desc(a_addr, 16, 1024);
            const uint64_t b_desc0 = p.b_mn ? make_smem_desc(b_addr, 8192, 1024) : make_smem_desc(b_addr, 16, 1024);
            const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
            const int ksteps = p.ksteps;
            uint32_t s = 0, ph = 0, off = 0;
            bool ok = true;
            for (int i = 0; i < nkb; ++i) {
                ok = mbar_wait(full0 + 8 * s, ph, abort_flag, p.status);
                if (!ok) break;
                tc_fence_after();
                const uint64_t a_desc = a_desc0 + off, b_desc = b_desc0 + off;
                tc_mma_bf16(tmem_base, a_desc, b_desc, idesc, i > 0 ? 1u : 0u);
                if (kMode == 0 || ksteps == 4) {
                    tc_mma_bf16(tmem_base, a_desc + a_step, b_desc + b_step, idesc, 1u);
                    tc_mma_bf16(tmem_base, a_desc + 2 * a_step, b_desc + 2 * b_step, idesc, 1u);
                    tc_mma_bf16(tmem_base, a_desc + 3 * a_step, b_desc + 3 * b_step, idesc, 1u);
                } else {
                    if (ksteps > 1) tc_mma_bf16(tmem_base, a_desc + a_step, b_desc + b_step, idesc, 1u);
                    if (ksteps > 2) tc_mma_bf16(tmem_base, a_desc + 2 * a_step, b_desc + 2 * b_step, idesc, 1u);
                }
                tc_commit(empty0 + 8 * s);             // frees the stage once these MMAs have read it
                off += kStageBytes >> 4;
                if (++s == NS) { s = 0; off = 0; ph ^= 1u; }
            }
            if (ok) tc_commit(smem_u32(&ctl->tmem_full));
        }
    } else if (warp < 6) {
        const int q = warp & 3;                          // TMEM lane quadrant this warp may access
        const bool ok = mbar_wait_warp(smem_u32(&ctl->tmem_full), 0, abort_flag, p.status);
        tc_fence_after();
        if (ok) {
            const uint32_t lane_base = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
            if (kAny ? p.partial != nullptr : p.splits > 1) {
                // fp32 slice: straight from registers, [quadrant][4-column group][row][4], so that every store
                // instruction of a warp is one run of 512 bytes; then the warp reports
                float* dst = p.partial + (static_cast<size_t>(tile) * p.splits + bz) * (kBM * BN) +
                             static_cast<size_t>(q * (BN / 4) * 32 + lane) * 4;
#pragma unroll 1
                for (int c = 0; c < BN / 64; ++c) {
                    uint32_t v[2][32];
                    tmem_ld32(lane_base + c * 64, v[0]);
                    tmem_ld32(lane_base + c * 64 + 32, v[1]);
                    tmem_ld_wait();
#pragma unroll
                    for (int g = 0; g < 16; ++g)
                        *reinterpret_cast<uint4*>(dst + static_cast<size_t>(c * 16 + g) * 128) =
                            make_uint4(v[g >> 3][4 * (g & 7)], v[g >> 3][4 * (g & 7) + 1], v[g >> 3][4 * (g & 7) + 2], v[g >> 3][4 * (g & 7) + 3]);
                }
                __syncwarp();
                if (lane == 0 && (!kAny || p.splits > 1)) red_release_gpu(p.counters + 2 * tile, 1u);
            } else {
                // every MMA has completed, so the pipeline stages are free: 16 KB of vector panels, then word panels
                uint32_t* stg = reinterpret_cast<uint32_t*>(tiles + 16384) + (warp - 2) * (32 * kRaggedWords);
                __nv_bfloat16* Cb = reinterpret_cast<__nv_bfloat16*>(p.C) + static_cast<long long>(bg) * p.c_gstride;
                const bool vec_ok = !kAny || ((p.ldc % 8) == 0 && (reinterpret_cast<uintptr_t>(Cb) & 15) == 0);
                if (vec_ok) {
                    // 16-byte aligned rows: stage 32 rows x 64 columns (128 bytes per row, 16-byte pieces
                    // XOR-swizzled by the row so that both passes are free of bank conflicts), then
                    // store four whole 128-byte row segments per instruction
                    const uint32_t panel = smem_u32(tiles) + static_cast<uint32_t>(warp - 2) * 4096u;
                    const uint32_t own = panel + static_cast<uint32_t>(lane) * 128u, sw = static_cast<uint32_t>(lane & 7);
                    const int sub = lane >> 3, piece = lane & 7;
                    int orow[8];              // output rows of this thread's pieces, -1 = not stored
#pragma unroll
                    for (int i = 0; i < 8; ++i) orow[i] = output_row<kMode>(p, org, bx, q * 32 + i * 4 + sub);
#pragma unroll 1
                    for (int c = 0; c < BN / 64; ++c) {
                        uint32_t v0[32], v1[32];
                        tmem_ld32(lane_base + c * 64, v0);
                        tmem_ld32(lane_base + c * 64 + 32, v1);
                        tmem_ld_wait();
                        if (kAny && kMode == 0 && (p.bias || p.act)) bias_act64(v0, v1, p.bias, p.act, n0 + c * 64, p.N, lane);
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            uint4 o;
                            o.x = pack_bf16x2(__uint_as_float(v0[8 * t + 0]), __uint_as_float(v0[8 * t + 1]));
                            o.y = pack_bf16x2(__uint_as_float(v0[8 * t + 2]), __uint_as_float(v0[8 * t + 3]));
                            o.z = pack_bf16x2(__uint_as_float(v0[8 * t + 4]), __uint_as_float(v0[8 * t + 5]));
                            o.w = pack_bf16x2(__uint_as_float(v0[8 * t + 6]), __uint_as_float(v0[8 * t + 7]));
                            st_shared_v4(own + ((static_cast<uint32_t>(t) ^ sw) << 4), o);
                            o.x = pack_bf16x2(__uint_as_float(v1[8 * t + 0]), __uint_as_float(v1[8 * t + 1]));
                            o.y = pack_bf16x2(__uint_as_float(v1[8 * t + 2]), __uint_as_float(v1[8 * t + 3]));
                            o.z = pack_bf16x2(__uint_as_float(v1[8 * t + 4]), __uint_as_float(v1[8 * t + 5]));
                            o.w = pack_bf16x2(__uint_as_float(v1[8 * t + 6]), __uint_as_float(v1[8 * t + 7]));
                            st_shared_v4(own + ((static_cast<uint32_t>(4 + t) ^ sw) << 4), o);
                        }
                        __syncwarp();
                        const int col = n0 + c * 64 + piece * 8;
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const int rr = i * 4 + sub;
                            const uint4 w = ld_shared_v4(panel + static_cast<uint32_t>(rr) * 128u +
                                                         ((static_cast<uint32_t>(piece) ^ static_cast<uint32_t>(rr & 7)) << 4));
                            if (orow[i] >= 0) {
                                __nv_bfloat16* dst = Cb + static_cast<size_t>(orow[i]) * p.ldc + col;
                                if (col + 8 <= p.N) {
                                    *reinterpret_cast<uint4*>(dst) = w;
                                } else {
                                    const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                                    for (int e = 0; e < 8; ++e)
                                        if (col + e < p.N)
                                            dst[e] = __ushort_as_bfloat16(static_cast<unsigned short>((ws[e >> 1] >> ((e & 1) * 16)) & 0xffffu));
                                }
                            }
                        }
                        if (kAny && p.C2) {          // the second copy, at a pitch that the first cannot have
                            stage_ragged(stg, v0, v1, lane);
                            __syncwarp();
                            store_ragged(stg, reinterpret_cast<__nv_bfloat16*>(p.C2) + static_cast<long long>(bg) * p.c2_gstride, p.ldc2, n0 + c * 64,
                                         p.N, lane, [&](int r) { return output_row<kMode>(p, org, bx, q * 32 + r); });
                        }
                        __syncwarp();
                    }
                } else if constexpr (kAny) {
#pragma unroll 1
                    for (int c = 0; c < BN / 64; ++c) {
                        uint32_t v0[32], v1[32];
                        tmem_ld32(lane_base + c * 64, v0);
                        tmem_ld32(lane_base + c * 64 + 32, v1);
                        tmem_ld_wait();
                        if (kAny && kMode == 0 && (p.bias || p.act)) bias_act64(v0, v1, p.bias, p.act, n0 + c * 64, p.N, lane);
                        stage_ragged(stg, v0, v1, lane);
                        __syncwarp();
                        store_ragged(stg, Cb, p.ldc, n0 + c * 64, p.N, lane, [&](int r) { return output_row<kMode>(p, org, bx, q * 32 + r); });
                        __syncwarp();
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, BN);
    if (p.splits <= 1) return;

    // ---- slice sum: wait until every slice of this tile is in the workspace (four warps of every slice report), then
    // sum a share of it, in slice order (bit-reproducible).  A warp sums units of 8 rows x 32 columns, up to eight
    // slices of a unit (16 loads per lane) in flight together, 32 bytes stored per row and 16 columns.  What bounds
    // it is latency: registers to workspace to registers, without shared memory in between, replaced a bulk copy out, the
    // fences between the proxies and a bulk copy back, which together took 6.3 us from the last MMA to the stored sum
    // (7 slices of 128 x 128).  Backward of 8192 rows, 512 -> 128 -> 2048: 24.6 -> 22.6 us; 1070 rows, 888 -> 208 ->
    // 3552: 28.0 -> 26.3.  One version of short code: it runs once, from a cold instruction cache, and variants per slice
    // count with deeper unrolling lost up to 5 us.  (Half the loads in flight: 24.2 and 28.8 us.)  All of these back to
    // back on one set of buffers, caches warm; with a cold L2 the two take 33.8 and 31.7 us.
    unsigned int* cnt = p.counters + 2 * tile;
    const int S = p.splits;
    if (threadIdx.x == 0) {
        uint32_t good = (*abort_flag == 0u) ? 1u : 0u;
        const unsigned int want = 4u * static_cast<unsigned int>(S);
        const long long t0 = clock64();
        while (good && ld_acquire_gpu(cnt) < want) {
            if (clock64() - t0 > kWaitCycleLimit) {
                good = 0u;
                if (p.status) atomicExch(p.status, kStatusTimeout);
            }
        }
        ctl->fix_ok = good;
    }
    __syncthreads();
    if (ctl->fix_ok) {
        __nv_bfloat16* Cb = reinterpret_cast<__nv_bfloat16*>(p.C) + static_cast<long long>(bg) * p.c_gstride;
        __nv_bfloat16* C2b = kAny && p.C2 ? reinterpret_cast<__nv_bfloat16*>(p.C2) + static_cast<long long>(bg) * p.c2_gstride : nullptr;
        // units of 8 rows x 32 columns: a lane holds two 4-column groups of a row, 16 columns apart
        constexpr int kUnits = kBM / 8 * (BN / 32);
        constexpr size_t kSlice = static_cast<size_t>(kBM) * BN / 4;       // float4s
        const int per = (kUnits + S - 1) / S, end = min(kUnits, (bz + 1) * per);
#pragma unroll 1
        for (int u = bz * per + warp; u < end; u += kGemmThreads / 32) {
            const int oct = u / (BN / 32), pc = (u - oct * (BN / 32)) * 8 + (lane >> 3), rr = oct * 8 + (lane & 7);
            const float4* src = reinterpret_cast<const float4*>(p.partial) + static_cast<size_t>(tile) * S * kSlice +
                                ((rr >> 5) * (BN / 4) + pc) * 32 + (rr & 31);
            float4 acc[2];
            acc[0] = acc[1] = make_float4(-0.f, -0.f, -0.f, -0.f);
#pragma unroll 1
            for (int s0 = 0; s0 < S; s0 += 8) {
                float4 w[8][2];
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (s0 + i < S) {
                        w[i][0] = __ldcg(src + static_cast<size_t>(s0 + i) * kSlice);
                        w[i][1] = __ldcg(src + static_cast<size_t>(s0 + i) * kSlice + 4 * 32);
                    }
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (s0 + i < S) {
#pragma unroll
                        for (int j = 0; j < 2; ++j) { acc[j].x += w[i][j].x; acc[j].y += w[i][j].y; acc[j].z += w[i][j].z; acc[j].w += w[i][j].w; }
                    }
            }
            const int row = output_row<kMode>(p, org, bx, rr);
            if (row < 0) continue;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int col = n0 + pc * 4 + j * 16;
                __nv_bfloat16* dst = Cb + static_cast<size_t>(row) * p.ldc + col;
                const uint32_t lo = pack_bf16x2(acc[j].x, acc[j].y), hi = pack_bf16x2(acc[j].z, acc[j].w);
                if (!kAny && col + 3 < p.N) *reinterpret_cast<uint2*>(dst) = make_uint2(lo, hi);
                else store_columns(dst, lo, hi, p.N - col);
                // the same sums once more, for a destination whose pitch the first cannot have
                if (kAny && C2b) store_columns(C2b + static_cast<size_t>(row) * p.ldc2 + col, lo, hi, p.N - col);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && ctl->fix_ok) {
        const unsigned int left = atomicAdd(cnt + 1, 1u);
        if (left + 1u == static_cast<unsigned int>(S)) {   // every slice has read what it needs
            cnt[0] = 0u;
            cnt[1] = 0u;
            __threadfence();
        }
    }
}

// Row and column tile of tile t of dX.  The classes of a block of pixels follow one another, so that blocks whose tiles are
// a number apart that shares no factor with the stride take tiles of every class.
template <int kMode>
__device__ __forceinline__ int run_tile(const GemmParams& p, int t, int* by) {
    *by = t / p.tiles_x;
    const int bx = t - *by * p.tiles_x;
    if (kMode == 0 || p.cv_stride == 1) return bx;
    const int classes = p.cv_stride * p.cv_stride, block = bx / classes;
    return (bx - block * classes) * p.cv_tiles_class + block;
}
// dX of a convolution (conv_mode 1): output tiles first, first + step, ... of 128 rows x BN columns.  A tile has few
// k-blocks (taps of its class x 64-rank blocks: 9 at stride 1, 1 to 4 at stride 2), so with one tile per block the
// start, the first loads and the epilogue cost as much as the products.  Here the producers run on into the next tiles
// while the epilogue warps store the last one from the other of two accumulators.  What bounds it now is the SM's load
// path.  Whole backward, one tile per block -> runs: 128 x 32 x 32, 128 -> 64 -> 256, stride 2: 42 -> 34 us; 128 x 16 x 16,
// 512 -> 128 -> 512: 114 -> 91 (against 256-column tiles); 128 x 32 x 32, 256 -> 64 -> 256: 122 -> 117 (back to back,
// caches warm, dT still one tile per block; with its runs 30.7, 90.5 and 114.6, with a cold L2 39.9, 101 and 128).
template <int BN, int kMode>
__device__ __forceinline__ void run_tiles(const CUtensorMap& tmA, const CUtensorMap& tmB, const GemmParams& p, const int first, const int step) {
    constexpr uint32_t kABytes = kBM * kBK * 2, kBBytes = BN * kBK * 2, kStageBytes = kABytes + kBBytes;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    uint8_t* smem = smem_raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);
    GemmCtl* ctl = reinterpret_cast<GemmCtl*>(smem);
    const uint32_t tiles = smem_u32(smem) + 1024u;
    volatile uint32_t* abort_flag = &ctl->abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t NS = static_cast<uint32_t>(p.num_stages);
    const int ntiles = p.tiles_x * p.tiles_y;

    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&ctl->full[s]), 2);
            mbar_init(smem_u32(&ctl->empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&ctl->acc_full[b]), 1);
            mbar_init(smem_u32(&ctl->acc_empty[b]), 4);
        }
        ctl->abort = 0;
        fence_barrier_init();
        fence_proxy_async_smem();
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
    }
    if (warp == 1) tmem_alloc(smem_u32(&ctl->tmem_base), 2 * BN);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const bool ahead = (warp == 0 && (p.early & kEarlyA)) || (warp == 6 && (p.early & kEarlyB));      // (see gemm_tile)
    if (!ahead) {
        pdl_wait();
        pdl_launch_dependents();
    }
    const uint32_t tmem_base = ctl->tmem_base;
    const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);

    if (warp == 0 || warp == 6) {
        if (elect_one()) {
            const bool do_a = warp == 0;
            const uint32_t my_bytes = do_a ? static_cast<uint32_t>(p.rows_tile) * 128u : kBBytes;
            const uint32_t base = tiles + (do_a ? 0u : kABytes);
            const int blks = p.cv_blks;
            uint32_t s = 0, ph = 1, dst = base;
            bool ok = true;
            for (int t = first; t < ntiles && ok; t += step) {
                int by;
                const int bx = run_tile<kMode>(p, t, &by);
                const TileOrigin org = tile_origin<kMode>(p, bx);
                const int ntb = org.nb, nkb = kMode == 1 ? org.na * ntb * blks : p.nkb_total;
                auto produce = [&](auto&& issue) {
                    for (int i = 0; i < nkb; ++i) {
                        ok = mbar_wait(empty0 + 8 * s, ph, abort_flag, p.status);
                        if (!ok) break;
                        const uint32_t full = full0 + 8 * s;
                        mbar_expect_tx(full, my_bytes);
                        issue(dst, full);
                        dst += kStageBytes;
                        if (++s == NS) { s = 0; dst = base; ph ^= 1u; }
                    }
                };
                int rb = 0, tb = 0;
                if constexpr (kMode == 0) {
                    if (do_a) {
                        produce([&](uint32_t to, uint32_t full) { tma_load_2d(to, &tmA, full, rb, bx * kBM); rb += kBK; });
                    } else {
                        produce([&](uint32_t to, uint32_t full) {
#pragma unroll
                            for (int h = 0; h < BN / 64; ++h) tma_load_2d(to + h * 8192, &tmB, full, by * BN + 64 * h, rb);
                            rb += kBK;
                        });
                    }
                } else if (do_a) {
                    const int y0 = org.ph + p.cv_pad - org.a0, xx = org.pw + p.cv_pad - org.b0;      // multiples of the stride
                    int y = org.row + (p.cv_stride > 1 ? y0 / p.cv_stride : y0);
                    const int x0 = p.cv_stride > 1 ? xx / p.cv_stride : xx, img = org.img;
                    produce([&](uint32_t to, uint32_t full) {
                        tma_load_4d(to, &tmA, full, rb * 64, x0 - tb, y, img);
                        if (++rb == blks) { rb = 0; if (++tb == ntb) { tb = 0; --y; } }
                    });
                } else {
                    int line = (org.a0 * p.cv_kw + org.b0) * p.cv_C + by * BN, at = line;      // row of U
                    const int step_b = p.cv_stride * p.cv_C, step_a = step_b * p.cv_kw;
                    produce([&](uint32_t to, uint32_t full) {
                        tma_load_2d(to, &tmB, full, rb * 64, at);
                        if (++rb == blks) {
                            rb = 0; at += step_b;
                            if (++tb == ntb) { tb = 0; line += step_a; at = line; }
                        }
                    });
                }
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            constexpr uint32_t kStepB = kMode == 0 ? 128 : 2;      // (plain: B is MN-major)
            const uint32_t idesc = make_idesc_bf16(kBM, BN, 0, kMode == 0);
            const uint64_t a_desc0 = make_smem_desc(tiles, 16, 1024), b_desc0 = make_smem_desc(tiles + kABytes, kMode == 0 ? 8192 : 16, 1024);
            const int ksteps = p.ksteps;
            uint32_t s = 0, ph = 0, off = 0, buf = 0, bph = 1;
            bool ok = true;
            for (int t = first; t < ntiles && ok; t += step) {
                int nkb = p.nkb_total;
                if constexpr (kMode == 1) {
                    int by;
                    const TileOrigin org = tile_origin<1>(p, run_tile<1>(p, t, &by));
                    nkb = org.na * org.nb * p.cv_blks;
                }
                ok = mbar_wait(smem_u32(&ctl->acc_empty[buf]), bph, abort_flag, p.status);
                if (!ok) break;
                tc_fence_after();
                const uint32_t d = tmem_base + buf * BN;
                for (int i = 0; i < nkb; ++i) {
                    ok = mbar_wait(full0 + 8 * s, ph, abort_flag, p.status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t a = a_desc0 + off, b = b_desc0 + off;
                    tc_mma_bf16(d, a, b, idesc, i > 0 ? 1u : 0u);
#pragma unroll
                    for (int k = 1; k < 4; ++k)
                        if (kMode == 0 || k < ksteps) tc_mma_bf16(d, a + 2 * k, b + kStepB * k, idesc, 1u);
                    tc_commit(empty0 + 8 * s);
                    off += kStageBytes >> 4;
                    if (++s == NS) { s = 0; off = 0; ph ^= 1u; }
                }
                if (ok) tc_commit(smem_u32(&ctl->acc_full[buf]));
                buf ^= 1u;
                if (buf == 0) bph ^= 1u;
            }
        }
    } else if (warp < 6) {
        const int q = warp & 3, sub = lane >> 2, piece = lane & 3;
        // 32 rows x 32 columns per warp behind the stages: rows of 64 bytes, their 16-byte pieces XOR-permuted
        const uint32_t panel = tiles + NS * kStageBytes + static_cast<uint32_t>(q) * kDxPanel;
        const uint32_t own = panel + static_cast<uint32_t>(lane) * 64u, sw = static_cast<uint32_t>(lane >> 1) & 3u;
        __nv_bfloat16* C = reinterpret_cast<__nv_bfloat16*>(p.C);
        uint32_t buf = 0, bph = 0;
        for (int t = first; t < ntiles; t += step) {
            int by;
            const int bx = run_tile<kMode>(p, t, &by);
            const TileOrigin org = tile_origin<kMode>(p, bx);
            int orow[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) orow[i] = output_row<kMode>(p, org, bx, q * 32 + i * 8 + sub);
            if (!mbar_wait_warp(smem_u32(&ctl->acc_full[buf]), bph, abort_flag, p.status)) break;
            tc_fence_after();
            const uint32_t acc = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + buf * BN;
#pragma unroll 1
            for (int c = 0; c < BN / 32; ++c) {
                uint32_t v[32];
                tmem_ld32(acc + c * 32, v);
                tmem_ld_wait();
                if (c + 1 == BN / 32) {               // read: hand the accumulator back before storing
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&ctl->acc_empty[buf]));
                }
#pragma unroll
                for (int g = 0; g < 4; ++g)
                    st_shared_v4(own + ((static_cast<uint32_t>(g) ^ sw) << 4),
                                 make_uint4(pack_bf16x2(__uint_as_float(v[8 * g]), __uint_as_float(v[8 * g + 1])),
                                            pack_bf16x2(__uint_as_float(v[8 * g + 2]), __uint_as_float(v[8 * g + 3])),
                                            pack_bf16x2(__uint_as_float(v[8 * g + 4]), __uint_as_float(v[8 * g + 5])),
                                            pack_bf16x2(__uint_as_float(v[8 * g + 6]), __uint_as_float(v[8 * g + 7]))));
                __syncwarp();
                const int col = by * BN + c * 32 + piece * 8;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint32_t rr = static_cast<uint32_t>(i * 8 + sub);
                    const uint4 w = ld_shared_v4(panel + rr * 64u + ((static_cast<uint32_t>(piece) ^ ((rr >> 1) & 3u)) << 4));
                    if (orow[i] >= 0 && col < p.N) *reinterpret_cast<uint4*>(C + static_cast<size_t>(orow[i]) * p.ldc + col) = w;   // N, ldc: multiples of 8
                }
                __syncwarp();
            }
            buf ^= 1u;
            if (buf == 0) bph ^= 1u;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_base, 2 * BN);
}

template <int BN, bool kRuns, bool kAny>
__global__ void __launch_bounds__(kGemmThreads, 2)
tc_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const GemmParams p) {
    if constexpr (kRuns) {
        run_tiles<BN, 0>(tmA, tmB, p, blockIdx.x, gridDim.x);
    } else {
        const int sl = p.splits < 1 ? 1 : p.splits;
        gemm_tile<BN, 0, kAny>(tmA, tmB, p, blockIdx.x, blockIdx.y, static_cast<int>(blockIdx.z) % sl, static_cast<int>(blockIdx.z) / sl);
    }
}

// Up to three independent products in one launch (dU = x^T G, dV = dY^T T and, where it is a plain
// product, dX of one layer): CTAs [0, end0) work on product 0, [end0, end1) on product 1, the rest on
// product 2; each decodes (row tile, column tile, slice) from its linear index.  One launch pays the
// start-up latency once and packs the short CTAs of one product beside the long ones of another.
// Tiles may be 64 or 128 columns wide per product.
template <bool kConv, bool kAny>
__device__ __forceinline__ void gemm_one(const CUtensorMap& tmA, const CUtensorMap& tmB, const GemmParams& p, int idx,
                                         const int2 t) {
    if constexpr (kConv) {
        if (p.conv_mode == 1) {             // t.x = the blocks that share the tiles
            if (p.bn == 64) run_tiles<64, 1>(tmA, tmB, p, idx, t.x);
            else run_tiles<128, 1>(tmA, tmB, p, idx, t.x);
            return;
        }
    }
    const int sl = p.splits < 1 ? 1 : p.splits;
    const int bx = idx % t.x, by = (idx / t.x) % t.y, zz = idx / (t.x * t.y);
    if constexpr (kConv) {
        if (p.conv_mode == 2) {
            if (p.bn == 64) gemm_tile<64, 2, kAny>(tmA, tmB, p, bx, by, zz, 0);
            else gemm_tile<128, 2, kAny>(tmA, tmB, p, bx, by, zz, 0);
            return;
        }
    }
    if (p.bn == 64) gemm_tile<64, 0, kAny>(tmA, tmB, p, bx, by, zz % sl, zz / sl);
    else gemm_tile<128, 0, kAny>(tmA, tmB, p, bx, by, zz % sl, zz / sl);
}
template <bool kConv, bool kAny>
__global__ void __launch_bounds__(kGemmThreads, 2)
tc_gemm3_kernel(const __grid_constant__ CUtensorMap tmA0, const __grid_constant__ CUtensorMap tmB0,
                const __grid_constant__ CUtensorMap tmA1, const __grid_constant__ CUtensorMap tmB1,
                const __grid_constant__ CUtensorMap tmA2, const __grid_constant__ CUtensorMap tmB2,
                const GemmParams p0, const GemmParams p1, const GemmParams p2, const int end0, const int end1,
                const int2 tiles0, const int2 tiles1, const int2 tiles2) {
    const int idx = blockIdx.x;
    if (idx < end0) gemm_one<kConv, kAny>(tmA0, tmB0, p0, idx, tiles0);
    else if (idx < end1) gemm_one<kConv, kAny>(tmA1, tmB1, p1, idx - end0, tiles1);
    else gemm_one<kConv, kAny>(tmA2, tmB2, p2, idx - end1, tiles2);
}

}  // namespace
}  // namespace tc
}  // namespace pf
#endif
