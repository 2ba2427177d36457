// 3 x 3, stride-1 convolutions whose image windows stay in shared memory: the images as one flat sequence of positions (see
// pf_tc_conv_res.cu), and what its kernels share.
#ifndef PF_TC_CONV_FLAT_CUH_
#define PF_TC_CONV_FLAT_CUH_

#include <cuda.h>

#include <algorithm>

#include "pf_tc.h"
#include "pf_tc_host.h"
#include "pf_tc_prims.cuh"

namespace pf {
namespace tc {
namespace {

// The flat view of the images.
struct FlatImage {
    int N, H, W, Wp, Hp;     // Wp = W + 1, Hp = H + 1
    int unit_rows;           // positions of one box: Wp (an image row) or Hp * Wp (an image)
    int per_image;           // boxes are whole images
};
__device__ __forceinline__ int floor_div(int a, int b) { return a >= 0 ? a / b : -((b - 1 - a) / b); }
// Pixel index of position q, -1 for the zero column and row (and behind the last image).
__device__ __forceinline__ int pixel_of(const FlatImage& f, int q) {
    const int R = q / f.Wp, w = q - R * f.Wp, n = R / f.Hp, h = R - n * f.Hp;
    return (w < f.W && h < f.H && n < f.N) ? (n * f.H + h) * f.W + w : -1;
}
// Loads boxes u0 .. u0 + count - 1 of 64 channels from channel c0 on, one after the other, to dst.
__device__ __forceinline__ void load_window(const FlatImage& f, const CUtensorMap* map, uint32_t dst, uint32_t bar, int u0, int count, int c0) {
    const uint32_t bytes = static_cast<uint32_t>(f.unit_rows) * 128u;
    if (f.per_image) {
        for (int u = 0; u < count; ++u) tma_load_4d(dst + u * bytes, map, bar, c0, 0, 0, u0 + u);
    } else {
        int n = floor_div(u0, f.Hp), h = u0 - n * f.Hp;
        for (int u = 0; u < count; ++u) {
            tma_load_4d(dst + u * bytes, map, bar, c0, 0, h, n);
            if (++h == f.Hp) { h = 0; ++n; }
        }
    }
}

// 32 rows x 128 columns of one accumulator: rounded to bf16 and stored as whole 16-byte pieces, four rows per
// instruction; pix is this lane's row (pixel, or -1).
__device__ __forceinline__ void store_block(uint32_t acc, uint32_t panel, int lane, int pix, __nv_bfloat16* out, int ld, int col0, int ncols,
                                            uint64_t* empty_bar) {
    const uint32_t own = panel + static_cast<uint32_t>(lane) * 128u, sw = static_cast<uint32_t>(lane & 7);
    const int sub = lane >> 3, piece = lane & 7;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        uint32_t v0[32], v1[32];
        tmem_ld32(acc + c * 64, v0);
        tmem_ld32(acc + c * 64 + 32, v1);
        tmem_ld_wait();
        if (c == 1) {                     // the accumulator has been read: hand it back before converting
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(empty_bar));
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const uint32_t* v = t < 4 ? v0 + 8 * t : v1 + 8 * (t - 4);
            st_shared_v4(own + ((static_cast<uint32_t>(t) ^ sw) << 4),
                         make_uint4(pack_bf16x2(__uint_as_float(v[0]), __uint_as_float(v[1])), pack_bf16x2(__uint_as_float(v[2]), __uint_as_float(v[3])),
                                    pack_bf16x2(__uint_as_float(v[4]), __uint_as_float(v[5])), pack_bf16x2(__uint_as_float(v[6]), __uint_as_float(v[7]))));
        }
        __syncwarp();
        const int col = col0 + c * 64 + piece * 8;
        if (col0 + c * 64 < ncols) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int rr = i * 4 + sub;
                const int px = __shfl_sync(0xffffffffu, pix, rr);
                const uint4 w = ld_shared_v4(panel + static_cast<uint32_t>(rr) * 128u + ((static_cast<uint32_t>(piece) ^ static_cast<uint32_t>(rr & 7)) << 4));
                if (px >= 0 && col < ncols) *reinterpret_cast<uint4*>(out + static_cast<size_t>(px) * ld + col) = w;
            }
        }
        __syncwarp();
    }
}

// Parameters of the backward's kernels (pf_tc_conv_bwd.cu).
struct DtDvParams {
    int rows, R;
    int tiles;                   // of 128 rows
    int panels, pairs;           // of 64 and 128 columns of dY
    int num_stages;
    __nv_bfloat16* dT;
    int ldt;                     // elements of a row of dT
    int early;                   // the launch before writes none of the operands
    float* partial;              // slices of dV: [tile][block][quadrant][4-column group][row][4]
    unsigned int* status;
};
struct SumPart {
    const float* partial;
    void* out;                   // fp32 or bf16, added to what it holds or not; plain: neither, on a 16-byte boundary
    int f32, accumulate, plain;
    int tiles, per_tap, rows, R;             // tiles of 128 rows; per_tap > 0: tile = tap * per_tap + block of 128 of `rows` rows per tap
    int split[2], tail;                      // slices of the tiles before `tail`, and from there on
};
struct DuParams {
    int C, tb;                   // blocks of 128 channels
    int split[2];                // slices of tap rows 0 and 1, and of tap row 2
    int blocks, per[2];          // blocks of positions, and of a slice
    int bh, nb, tpi, kpix_x, kpix_t, ksteps, steps_row;      // kpix: positions of a block in x's and dT's tiles
    float* partial;              // [tile][slice]..., tile = tap * tb + block of channels
    SumPart sum;                 // dV
    unsigned int* status;
};
struct DxParams {
    FlatImage f;
    int tiles, step, C, nblk, ksteps;
    __nv_bfloat16* out;
    const __nv_bfloat16 *x, *dT;     // (for sums of dU that are NaN)
    int ldt;
    uint32_t a_bytes, a_off, stg_off, ring_off;
    int num_stages;
    SumPart sum;                 // dU
    unsigned int* status;
};

// ------------------------------------------------------------------------------ host
inline FlatImage flat_image(int N, int H, int W) {
    FlatImage f;
    f.N = N; f.H = H; f.W = W; f.Wp = W + 1; f.Hp = H + 1;
    f.per_image = f.Wp * f.Hp <= 64;                 // boxes of a few KB at least: a TMA instruction costs 40 ns
    f.unit_rows = f.per_image ? f.Wp * f.Hp : f.Wp;
    return f;
}
// Positions of a window that covers `span` consecutive positions wherever they start.
inline int window_rows(const FlatImage& f, int span) { return ((span + f.unit_rows - 2) / f.unit_rows + 1) * f.unit_rows; }
inline bool window_map(CUtensorMap* map, const FlatImage& f, const void* p, int channels, int64_t ld = 0) {
    return cached_map_nhwc(map, p, f.N, f.H, f.W, channels, f.Wp, f.per_image ? f.Hp : 1, 1, 1, ld);
}
// A persistent grid of equally loaded CTAs.
inline int even_grid(int tiles) { return static_cast<int>(ceil_div(tiles, ceil_div(tiles, num_sms()))); }

}  // namespace
}  // namespace tc
}  // namespace pf
#endif
