// fp32 products on the tensor cores (sm_100a): every fp32 operand value is split exactly into three bf16 values
//   2^16 x = x1 + x2 + x3,  x1 = bf16(2^16 x), x2 = bf16(2^16 x - x1), x3 = 2^16 x - x1 - x2
// (8 + 8 + 8 significand bits), and a product a b is the sum of the six partial products that reach fp32
// precision: a1 b1 | a1 b2 + a2 b1 + a2 b2 + a1 b3 + a3 b1 (the three left out are below 2^-24 of it).
//
// Range.  The last bit of an fp32 number is 2^-149 or more, that of a bf16 number 2^-133 or more: with the factor 2^16 the
// split is exact down to the last subnormal (without it operands below 2^-110 lose digits).  The sums leave
// the chip with 2^-32.  At the other end, operands from 2^112 on, infinities and NaN have a part that is
// not finite, and sums from 2^96 on overflow: where a CTA finds such a sum it computes its outputs once more with
// fp32 FMAs (f32_repair), which give what such operands give in fp32.
//
// Accumulation.  A tcgen05.mma truncates when it adds to its fp32 accumulator (measured: -0.5 ulp per MMA on
// sums of one sign), so long sums must not stay in tensor memory: the main products a1 b1 accumulate over 64
// elements of the contraction in one of two accumulators, which the worker warps then add, with
// round-to-nearest, to fp32 sums in their registers.  The five correction products, at most 2^-7 of the sum, have an
// accumulator of their own for 2048 elements: then a chunk's main products go on top of it, so that it is drained as
// that chunk's accumulator, and the buffer they would have used takes the corrections from there on.  640 truncated
// additions lose at most 640 ulps of that 2^-7th, 6e-7 of the sum, whatever its length; left to pile up over 32768
// elements of one sign they lost 6.9e-6.  (Not more often: the chunk on top of the corrections is truncated once
// more, 1 % of the error of random sums at every 512 elements.)  The result is as accurate as an fp32 FMA kernel.
//
// One CTA computes a 128 x BN tile of C = A * B or one slice of its contraction.  Warps: 0 = TMA producer of
// A, 1 = tensor memory + MMA issue, 2..17 = workers (split the operands, drain the accumulators, epilogue),
// 18 = TMA producer of B.  A k-block is 32 elements: the fp32 tiles (128-byte-swizzled boxes of 32 floats)
// arrive in a ring and the workers split them into one of two half buffers of planes, which 12 MMAs read.  The
// workers are two groups of eight warps that take alternate k-blocks (and half buffers): one k-block is a chain
// of waits and shared-memory round trips of about 1 us for a warp whatever it computes.
// Splitting on chip rather than in a pass of its own: no workspace, no extra launch, 32 KB of loads per
// k-block instead of 48 KB.
// An MMA that takes both operands from shared memory reads 128 bytes per clock, all there is, while TMA writes and the
// workers read and write the tiles.  So the planes of A go to TENSOR memory (a thread splits 16 contraction elements of its row, whatever the operand's
// orientation) and only B's planes, shared by all rows, to shared memory: 136 KB instead of 208 KB through
// shared memory per k-block of a 128 x 128 tile.  A k-block takes 0.95 us with all SMs at work (0.67 us of a 128 x 64
// tile), of which the MMAs are 0.4; a contraction of 4096 against one of 2048, caches warm.  What bounds it is that
// chain of waits: on 18944 x 4096 -> 128 the tensor pipe is busy 40 % of the time, the shared-memory data pipe 54 %
// (21 MMAs, 33 workers), the issue slots 58 %; in a step of 2048 x 512 -> 128 -> 2048 all of them less.
#ifndef PF_TC_F32_KERNEL_CUH_
#define PF_TC_F32_KERNEL_CUH_

#include <cuda.h>

#include "pf_tc_prims.cuh"

namespace pf {
namespace tc {

struct F32Params {
    int M, N;
    int a_mn, b_mn;          // 1 = operand stored with the M/N index contiguous
    int bn;                  // columns of a tile: 64 or 128
    int nkb, kb_per_split, splits;     // 32-element k-blocks
    int num_stages;
    int mode;                // 0 = plain, 1 / 2 / 3 = the convolution products below
    int tiles_x, tiles_y;
    const float *A, *B;      // the operands, as f32_repair reads them (the tiles come through the tensor maps)
    long long lda, ldb;
    int K, cv_H, cv_W, cv_R;         // cv_H x cv_W: the image that A is
    float* C;
    long long ldc;
    float* C2;               // optional second copy at another pitch
    long long ldc2;
    const float* bias;       // optional epilogue of an unsplit product: C = act(A B + bias)
    int act;
    float* partial;          // splits > 1: slices, [tile][slice][column quarter][32-row quadrant][4-column group][row][4]
    unsigned int* counters;
    unsigned int* status;
    // Convolution (kMode 1 = dX, 2 = dU, 3 = the thin convolution forward); names as in pf_tc_gemm_kernel.cuh, with 32-channel
    // blocks.  Tiles of modes 1 and 3 are blocks of pixels of an image of out_h x out_w output pixels, `step` pixels apart.
    int cv_blks, cv_kw, cv_kh, cv_pad, cv_stride, cv_C, cv_bh, cv_nb, cv_tpi, cv_N, cv_bw, cv_inv_bw, cv_inv_bh, cv_tiles_class;
    int out_h, out_w, step;
    int cv_blocks;           // dU: 32-channel blocks of the unrolled factor
    int cv_wblk;             // dU: blocks of cv_bw pixels per image row
    int rows_tile, kpix;
    int ragged;              // mode 3: C is not a multiple of 32, tmB is [taps][C][R]
    int early;               // kEarlyA | kEarlyB
};

struct F32Launch {
    CUtensorMap ta[3], tb[3];
    F32Params p[3];
    int end[3];              // running total of blocks
};
// Launch of the instantiation with the convolution's modes (pf_tc_f32_conv.cu).
cudaError_t launch_f32_conv(int blocks, size_t smem, cudaStream_t stream, const F32Launch& a);

namespace {

constexpr int kF32Threads = 608;
constexpr int kF32MaxStages = 8;
constexpr int kChunk = 2;                    // k-blocks per main accumulator: 64 elements of the contraction
static_assert(kChunk == 2, "one k-block per worker group and chunk");
constexpr int kCorrChunks = 32;              // chunks per correction accumulator
static_assert(kCorrChunks % 2 == 0, "it changes places with the accumulator of the odd chunks");
constexpr uint32_t kF32TileA = 16384;        // 128 x 32 floats
constexpr uint32_t kColsA = 16;              // tensor-memory columns of one plane of A's k-block (32 bf16 per row)

struct F32Ctl {
    uint64_t full[kF32MaxStages];
    uint64_t empty[kF32MaxStages];
    uint64_t split_full[2];      // a half buffer of planes is complete (8 worker warps)
    uint64_t split_empty[2];     // the MMAs have read it
    uint64_t main_full[2];       // a main accumulator holds its chunk
    uint64_t main_empty[2];      // the workers have drained it (16 warps)
    uint64_t corr_full;
    uint32_t tmem_base;
    uint32_t abort;
    uint32_t fix_ok;
    uint32_t repair;             // a sum is not finite
};

__device__ __forceinline__ uint32_t cvt_bf16x2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
constexpr float kScale = 65536.f, kUnscale = 1.f / (65536.f * 65536.f);
// The three bf16 planes of a pair of floats.
__device__ __forceinline__ void split_pair(float lo, float hi, uint32_t& p1, uint32_t& p2, uint32_t& p3) {
    asm("{\n .reg .b64 v, s;\n mov.b64 v, {%0, %1};\n mov.b64 s, {%2, %2};\n mul.rn.f32x2 v, v, s;\n mov.b64 {%0, %1}, v;\n}"
        : "+f"(lo), "+f"(hi) : "f"(kScale));
    p1 = cvt_bf16x2(lo, hi);
    lo -= __uint_as_float(p1 << 16);
    hi -= __uint_as_float(p1 & 0xffff0000u);
    p2 = cvt_bf16x2(lo, hi);
    lo -= __uint_as_float(p2 << 16);
    hi -= __uint_as_float(p2 & 0xffff0000u);
    p3 = __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632);      // what is left has at most 8 bits: no rounding
}
__device__ __forceinline__ void st_shared_v2(uint32_t addr, uint32_t a, uint32_t b) {
    asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}

// A: the thread owns row q * 32 + lane of the tile and 16 of the k-block's elements (half kh), whose planes it writes to
// tensor memory.  K-major tile: four 16-byte chunks of the row; MN-major: box q holds the rows' 32 columns, one
// word per contraction row (both free of bank conflicts).
__device__ __forceinline__ void split_a(uint32_t src, uint32_t taddr, bool mn, int q, int kh, int lane) {
    float x[16];
    if (mn) {
        const uint32_t box = src + static_cast<uint32_t>(q) * 4096u + static_cast<uint32_t>(kh) * 2048u + static_cast<uint32_t>(lane & 3) * 4u;
#pragma unroll
        for (int k = 0; k < 16; ++k)
            x[k] = __uint_as_float(ld_shared_u32(box + static_cast<uint32_t>(k) * 128u + (static_cast<uint32_t>((lane >> 2) ^ (k & 7)) << 4)));
    } else {
        const uint32_t row = src + static_cast<uint32_t>(q * 32 + lane) * 128u;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const uint4 v = ld_shared_v4(row + (static_cast<uint32_t>((kh * 4 + c) ^ (lane & 7)) << 4));
            x[4 * c] = __uint_as_float(v.x); x[4 * c + 1] = __uint_as_float(v.y);
            x[4 * c + 2] = __uint_as_float(v.z); x[4 * c + 3] = __uint_as_float(v.w);
        }
    }
    uint32_t p1[8], p2[8], p3[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) split_pair(x[2 * c], x[2 * c + 1], p1[c], p2[c], p3[c]);
    tmem_st8(taddr, p1);
    tmem_st8(taddr + kColsA, p2);
    tmem_st8(taddr + 2 * kColsA, p3);
}

// B: each warp splits kRows / 8 rows of 32 floats (row = 128 bytes, 16-byte chunks XOR-swizzled by the row, as TMA
// wrote them) into the planes.  K-major: row r is row r of a plane, its 64 bytes go to half h of the 128-byte
// row.  MN-major: the rows are [box of 32 columns][contraction row], a panel of 64 columns is two boxes and
// the contraction row lies in half h of the panel.  Eight lanes read one row's eight chunks (no conflicts);
// the rows of a half warp differ by 4, so that their 64-byte runs fall into different banks.  All loads
// come before the first store (asm statements keep their order).
template <int kRows>
__device__ __forceinline__ void split_b(uint32_t src, uint32_t dst, uint32_t plane, bool mn, uint32_t h, int w, int lane) {
    const int q = lane >> 3, j = lane & 7;
    uint4 v[kRows / 32];
    auto row_of = [&](int it) { return w * (kRows / 8) + (it >> 1) * 8 + (it & 1) * 2 + (q & 1) * 4 + (q >> 1); };
#pragma unroll
    for (int it = 0; it < kRows / 32; ++it) {
        const int r = row_of(it);
        v[it] = ld_shared_v4(src + static_cast<uint32_t>(r) * 128u + (static_cast<uint32_t>(j ^ (r & 7)) << 4));
    }
#pragma unroll
    for (int it = 0; it < kRows / 32; ++it) {
        const int r = row_of(it);
        const uint32_t hi = mn ? static_cast<uint32_t>(r >> 5) & 1u : h;
        const uint32_t row = mn ? (static_cast<uint32_t>(r >> 6) << 6) + 32u * h + static_cast<uint32_t>(r & 31) : static_cast<uint32_t>(r);
        const uint32_t at = dst + row * 128u + ((((hi << 2) + static_cast<uint32_t>(j >> 1)) ^ static_cast<uint32_t>(r & 7)) << 4) +
                            static_cast<uint32_t>(j & 1) * 8u;
        uint32_t a1, a2, a3, b1, b2, b3;
        split_pair(__uint_as_float(v[it].x), __uint_as_float(v[it].y), a1, a2, a3);
        split_pair(__uint_as_float(v[it].z), __uint_as_float(v[it].w), b1, b2, b3);
        st_shared_v2(at, a1, b1);
        st_shared_v2(at + plane, a2, b2);
        st_shared_v2(at + 2 * plane, a3, b3);
    }
}

struct F32Origin {
    int img, row, ph, pw, na, nb, a0, b0;
};
template <int kMode>
__device__ __forceinline__ F32Origin f32_origin(const F32Params& p, int bx) {
    F32Origin o = {};
    if constexpr (kMode == 1 || kMode == 3) {
        int t = bx;
        o.na = p.cv_kh;
        o.nb = p.cv_kw;
        if (kMode == 1 && p.cv_stride > 1) {
            const int s = p.cv_stride, cls = bx / p.cv_tiles_class;
            t = bx - cls * p.cv_tiles_class;
            o.ph = cls / s;
            o.pw = cls - o.ph * s;
            o.a0 = (o.ph + p.cv_pad) % s;
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
__device__ __forceinline__ int f32_row(const F32Params& p, const F32Origin& o, int bx, int r) {
    if constexpr (kMode == 0) {
        const int row = bx * 128 + r;
        return row < p.M ? row : -1;
    } else if constexpr (kMode == 2) {
        const int blk = bx * 4 + (r >> 5), tap = blk / p.cv_blks, c = (blk - tap * p.cv_blks) * 32 + (r & 31);
        return (blk < p.cv_blocks && c < p.cv_C) ? tap * p.cv_C + c : -1;
    } else {
        const int line = (r * p.cv_inv_bw) >> 16, w = (r - line * p.cv_bw) * p.step + o.pw;
        const int i = (line * p.cv_inv_bh) >> 16, img = o.img + i, h = (o.row + line - i * p.cv_bh) * p.step + o.ph;
        return (r < p.rows_tile && img < p.cv_N && h < p.out_h && w < p.out_w) ? (img * p.out_h + h) * p.out_w + w : -1;
    }
}

// Adds `len` products a[i sa] * b[i sb + c sc] to acc[c], c < n, 64 at a time.
__device__ __forceinline__ void repair_run(const float* a, long long sa, const float* b, long long sb, long long sc, int len, int n, float (&acc)[4]) {
#pragma unroll 1
    for (int i0 = 0; i0 < len; i0 += 64) {
        float part[4] = {0.f, 0.f, 0.f, 0.f};
        const int end = min(len, i0 + 64);
#pragma unroll 4
        for (int i = i0; i < end; ++i) {
            const float v = __ldcg(a + i * sa);
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (c < n) part[c] = fmaf(v, __ldcg(b + i * sb + c * sc), part[c]);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[c] += part[c];
    }
}
// The outputs of this CTA (its share of the tile's units of 8 rows x 16 columns) from the operands in global memory,
// by the definition of the product.  Rare and therefore plain: a lane sums one row's four columns.  The test for it
// and the factor cost 0-2 % (training step of 2048 rows, 512 -> 128 -> 2048, cold L2: 73.2 -> 74.1 us; 32 x 28 x 28, 128 ->
// 32 -> 256, stride 2: 86.0 -> 88.1, stride 1 176.1 before and after); with a NaN in every row that linear step takes 1.8 ms.
// (A second pass over the ring by the same roles was slower where nothing is repaired: 83 us.)
template <int BN, int kMode>
__device__ __noinline__ void f32_repair(const F32Params& p, int bx, int by, int bz) {
    constexpr int kUnits = 16 * (BN / 16);
    const F32Origin org = f32_origin<kMode>(p, bx);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, per = (kUnits + p.splits - 1) / p.splits, end = min(kUnits, (bz + 1) * per);
    const int s = p.cv_stride;
    const long long C = p.cv_C, R = p.cv_R;
#pragma unroll 1
    for (int u = bz * per + warp; u < end; u += kF32Threads / 32) {
        const int oct = u / (BN / 16), row = f32_row<kMode>(p, org, bx, oct * 8 + (lane & 7));
        const int col = by * BN + (u - oct * (BN / 16)) * 16 + (lane >> 3) * 4, n = min(4, p.N - col);
        if (row < 0 || n <= 0) continue;
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        if constexpr (kMode == 0) {
            repair_run(p.A + (p.a_mn ? row : row * p.lda), p.a_mn ? p.lda : 1, p.B + (p.b_mn ? col : col * p.ldb), p.b_mn ? p.ldb : 1,
                       p.b_mn ? 1 : p.ldb, p.K, n, acc);
        } else if constexpr (kMode == 2) {          // rows (tap, channel), contraction over the output pixels
            const int tap = row / p.cv_C, ta = tap / p.cv_kw, dx = tap - ta * p.cv_kw - p.cv_pad, dy = ta - p.cv_pad;
            const int w0 = dx >= 0 ? 0 : (s - 1 - dx) / s, w1 = min(p.out_w, (p.cv_W - 1 - dx + s) / s);
#pragma unroll 1
            for (int i = 0; i < p.cv_N * p.out_h; ++i) {
                const int img = i / p.out_h, h = (i - img * p.out_h) * s + dy;
                if (h < 0 || h >= p.cv_H || w0 >= w1) continue;
                repair_run(p.A + ((static_cast<long long>(img) * p.cv_H + h) * p.cv_W + w0 * s + dx) * C + (row - tap * p.cv_C), s * C,
                           p.B + (static_cast<long long>(i) * p.out_w + w0) * R + col, R, 1, w1 - w0, n, acc);
            }
        } else {                                    // rows are pixels, contraction over (tap, channel or rank)
            const int w = row % p.out_w, t = row / p.out_w, img = t / p.out_h, h = t - img * p.out_h;
#pragma unroll 1
            for (int tap = 0; tap < p.cv_kh * p.cv_kw; ++tap) {
                const int ta = tap / p.cv_kw, tb = tap - ta * p.cv_kw;
                int y = h * s - p.cv_pad + ta, x = w * s - p.cv_pad + tb;
                if constexpr (kMode == 1) {         // A = dT: the output pixel that this tap takes from the input pixel
                    y = h + p.cv_pad - ta; x = w + p.cv_pad - tb;
                    if (y < 0 || x < 0 || y % s != 0 || x % s != 0) continue;
                    y /= s; x /= s;
                }
                if (y < 0 || x < 0 || y >= p.cv_H || x >= p.cv_W) continue;
                const long long pix = (static_cast<long long>(img) * p.cv_H + y) * p.cv_W + x;
                if constexpr (kMode == 1) repair_run(p.A + pix * R, 1, p.B + (tap * C + col) * R, 1, R, p.cv_R, n, acc);
                else repair_run(p.A + pix * C, 1, p.B + tap * C * R + col, R, 1, p.cv_C, n, acc);
            }
        }
        for (int c = 0; c < n; ++c) {
            float v = acc[c] + (p.bias ? p.bias[col + c] : 0.f);
            if (p.act == 1) v = fmaxf(v, 0.f);
            p.C[static_cast<size_t>(row) * p.ldc + col + c] = v;
            if (p.C2) p.C2[static_cast<size_t>(row) * p.ldc2 + col + c] = v;
        }
    }
}

template <int BN, int kMode>
__device__ __forceinline__ void f32_tile(const CUtensorMap& tmA, const CUtensorMap& tmB, const F32Params& p, const int bx, const int by,
                                         const int bz) {
    constexpr uint32_t kTileB = BN * 128;                 // BN x 32 floats
    constexpr uint32_t kStage = kF32TileA + kTileB;
    constexpr uint32_t kPlaneB = BN * 128;                // BN x 64 bf16
    constexpr int kCols = BN / 4;                         // columns of a worker warp
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t* smem = smem_raw + (((raw + 1023u) & ~1023u) - raw);
    F32Ctl* ctl = reinterpret_cast<F32Ctl*>(smem);
    const uint32_t planes_b = smem_u32(smem + 1024);      // three planes of B (A's are in tensor memory)
    constexpr uint32_t kTmemA = 3 * BN;                   // after two main accumulators and the correction's: two half buffers
    const uint32_t ring = planes_b + 3 * kPlaneB;
    volatile uint32_t *abort_flag = &ctl->abort, *repair = &ctl->repair;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n0 = by * BN;
    const F32Origin org = f32_origin<kMode>(p, bx);
    const int nkb_total = kMode == 1 ? org.na * org.nb * p.cv_blks : p.nkb;
    const int kb_beg = bz * p.kb_per_split;
    const int nkb = min(nkb_total, kb_beg + p.kb_per_split) - kb_beg;
    const uint32_t NS = static_cast<uint32_t>(p.num_stages);
    const int tile = by * p.tiles_x + bx;

    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&ctl->full[s]), 2);
            mbar_init(smem_u32(&ctl->empty[s]), 8);
        }
        for (int h = 0; h < 2; ++h) {
            mbar_init(smem_u32(&ctl->split_full[h]), 8);
            mbar_init(smem_u32(&ctl->split_empty[h]), 1);
            mbar_init(smem_u32(&ctl->main_full[h]), 1);
            mbar_init(smem_u32(&ctl->main_empty[h]), 16);
        }
        mbar_init(smem_u32(&ctl->corr_full), 1);
        ctl->abort = 0;
        ctl->fix_ok = 0;
        ctl->repair = 0;
        fence_barrier_init();
        fence_proxy_async_smem();
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
    }
    if (kMode == 2 && p.kpix < 32) {
        // contraction rows that TMA never writes must read as zero in every 32-row box of every stage
        const int pieces = (32 - p.kpix) * 8, boxes = static_cast<int>(kStage / 4096) * static_cast<int>(NS);
        for (int i = threadIdx.x; i < boxes * pieces; i += blockDim.x) {
            const int box = i / pieces;
            st_shared_v4(ring + box * 4096 + p.kpix * 128 + (i - box * pieces) * 16, make_uint4(0, 0, 0, 0));
        }
        fence_proxy_async_smem();
    }
    if (warp == 1) tmem_alloc(smem_u32(&ctl->tmem_base), 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const bool ahead = (warp == 0 && (p.early & kEarlyA)) || (warp == 18 && (p.early & kEarlyB));
    if (!ahead) {               // everything above overlapped the previous kernel's tail, as do the loads of an early operand
        pdl_wait();
        pdl_launch_dependents();
    }
    const uint32_t tmem = ctl->tmem_base;
    const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);

    if (warp == 0 || warp == 18) {
        if (elect_one()) {
            const bool do_a = warp == 0;
            const uint32_t base = ring + (do_a ? 0u : kF32TileA);
            uint32_t bytes = do_a ? kF32TileA : kTileB;
            int boxes = 4;                                 // dU: 32-channel blocks of A that exist
            if constexpr (kMode == 2) {
                boxes = min(4, p.cv_blocks - bx * 4);
                bytes = static_cast<uint32_t>(p.kpix) * 128u * static_cast<uint32_t>(do_a ? boxes : BN / 32);
            } else if constexpr (kMode != 0) {
                if (do_a) bytes = static_cast<uint32_t>(p.rows_tile) * 128u;
            }
            auto produce = [&](auto&& issue) {
                uint32_t s = 0, ph = 1, dst = base;
                for (int i = 0; i < nkb; ++i) {
                    if (!mbar_wait(empty0 + 8 * s, ph, abort_flag, p.status)) break;
                    const uint32_t full = full0 + 8 * s;
                    mbar_expect_tx(full, bytes);
                    issue(dst, full);
                    dst += kStage;
                    if (++s == NS) { s = 0; dst = base; ph ^= 1u; }
                }
            };
            int k0 = kb_beg * 32;
            if constexpr (kMode == 0) {
                const int mn0 = do_a ? bx * 128 : n0, width = do_a ? 4 : BN / 32;
                const CUtensorMap* map = do_a ? &tmA : &tmB;
                if (do_a ? p.a_mn : p.b_mn) {
                    produce([&](uint32_t dst, uint32_t full) {
                        for (int b = 0; b < width; ++b) tma_load_2d(dst + b * 4096, map, full, mn0 + b * 32, k0);
                        k0 += 32;
                    });
                } else {
                    produce([&](uint32_t dst, uint32_t full) { tma_load_2d(dst, map, full, k0, mn0); k0 += 32; });
                }
            } else if constexpr (kMode == 2) {
                const int bh = p.cv_bh, bw = p.cv_bw, nwb = p.cv_wblk, tpi = p.cv_tpi;
                int wb = kb_beg % nwb, t = kb_beg / nwb, img = t / tpi;
                t -= img * tpi;
                img *= p.cv_nb;
                auto advance = [&] {
                    if (++wb == nwb) { wb = 0; if (++t == tpi) { t = 0; img += p.cv_nb; } }
                };
                if (do_a) {
                    int c[4], x[4], y[4];
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        const int blk = bx * 4 + b, tap = blk / p.cv_blks, ta = tap / p.cv_kw;
                        c[b] = (blk - tap * p.cv_blks) * 32;
                        x[b] = tap - ta * p.cv_kw - p.cv_pad;
                        y[b] = ta - p.cv_pad;
                    }
                    const int s = p.cv_stride;
                    produce([&](uint32_t dst, uint32_t full) {
                        const int x0 = wb * bw * s, y0 = t * bh * s;
#pragma unroll
                        for (int b = 0; b < 4; ++b)
                            if (b < boxes) tma_load_4d(dst + b * 4096, &tmA, full, c[b], x0 + x[b], y0 + y[b], img);
                        advance();
                    });
                } else {
                    produce([&](uint32_t dst, uint32_t full) {
#pragma unroll
                        for (int b = 0; b < BN / 32; ++b) tma_load_4d(dst + b * 4096, &tmB, full, n0 + 32 * b, wb * bw, t * bh, img);
                        advance();
                    });
                }
            } else {
                const int blks = p.cv_blks, ntb = org.nb;
                int cb = kb_beg % blks, tb = kb_beg / blks, ta = tb / ntb;
                tb -= ta * ntb;
                auto advance = [&] {
                    if (++cb == blks) { cb = 0; if (++tb == ntb) { tb = 0; ++ta; } }
                };
                if (do_a) {
                    const int s = p.cv_stride, sign = kMode == 1 ? -1 : 1;
                    const int y0 = kMode == 1 ? org.row + (org.ph + p.cv_pad - org.a0) / s : org.row * s - p.cv_pad;
                    const int x0 = kMode == 1 ? (org.pw + p.cv_pad - org.b0) / s : -p.cv_pad;
                    produce([&](uint32_t dst, uint32_t full) {
                        tma_load_4d(dst, &tmA, full, cb * 32, x0 + sign * tb, y0 + sign * ta, org.img);
                        advance();
                    });
                } else if constexpr (kMode == 1) {
                    const int s = p.cv_stride;
                    produce([&](uint32_t dst, uint32_t full) {
                        tma_load_2d(dst, &tmB, full, cb * 32, ((org.a0 + ta * s) * p.cv_kw + org.b0 + tb * s) * p.cv_C + n0);
                        advance();
                    });
                } else if (p.ragged) {
                    produce([&](uint32_t dst, uint32_t full) {
                        for (int b = 0; b < BN / 32; ++b) tma_load_3d(dst + b * 4096, &tmB, full, n0 + 32 * b, cb * 32, ta * ntb + tb);
                        advance();
                    });
                } else {
                    produce([&](uint32_t dst, uint32_t full) {
                        for (int b = 0; b < BN / 32; ++b) tma_load_2d(dst + b * 4096, &tmB, full, n0 + 32 * b, k0);
                        k0 += 32;
                    });
                }
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            const uint32_t idesc = make_idesc_bf16(128, BN, 0, p.b_mn);
            const uint64_t b_desc0 = p.b_mn ? make_smem_desc(planes_b, 8192, 1024) : make_smem_desc(planes_b, 16, 1024);
            const uint32_t b_half = p.b_mn ? 256u : 4u;      // 16-byte units to half 1
            const uint32_t b_step = p.b_mn ? 128u : 2u;      // ... to the next 16 elements
            constexpr uint32_t pb = kPlaneB >> 4;
            bool ok = true;
            int in_chunk = 0;
            uint32_t odd = tmem + BN, corr = tmem + 2 * BN;      // accumulators of the odd chunks (the even ones': tmem) and of the corrections
            uint32_t main_acc = 0, corr_acc = 0;          // 0: the next product starts the accumulator
            uint32_t buf = 0, bufph = 1;                  // phase of main_empty[buf]: the first use of each finds it free
            for (int i = 0; i < nkb; ++i) {
                const uint32_t h = static_cast<uint32_t>(i) & 1u;
                if (in_chunk == 0) {
                    ok = mbar_wait(smem_u32(&ctl->main_empty[buf]), bufph, abort_flag, p.status);
                    if (!ok) break;
                    main_acc = 0;
                    if ((i / kChunk) % kCorrChunks == kCorrChunks - 1) {      // on top of the corrections so far
                        const uint32_t c = odd;
                        odd = corr;
                        corr = c;
                        main_acc = 1;
                        corr_acc = 0;
                    }
                }
                ok = mbar_wait(smem_u32(&ctl->split_full[h]), static_cast<uint32_t>(i >> 1) & 1u, abort_flag, p.status);
                if (!ok) break;
                tc_fence_after();
                const uint64_t b0 = b_desc0 + h * b_half;
                const uint32_t a0 = tmem + kTmemA + h * (3 * kColsA);
                const uint32_t d = buf ? odd : tmem;
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) {
                    const uint64_t b = b0 + ks * b_step;
                    const uint32_t a = a0 + ks * 8u;
                    tc_mma_bf16_ta(corr, a + 2 * kColsA, b, idesc, ks > 0 ? 1u : corr_acc);
                    tc_mma_bf16_ta(corr, a, b + 2 * pb, idesc, 1u);
                    tc_mma_bf16_ta(corr, a + kColsA, b + pb, idesc, 1u);
                    tc_mma_bf16_ta(corr, a + kColsA, b, idesc, 1u);
                    tc_mma_bf16_ta(corr, a, b + pb, idesc, 1u);
                    tc_mma_bf16_ta(d, a, b, idesc, ks > 0 ? 1u : main_acc);
                }
                main_acc = corr_acc = 1;
                tc_commit(smem_u32(&ctl->split_empty[h]));
                if (++in_chunk == kChunk || i + 1 == nkb) {
                    tc_commit(smem_u32(&ctl->main_full[buf]));
                    in_chunk = 0;
                    buf ^= 1u;
                    if (buf == 0) bufph ^= 1u;
                }
            }
            if (ok) tc_commit(smem_u32(&ctl->corr_full));
        }
    } else {
        const int w = (warp - 2) & 7, grp = (warp - 2) >> 3, q = warp & 3, kh = w >> 2, colq = grp * 2 + kh;
        const uint32_t rows_base = tmem + (static_cast<uint32_t>(q * 32) << 16);
        const uint32_t lane_base = rows_base + static_cast<uint32_t>(colq * kCols);
        const bool a_mn = p.a_mn, b_mn = p.b_mn;
        const uint32_t h = static_cast<uint32_t>(grp);
        const uint32_t a_dst = rows_base + kTmemA + h * (3 * kColsA) + static_cast<uint32_t>(kh * 8);
        const int chunks = (nkb + kChunk - 1) / kChunk;
        float acc[kCols];
#pragma unroll
        for (int c = 0; c < kCols; ++c) acc[c] = 0.f;
        auto add_from = [&](uint32_t taddr) {
            uint32_t v[kCols];
            if constexpr (kCols == 32) tmem_ld32(taddr, v);
            else tmem_ld16(taddr, v);
            tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < kCols; ++e) acc[e] += __uint_as_float(v[e]);
        };
        bool ok = true;
        uint32_t odd = BN;         // columns of the odd chunks' accumulator; the corrections have the other of BN and 2 BN
        auto drain = [&](int c) {
            const uint32_t b = static_cast<uint32_t>(c) & 1u;
            ok = mbar_wait_warp(smem_u32(&ctl->main_full[b]), static_cast<uint32_t>(c >> 1) & 1u, abort_flag, p.status);
            tc_fence_after();
            if (!ok) return;
            if (c % kCorrChunks == kCorrChunks - 1) odd = 3 * BN - odd;
            add_from(lane_base + (b ? odd : 0u));
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctl->main_empty[b]));
        };
        uint32_t s = static_cast<uint32_t>(grp), sph = 0;          // ring position of this group's next k-block
        for (int c = 0; c < chunks && ok; ++c) {
            const int i = c * kChunk + grp;
            if (i < nkb) {
                ok = mbar_wait_warp(smem_u32(&ctl->split_empty[h]), (static_cast<uint32_t>(c) & 1u) ^ 1u, abort_flag, p.status);
                if (!ok) break;
                ok = mbar_wait_warp(full0 + 8 * s, sph, abort_flag, p.status);
                if (!ok) break;
                __syncwarp();                 // orders every lane's reads of the tile after lane 0's wait
                tc_fence_after();             // the MMAs of two k-blocks ago have read this half buffer
                const uint32_t stage = ring + s * kStage;
                split_a(stage, a_dst, a_mn, q, kh, lane);
                split_b<BN>(stage + kF32TileA, planes_b, kPlaneB, b_mn, h, w, lane);
                tmem_st_wait();
                tc_fence_before();
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(smem_u32(&ctl->split_full[h]));
                    mbar_arrive(empty0 + 8 * s);
                }
                s += 2;
                if (s >= NS) { s -= NS; sph ^= 1u; }
            }
            if (c > 0) drain(c - 1);
        }
        if (ok) drain(chunks - 1);
        if (ok) {
            ok = mbar_wait_warp(smem_u32(&ctl->corr_full), 0, abort_flag, p.status);
            tc_fence_after();
        }
        if (ok) {
            add_from(lane_base + (3 * BN - odd));
            constexpr uint32_t kPieces = kCols / 4, kRowBytes = kCols * 4;
            if (p.splits > 1) {
                // slice: straight to the workspace, [column quarter][quadrant][4-column group][row][4], a run of 512 bytes
                // per instruction; then the warp reports
                float* dst = p.partial + (static_cast<size_t>(tile) * p.splits + bz) * (128u * BN) +
                             static_cast<size_t>(colq * 4 + q) * (32 * kCols) + lane * 4;
#pragma unroll
                for (uint32_t g = 0; g < kPieces; ++g)
                    *reinterpret_cast<float4*>(dst + g * 128) = make_float4(acc[4 * g], acc[4 * g + 1], acc[4 * g + 2], acc[4 * g + 3]);
                __syncwarp();
                if (lane == 0) red_release_gpu(p.counters + 2 * tile, 1u);
            } else {
                // 32 rows of kCols floats go through shared memory (the ring is idle: every warp has split its last k-block once
                // corr_full fired), 16-byte pieces XOR-permuted by the row against bank conflicts
                const uint32_t panel = ring + static_cast<uint32_t>(colq * 128 + q * 32) * kRowBytes;
                const uint32_t own = panel + static_cast<uint32_t>(lane) * kRowBytes;
    #pragma unroll
                for (uint32_t g = 0; g < kPieces; ++g)
                    st_shared_v4(own + ((g ^ (static_cast<uint32_t>(lane) & (kPieces - 1))) << 4),
                                 make_uint4(__float_as_uint(acc[4 * g]), __float_as_uint(acc[4 * g + 1]), __float_as_uint(acc[4 * g + 2]),
                                            __float_as_uint(acc[4 * g + 3])));
                // stored as whole row segments, 32 / kPieces rows per instruction
                __syncwarp();
                constexpr int kRowsPer = 32 / static_cast<int>(kPieces);
                const int sub = lane / static_cast<int>(kPieces), piece = lane % static_cast<int>(kPieces);
                const bool vec = (p.ldc % 4) == 0 && (reinterpret_cast<uintptr_t>(p.C) & 15) == 0;
                const int col = n0 + colq * kCols + piece * 4;
                float4 b = make_float4(0.f, 0.f, 0.f, 0.f);
                if (p.bias) {
                    if (col < p.N) b.x = __ldg(p.bias + col);
                    if (col + 1 < p.N) b.y = __ldg(p.bias + col + 1);
                    if (col + 2 < p.N) b.z = __ldg(p.bias + col + 2);
                    if (col + 3 < p.N) b.w = __ldg(p.bias + col + 3);
                }
                float probe = 0.f;        // becomes NaN with a sum that is not finite
#pragma unroll 4
                for (int i = 0; i < 32 / kRowsPer; ++i) {
                    const int rr = i * kRowsPer + sub;
                    const uint4 u = ld_shared_v4(panel + static_cast<uint32_t>(rr) * kRowBytes +
                                                 ((static_cast<uint32_t>(piece) ^ (static_cast<uint32_t>(rr) & (kPieces - 1))) << 4));
                    float4 v = make_float4(fmaf(__uint_as_float(u.x), kUnscale, b.x), fmaf(__uint_as_float(u.y), kUnscale, b.y),
                                           fmaf(__uint_as_float(u.z), kUnscale, b.z), fmaf(__uint_as_float(u.w), kUnscale, b.w));
                    const int row = f32_row<kMode>(p, org, bx, q * 32 + rr);
                    if (row < 0) continue;
                    probe = fmaf(__uint_as_float(u.x), 0.f, fmaf(__uint_as_float(u.y), 0.f, fmaf(__uint_as_float(u.z), 0.f, fmaf(__uint_as_float(u.w), 0.f, probe))));
                    if (p.act == 1) v = make_float4(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f), fmaxf(v.z, 0.f), fmaxf(v.w, 0.f));
                    float* dst = p.C + static_cast<size_t>(row) * p.ldc + col;
                    if (vec && col + 3 < p.N) {
                        *reinterpret_cast<float4*>(dst) = v;
                    } else {
                        if (col < p.N) dst[0] = v.x;
                        if (col + 1 < p.N) dst[1] = v.y;
                        if (col + 2 < p.N) dst[2] = v.z;
                        if (col + 3 < p.N) dst[3] = v.w;
                    }
                    if (p.C2) {
                        float* d2 = p.C2 + static_cast<size_t>(row) * p.ldc2 + col;
                        if (col < p.N) d2[0] = v.x;
                        if (col + 1 < p.N) d2[1] = v.y;
                        if (col + 2 < p.N) d2[2] = v.z;
                        if (col + 3 < p.N) d2[3] = v.w;
                    }
                }
                if (probe != 0.f) *repair = 1u;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, 512);
    if (p.splits <= 1) {
        if (*repair) f32_repair<BN, kMode>(p, bx, by, bz);
        return;
    }

    // ---- slice sum (as in pf_tc_gemm_kernel.cuh): once all slices of the tile are in the workspace, each CTA adds its
    // share of them in slice order and stores the sums
    unsigned int* cnt = p.counters + 2 * tile;
    const int S = p.splits;
    if (threadIdx.x == 0) {
        uint32_t good = (*abort_flag == 0u) ? 1u : 0u;
        const unsigned int want = 16u * static_cast<unsigned int>(S);
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
        // units of 8 rows x 16 columns, one per warp and step
        constexpr int kUnits = 16 * (BN / 16), kQuarter = kCols / 16 > 0 ? kCols / 16 : 1;
        constexpr size_t kSlice = 128 * BN / 4;                  // float4s
        const bool vec = (p.ldc % 4) == 0 && (reinterpret_cast<uintptr_t>(p.C) & 15) == 0;
        const int per = (kUnits + S - 1) / S, end = min(kUnits, (bz + 1) * per);
#pragma unroll 1
        for (int u = bz * per + warp; u < end; u += kF32Threads / 32) {
            const int oct = u / (BN / 16), cell = u - oct * (BN / 16), cq = cell / kQuarter;
            const int pc = (cell - cq * kQuarter) * 4 + (lane >> 3), rr = oct * 8 + (lane & 7);
            const float4* src = reinterpret_cast<const float4*>(p.partial) + static_cast<size_t>(tile) * S * kSlice +
                                ((cq * 4 + (rr >> 5)) * (kCols / 4) + pc) * 32 + (rr & 31);
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
            for (int s0 = 0; s0 < S; s0 += 8) {
                float4 w[8];
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (s0 + i < S) w[i] = __ldcg(src + static_cast<size_t>(s0 + i) * kSlice);
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (s0 + i < S) { a.x += w[i].x; a.y += w[i].y; a.z += w[i].z; a.w += w[i].w; }
            }
            const int row = f32_row<kMode>(p, org, bx, rr), col = n0 + cq * kCols + pc * 4;
            if (row < 0) continue;
            if (fmaf(a.x, 0.f, fmaf(a.y, 0.f, fmaf(a.z, 0.f, a.w * 0.f))) != 0.f) *repair = 1u;
            a = make_float4(a.x * kUnscale, a.y * kUnscale, a.z * kUnscale, a.w * kUnscale);
            const float v[4] = {a.x, a.y, a.z, a.w};
            float* dst = p.C + static_cast<size_t>(row) * p.ldc + col;
            if (vec && col + 3 < p.N) *reinterpret_cast<float4*>(dst) = a;
            else
                for (int e = 0; e < 4; ++e)
                    if (col + e < p.N) dst[e] = v[e];
            if (p.C2)
                for (int e = 0; e < 4; ++e)
                    if (col + e < p.N) p.C2[static_cast<size_t>(row) * p.ldc2 + col + e] = v[e];
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
    if (*repair) f32_repair<BN, kMode>(p, bx, by, bz);
}

// Up to three independent products in one launch, blocks [end[i - 1], end[i]) working on product i; kConv compiles the
// convolution's addressing modes in (a translation unit of its own, as for the bf16 kernels).
template <int kMode>
__device__ __forceinline__ void f32_any(const CUtensorMap& ta, const CUtensorMap& tb, const F32Params& p, int idx) {
    const int bx = idx % p.tiles_x, by = (idx / p.tiles_x) % p.tiles_y, bz = idx / (p.tiles_x * p.tiles_y);
    if (p.bn == 64) f32_tile<64, kMode>(ta, tb, p, bx, by, bz);
    else f32_tile<128, kMode>(ta, tb, p, bx, by, bz);
}
template <bool kConv>
__device__ __forceinline__ void f32_product(const CUtensorMap& ta, const CUtensorMap& tb, const F32Params& p, int idx) {
    if constexpr (kConv) {
        if (p.mode == 1) return f32_any<1>(ta, tb, p, idx);
        if (p.mode == 2) return f32_any<2>(ta, tb, p, idx);
        if (p.mode == 3) return f32_any<3>(ta, tb, p, idx);
    }
    f32_any<0>(ta, tb, p, idx);
}
template <bool kConv>
__global__ void __launch_bounds__(kF32Threads, 1)
tc_f32_kernel(const __grid_constant__ F32Launch a) {
    const int idx = blockIdx.x;
    const int i = idx < a.end[0] ? 0 : idx < a.end[1] ? 1 : 2;
    f32_product<kConv>(a.ta[i], a.tb[i], a.p[i], idx - (i > 0 ? a.end[i - 1] : 0));
}

}  // namespace
}  // namespace tc
}  // namespace pf
#endif
