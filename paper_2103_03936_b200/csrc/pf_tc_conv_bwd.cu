// Backward of 3 x 3, stride-1 convolutions (padding 1, R <= 64) in three launches that each read their images once or
// nearly so:
//   tc_conv_dt_dv_kernel   dT = dY V and dV = dY^T T from one pass over dY: a block's rows of dY lie in shared memory once, as the
//                          K-major operand of the first product and the MN-major one of the second
//   tc_conv_du_kernel      dU: per (128 channels, tap row) one accumulator of 128 x 192, the row's three taps side by side: the image
//                          of dT lies in the flat sequence of pf_tc_conv_flat.cuh, in which the taps of a row are the same tile read
//                          one position (128 bytes) further, i.e. three column panels 128 bytes apart
//   tc_conv_dx_kernel      dX = taps(dT, U^T) on resident windows of dT, as the forward's first product
// The two reductions leave slices in the workspace, which warps of the launch behind add up beside its products: nothing waits
// for the sums.
// The form before (dT; then dU, dV and dX in one launch of 128 x 128 and 128 x 64 tiles) moves 1.6 GB through the SMs' load paths at
// 128 x 32 x 32, 256 -> 64 -> 256 (x once per tap for dU, dT once per tap for dX), 0.45 here: backward 111.6 -> 85.2 us, training step
// 196.4 -> 162.  By ncu, one launch at a time, they take 24, 32 and 36 us: the first is bound by memory (104 MB and 7 of slices), the second
// by the tensor cores (busy 58 %; a 128 x 192 x 16 MMA takes 101 clocks) and its 29 MB of slices, the third by the pace at which one
// thread issues MMAs and by shared memory (a 128 x 128 x 16 MMA reads 8 KB in its 64 clocks, all there is).
#include <cmath>

#include "pf_tc_conv_flat.cuh"

namespace pf {
namespace tc {
namespace {

// ------------------------------------------------------------------------------ dT and dV
constexpr int kStreamThreads = 192;          // 0 loads, 1 MMAs, 2..5 epilogue
constexpr int kStreamMaxStages = 5;
constexpr uint32_t kPanel = 16384;           // 128 rows x 64 columns
constexpr uint32_t kStreamStage = 2 * kPanel;
struct DtDvCtl {
    uint64_t v_full, t_full[2], t_empty[2], full[kStreamMaxStages], empty[kStreamMaxStages];
    uint64_t dt_full[2], dt_empty[2], dv_full;
    uint32_t tmem_base, abort;
};
__global__ void __launch_bounds__(kStreamThreads, 1)
tc_conv_dt_dv_kernel(const __grid_constant__ CUtensorMap tmY, const __grid_constant__ CUtensorMap tmT, const __grid_constant__ CUtensorMap tmV,
                     const __grid_constant__ DtDvParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t* smem = smem_raw + (((raw + 1023u) & ~1023u) - raw);
    DtDvCtl* ctl = reinterpret_cast<DtDvCtl*>(smem);
    const uint32_t base = smem_u32(smem);
    const uint32_t sT = base + 1024u, stg = sT + 2 * kPanel, sV = stg + 4 * 4096u, ring = sV + static_cast<uint32_t>(p.panels) * 8192u;
    volatile uint32_t* abort_flag = &ctl->abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t NS = static_cast<uint32_t>(p.num_stages);
    const int first = static_cast<int>(blockIdx.x), step = static_cast<int>(gridDim.x);

    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&ctl->v_full), 1);
        mbar_init(smem_u32(&ctl->dv_full), 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&ctl->t_full[b]), 1);
            mbar_init(smem_u32(&ctl->t_empty[b]), 1);
            mbar_init(smem_u32(&ctl->dt_full[b]), 1);
            mbar_init(smem_u32(&ctl->dt_empty[b]), 4);
        }
        for (uint32_t s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&ctl->full[s]), 1);
            mbar_init(smem_u32(&ctl->empty[s]), 1);
        }
        ctl->abort = 0;
        fence_barrier_init();
        fence_proxy_async_smem();
        tma_prefetch_desc(&tmY);
        tma_prefetch_desc(&tmT);
        tma_prefetch_desc(&tmV);
    }
    if (warp == 1) tmem_alloc(smem_u32(&ctl->tmem_base), 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp != 0 || !p.early) {
        pdl_wait();
        pdl_launch_dependents();
    }
    const uint32_t tmem = ctl->tmem_base;

    if (warp == 0) {
        if (elect_one()) {
            const uint32_t v_full = smem_u32(&ctl->v_full);
            uint32_t s = 0, ph = 1;
            bool ok = true;
            for (int t = first, i = 0; t < p.tiles && ok; t += step, ++i) {
                const uint32_t b = static_cast<uint32_t>(i) & 1u;
                for (int c = 0; c < p.pairs; ++c) {
                    ok = mbar_wait(smem_u32(&ctl->empty[s]), ph, abort_flag, p.status);
                    if (!ok) break;
                    const uint32_t full = smem_u32(&ctl->full[s]), dst = ring + s * kStreamStage;
                    const bool two = 2 * c + 1 < p.panels;
                    mbar_expect_tx(full, two ? kStreamStage : kPanel);
                    tma_load_2d(dst, &tmY, full, c * 128, t * 128);
                    if (two) tma_load_2d(dst + kPanel, &tmY, full, c * 128 + 64, t * 128);
                    if (++s == NS) { s = 0; ph ^= 1u; }
                    if (c == 0) {
                        if (i == 0) {
                            mbar_expect_tx(v_full, static_cast<uint32_t>(p.panels) * 8192u);
                            for (int k = 0; k < p.panels; ++k) tma_load_2d(sV + k * 8192, &tmV, v_full, 0, k * 64);
                        }
                        ok = mbar_wait(smem_u32(&ctl->t_empty[b]), (static_cast<uint32_t>(i >> 1) & 1u) ^ 1u, abort_flag, p.status);
                        if (!ok) break;
                        const uint32_t tf = smem_u32(&ctl->t_full[b]);
                        mbar_expect_tx(tf, kPanel);
                        tma_load_2d(sT + b * kPanel, &tmT, tf, 0, t * 128);
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            const uint32_t idesc_t = make_idesc_bf16(128, 64, 0, 1), idesc_v = make_idesc_bf16(128, 64, 1, 1);
            uint32_t s = 0, ph = 0;
            bool ok = mbar_wait(smem_u32(&ctl->v_full), 0, abort_flag, p.status);
            for (int t = first, i = 0; t < p.tiles && ok; t += step, ++i) {
                const uint32_t b = static_cast<uint32_t>(i) & 1u, par = static_cast<uint32_t>(i >> 1) & 1u;
                ok = mbar_wait(smem_u32(&ctl->dt_empty[b]), par ^ 1u, abort_flag, p.status) && mbar_wait(smem_u32(&ctl->t_full[b]), par, abort_flag, p.status);
                if (!ok) break;
                const uint64_t bt = make_smem_desc(sT + b * kPanel, 8192, 1024);
                for (int c = 0; c < p.pairs; ++c) {
                    ok = mbar_wait(smem_u32(&ctl->full[s]), ph, abort_flag, p.status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t at = ring + s * kStreamStage;
                    const int n = min(2, p.panels - 2 * c);
                    for (int h = 0; h < n; ++h) {
                        const uint64_t a = make_smem_desc(at + h * kPanel, 16, 1024), v = make_smem_desc(sV + (2 * c + h) * 8192, 8192, 1024);
#pragma unroll
                        for (int k = 0; k < 4; ++k) tc_mma_bf16(tmem + b * 64, a + 2 * k, v + 128 * k, idesc_t, c + h + k > 0 ? 1u : 0u);
                    }
                    const uint64_t a = make_smem_desc(at, kPanel, 1024);
#pragma unroll
                    for (int k = 0; k < 8; ++k) tc_mma_bf16(tmem + 128 + c * 64, a + 128 * k, bt + 128 * k, idesc_v, i + k > 0 ? 1u : 0u);
                    tc_commit(smem_u32(&ctl->empty[s]));
                    if (++s == NS) { s = 0; ph ^= 1u; }
                }
                if (!ok) break;
                tc_commit(smem_u32(&ctl->t_empty[b]));
                tc_commit(smem_u32(&ctl->dt_full[b]));
            }
            if (ok) tc_commit(smem_u32(&ctl->dv_full));
        }
    } else {
        const int q = warp & 3, sub = lane >> 3, piece = lane & 7;
        const uint32_t lanes = tmem + (static_cast<uint32_t>(q * 32) << 16);
        const uint32_t panel = stg + static_cast<uint32_t>(warp - 2) * 4096u, own = panel + static_cast<uint32_t>(lane) * 128u, sw = static_cast<uint32_t>(lane & 7);
        bool ok = true;
        for (int t = first, i = 0; t < p.tiles; t += step, ++i) {
            const uint32_t b = static_cast<uint32_t>(i) & 1u;
            ok = mbar_wait_warp(smem_u32(&ctl->dt_full[b]), static_cast<uint32_t>(i >> 1) & 1u, abort_flag, p.status);
            tc_fence_after();
            if (!ok) break;
            uint32_t v0[32], v1[32];
            tmem_ld32(lanes + b * 64, v0);
            tmem_ld32(lanes + b * 64 + 32, v1);
            tmem_ld_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctl->dt_empty[b]));
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const uint32_t* v = e < 4 ? v0 + 8 * e : v1 + 8 * (e - 4);
                st_shared_v4(own + ((static_cast<uint32_t>(e) ^ sw) << 4),
                             make_uint4(pack_bf16x2(__uint_as_float(v[0]), __uint_as_float(v[1])), pack_bf16x2(__uint_as_float(v[2]), __uint_as_float(v[3])),
                                        pack_bf16x2(__uint_as_float(v[4]), __uint_as_float(v[5])), pack_bf16x2(__uint_as_float(v[6]), __uint_as_float(v[7]))));
            }
            __syncwarp();
            const int row0 = t * 128 + q * 32;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int rr = e * 4 + sub;
                const uint4 w = ld_shared_v4(panel + static_cast<uint32_t>(rr) * 128u + ((static_cast<uint32_t>(piece) ^ static_cast<uint32_t>(rr & 7)) << 4));
                if (row0 + rr < p.rows && piece * 8 < p.R) *reinterpret_cast<uint4*>(p.dT + static_cast<size_t>(row0 + rr) * p.ldt + piece * 8) = w;
            }
            __syncwarp();
        }
        if (ok) ok = mbar_wait_warp(smem_u32(&ctl->dv_full), 0, abort_flag, p.status);
        tc_fence_after();
        for (int c = 0; c < p.pairs && ok; ++c) {
            uint32_t v[2][32];
            tmem_ld32(lanes + 128 + c * 64, v[0]);
            tmem_ld32(lanes + 128 + c * 64 + 32, v[1]);
            tmem_ld_wait();
            float* dst = p.partial + (static_cast<size_t>(c) * gridDim.x + blockIdx.x) * 8192u + static_cast<size_t>(q * 16 * 32 + lane) * 4;
#pragma unroll
            for (int g = 0; g < 16; ++g)
                *reinterpret_cast<uint4*>(dst + static_cast<size_t>(g) * 128) =
                    make_uint4(v[g >> 3][4 * (g & 7)], v[g >> 3][4 * (g & 7) + 1], v[g >> 3][4 * (g & 7) + 2], v[g >> 3][4 * (g & 7) + 3]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tmem_dealloc(tmem, 512);
    }
}

// ------------------------------------------------------------------------------ sums of slices
// Units of 8 rows x 16 columns: a lane sums four columns of a row over all slices, in slice order, kDeep slices in flight.
struct SumAt {
    int row, col;                // of the result; row -1: none
    float4 v;
};
template <int kDeep>
__device__ __forceinline__ SumAt sum_unit(const SumPart& s, int u, int lane) {
    const int tile = u >> 6, in = u & 63, rr = (in >> 2) * 8 + (lane & 7), pc = (in & 3) * 4 + (lane >> 3);
    const bool tail = tile >= s.tail;
    const int S = tail ? s.split[1] : s.split[0];
    const size_t base = tail ? static_cast<size_t>(s.tail) * s.split[0] + static_cast<size_t>(tile - s.tail) * S : static_cast<size_t>(tile) * S;
    const float4* src = reinterpret_cast<const float4*>(s.partial) + base * 2048u + ((rr >> 5) * 16 + pc) * 32 + (rr & 31);
    float4 a = make_float4(-0.f, -0.f, -0.f, -0.f);
#pragma unroll 1
    for (int s0 = 0; s0 < S; s0 += kDeep) {
        float4 w[kDeep];
#pragma unroll
        for (int i = 0; i < kDeep; ++i)
            if (s0 + i < S) w[i] = __ldcg(src + static_cast<size_t>(s0 + i) * 2048u);
#pragma unroll
        for (int i = 0; i < kDeep; ++i)
            if (s0 + i < S) { a.x += w[i].x; a.y += w[i].y; a.z += w[i].z; a.w += w[i].w; }
    }
    int row = tile * 128 + rr;
    if (s.per_tap > 0) {
        const int tap = tile / s.per_tap, c = (tile - tap * s.per_tap) * 128 + rr;
        row = c < s.rows ? tap * s.rows + c : -1;
    } else if (row >= s.rows) {
        row = -1;
    }
    return SumAt{pc * 4 < s.R ? row : -1, pc * 4, a};
}
// kPlain: bf16, not added to anything, on a 16-byte boundary.
template <bool kPlain>
__device__ __forceinline__ void put_sum(const SumPart& s, const SumAt& a) {
    const size_t at = static_cast<size_t>(a.row) * s.R + a.col;
    if (kPlain) {
        *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(s.out) + at) = make_uint2(pack_bf16x2(a.v.x, a.v.y), pack_bf16x2(a.v.z, a.v.w));
        return;
    }
    const float v[4] = {a.v.x, a.v.y, a.v.z, a.v.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        if (s.f32) {
            float* o = static_cast<float*>(s.out) + at + e;
            *o = s.accumulate ? *o + v[e] : v[e];
        } else {
            __nv_bfloat16* o = static_cast<__nv_bfloat16*>(s.out) + at + e;
            *o = __float2bfloat16_rn(s.accumulate ? __bfloat162float(*o) + v[e] : v[e]);
        }
    }
}
__device__ __forceinline__ bool has_nan(const float4& v) { return v.x != v.x || v.y != v.y || v.z != v.z || v.w != v.w; }
// One unit per warp and step; returns whether this lane has left out sums that are NaN (kLeave).
template <bool kLeave, bool kPlain>
__device__ __forceinline__ bool sum_units(const SumPart& s, int first, int step, int lane) {
    bool left = false;
#pragma unroll 1
    for (int u = first; u < s.tiles * 64; u += step) {
        const SumAt a = sum_unit<16>(s, u, lane);
        if (a.row < 0) continue;
        if (kLeave && has_nan(a.v)) left = true;
        else put_sum<kPlain>(s, a);
    }
    return left;
}
template <bool kLeave>
__device__ __forceinline__ bool sum_slices(const SumPart& s, int first, int step, int lane) {
    return s.plain ? sum_units<kLeave, true>(s, first, step, lane) : sum_units<kLeave, false>(s, first, step, lane);
}

// The sums of dU that sum_slices has left out.  The MMAs of tc_conv_du_kernel take the three taps of a row from one tile of x, so they
// multiply border pixels by the zeros around dT for the taps that pair them with nothing: an infinity or NaN there makes those taps' sums
// NaN.  So each NaN is computed once more, over the pairs that exist, in fp32: a warp for 8 columns of a row, lanes along the
// pixels, up to where all 8 are NaN.  Finite data pay nothing (backward of 128 x 32 x 32, 256 -> 64 -> 256: 84.7 us with and without);
// one infinity at a border makes it 2.4 ms, a column of them 19, one pixel in 10000 42.  (In few registers, for they are the kernel's: with 128, 8 columns in
// flight more, no block of the next kernel fits beside and the training step of that size took 164 us, 162 with 108.)
__device__ __noinline__ void mend_sums(const DxParams& p, int first, int step, int lane) {
    const FlatImage& f = p.f;
    const SumPart& s = p.sum;
#pragma unroll 1
    for (int u = first; u < s.tiles * 64; u += step) {
        SumAt a = sum_unit<4>(s, u, lane);
        const bool bad = a.row >= 0 && has_nan(a.v);
        uint32_t rows = __ballot_sync(0xffffffffu, bad);
        rows = (rows | rows >> 8 | rows >> 16 | rows >> 24) & 0xffu;
        const int col0 = (u & 3) * 16;
#pragma unroll 1
        for (; rows != 0; rows &= rows - 1) {
            const int r = __ffs(rows) - 1, row = __shfl_sync(0xffffffffu, a.row, r), tap = row / s.rows, c = row - tap * s.rows;
            const int dy = tap / 3 - 1, dx = tap - tap / 3 * 3 - 1, y0 = max(0, -dy), x0 = max(0, -dx);
            const int cols = f.W - abs(dx), per_image = (f.H - abs(dy)) * cols, count = f.N * per_image;
#pragma unroll 1
            for (int half = 0; half < 2 && col0 + 8 * half < s.R; ++half) {
                float sum[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) sum[j] = 0.f;
#pragma unroll 1
                for (int i0 = 0; i0 < count; i0 += 1024) {
                    float part[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) part[j] = 0.f;
#pragma unroll 4
                    for (int i = i0 + lane; i < min(count, i0 + 1024); i += 32) {
                        const int n = i / per_image, in = i - n * per_image, y = in / cols;
                        const int64_t pix = (static_cast<int64_t>(n) * f.H + y0 + y) * f.W + x0 + in - y * cols;
                        const float v = __bfloat162float(p.x[(pix + dy * f.W + dx) * p.C + c]);
                        const uint4 d = *reinterpret_cast<const uint4*>(p.dT + pix * p.ldt + col0 + 8 * half);
                        const uint32_t w[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            part[2 * j] = fmaf(v, __uint_as_float(w[j] << 16), part[2 * j]);
                            part[2 * j + 1] = fmaf(v, __uint_as_float(w[j] & 0xffff0000u), part[2 * j + 1]);
                        }
                    }
                    uint32_t nan = 0;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        sum[j] += part[j];
                        if (sum[j] != sum[j]) nan |= 1u << j;
                    }
                    if (__reduce_or_sync(0xffffffffu, nan) == 0xffu) break;
                }
                float t[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int j = 0; j < 8; ++j) {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) sum[j] += __shfl_xor_sync(0xffffffffu, sum[j], o);
                    if ((lane >> 3 & 1) == j >> 2) t[j & 3] = sum[j];
                }
                if ((lane & 7) == r && lane >> 4 == half) {
                    if (a.v.x != a.v.x) a.v.x = t[0];
                    if (a.v.y != a.v.y) a.v.y = t[1];
                    if (a.v.z != a.v.z) a.v.z = t[2];
                    if (a.v.w != a.v.w) a.v.w = t[3];
                }
            }
        }
        if (bad) put_sum<false>(s, a);
    }
}

// ------------------------------------------------------------------------------ dU
// The contraction runs over blocks of at most 64 positions: whole rows of an image (or whole images), whose columns are the image's
// where 16 divides its width, else the flat sequence's (one zero column more).  dT always has that column, so that
// the neighbour of a row's first and last pixel is zero.  A block's CTA holds two accumulators ("units"): tap rows 0 and 1 of
// 128 channels, or tap row 2 of two blocks of 128 channels.
constexpr int kDuThreads = 224;              // 0 loads x, 1 MMAs, 2..5 epilogue, 6 loads dT
constexpr int kDuStages = 5;
constexpr uint32_t kDuX = 8192;              // 64 positions x 64 channels
constexpr uint32_t kDuLead = 8;              // zero rows in front of dT's
constexpr uint32_t kDuT = 88 * 128;
constexpr uint32_t kDuStage = 4 * kDuX + kDuT;        // four panels of x and one copy of dT (tap row 2), or two and two
static_assert(kDuStage >= 2 * kDuX + 2 * kDuT && kDuStage % 1024 == 0 && kDuT % 1024 == 0, "");
struct DuCtl {
    uint64_t full[kDuStages], empty[kDuStages], acc_full;
    uint32_t tmem_base, abort;
};
__global__ void __launch_bounds__(kDuThreads, 1)
tc_conv_du_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmT, const __grid_constant__ DuParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t* smem = smem_raw + (((raw + 1023u) & ~1023u) - raw);
    DuCtl* ctl = reinterpret_cast<DuCtl*>(smem);
    const uint32_t ring = smem_u32(smem) + 1024u;
    volatile uint32_t* abort_flag = &ctl->abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // which units: block b of channels with tap rows 0 and 1, or blocks b and b + 1 with tap row 2
    int idx = static_cast<int>(blockIdx.x);
    const bool rows01 = idx < p.tb * p.split[0];
    if (!rows01) idx -= p.tb * p.split[0];
    const int S = p.split[rows01 ? 0 : 1], cls = idx / S, slice = idx - cls * S;
    const int b0 = rows01 ? cls : 2 * cls, units = rows01 || b0 + 1 < p.tb ? 2 : 1;
    const int beg = slice * p.per[rows01 ? 0 : 1], n = min(p.blocks, beg + p.per[rows01 ? 0 : 1]) - beg;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kDuStages; ++s) {
            mbar_init(smem_u32(&ctl->full[s]), 2);
            mbar_init(smem_u32(&ctl->empty[s]), 1);
        }
        mbar_init(smem_u32(&ctl->acc_full), 1);
        ctl->abort = 0;
        fence_barrier_init();
        tma_prefetch_desc(&tmX);
        tma_prefetch_desc(&tmT);
    }
    // rows that TMA never writes have to read as zero
    for (uint32_t i = threadIdx.x; i < kDuStages * kDuStage / 16; i += kDuThreads) st_shared_v4(ring + i * 16, make_uint4(0, 0, 0, 0));
    fence_proxy_async_smem();
    if (warp == 1) tmem_alloc(smem_u32(&ctl->tmem_base), 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp != 0) {            // (x was complete before the launch that writes dT: see kEarlyA)
        pdl_wait();
        pdl_launch_dependents();
    }
    const uint32_t tmem = ctl->tmem_base;

    if (warp == 0 || warp == 6) {
        if (elect_one()) {
            const bool do_x = warp == 0;
            const int panels = rows01 ? 2 : 4, c0 = b0 * 128, have = min(panels, (p.C - c0 + 63) / 64);
            const uint32_t bytes = do_x ? static_cast<uint32_t>(have * p.kpix_x) * 128u : static_cast<uint32_t>((rows01 ? 2 : 1) * p.kpix_t) * 128u;
            const uint32_t to_t = static_cast<uint32_t>(panels) * kDuX + kDuLead * 128u;
            int g = beg / p.tpi, t = beg - g * p.tpi;
            uint32_t s = 0, ph = 1;
            for (int i = 0; i < n; ++i) {
                if (!mbar_wait(smem_u32(&ctl->empty[s]), ph, abort_flag, p.status)) break;
                const uint32_t full = smem_u32(&ctl->full[s]), dst = ring + s * kDuStage;
                mbar_expect_tx(full, bytes);
                const int y = t * p.bh, img = g * p.nb;
                if (do_x) {
                    for (int k = 0; k < have; ++k) tma_load_4d(dst + k * kDuX, &tmX, full, c0 + 64 * k, 0, y, img);
                } else if (rows01) {           // tap row ky pairs pixel row y with row y - (ky - 1) of dT
                    tma_load_4d(dst + to_t, &tmT, full, 0, 0, y + 1, img);
                    tma_load_4d(dst + to_t + kDuT, &tmT, full, 0, 0, y, img);
                } else {
                    tma_load_4d(dst + to_t, &tmT, full, 0, 0, y - 1, img);
                }
                if (++t == p.tpi) { t = 0; ++g; }
                if (++s == kDuStages) { s = 0; ph ^= 1u; }
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            const uint32_t idesc = make_idesc_bf16(128, 192, 1, 1);
            const uint32_t to_t = static_cast<uint32_t>(rows01 ? 2 : 4) * kDuX + (kDuLead - 1) * 128u;
            // second unit: the other copy of dT, or the other channels
            const uint32_t da = rows01 ? 0u : (2 * kDuX) >> 4, db = rows01 ? kDuT >> 4 : 0u;
            const uint64_t a_desc = make_smem_desc(ring, kDuX, 1024), b_desc = make_smem_desc(ring + to_t, 128, 1024);
            const uint32_t ah = desc_hi(a_desc), bh = desc_hi(b_desc), full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
            uint32_t a = desc_lo(a_desc), b = desc_lo(b_desc);
            // a step of 16 positions: 16 rows, and over dT's zero column at the end of an image row
            uint32_t to[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) to[k] = 128u * k + 8u * static_cast<uint32_t>(k / p.steps_row);
            const int ksteps = p.ksteps;
            uint32_t s = 0, ph = 0;
            bool ok = true;
            for (int i = 0; i < n; ++i) {
                ok = mbar_wait(full0 + 8 * s, ph, abort_flag, p.status);
                if (!ok) break;
                tc_fence_after();
                auto step = [&](uint32_t k, uint32_t more) {
                    tc_mma_bf16_words(tmem, a + 128 * k, ah, b + to[k], bh, idesc, more);
                    if (units == 2) tc_mma_bf16_words(tmem + 192, a + da + 128 * k, ah, b + db + to[k], bh, idesc, more);
                };
                step(0, i > 0 ? 1u : 0u);
                if (ksteps == 4) {
                    step(1, 1u);
                    step(2, 1u);
                    step(3, 1u);
                } else {
                    if (ksteps > 1) step(1, 1u);
                    if (ksteps > 2) step(2, 1u);
                }
                tc_commit(empty0 + 8 * s);
                a += kDuStage >> 4;
                b += kDuStage >> 4;
                if (++s == kDuStages) { s = 0; a -= kDuStages * (kDuStage >> 4); b -= kDuStages * (kDuStage >> 4); ph ^= 1u; }
            }
            if (ok) tc_commit(smem_u32(&ctl->acc_full));
        }
    } else {
        const int q = warp & 3;
        const uint32_t lanes = tmem + (static_cast<uint32_t>(q * 32) << 16);
        // while the products run: the slices of dV, which the launch before has left
        sum_slices<false>(p.sum, static_cast<int>(blockIdx.x) * 4 + warp - 2, static_cast<int>(gridDim.x) * 4, lane);
        const bool ok = mbar_wait_warp(smem_u32(&ctl->acc_full), 0, abort_flag, p.status);
        tc_fence_after();
        if (ok) {
#pragma unroll 1
            for (int e = 0; e < units * 3; ++e) {
                const int u = e / 3, j = e - 3 * u;
                const int ky = rows01 ? u : 2, tap = ky * 3 + 2 - j, tile = tap * p.tb + (rows01 ? b0 : b0 + u);
                const size_t first = rows01 ? static_cast<size_t>(tile) * p.split[0]
                                            : static_cast<size_t>(6 * p.tb) * p.split[0] + static_cast<size_t>(tile - 6 * p.tb) * p.split[1];
                uint32_t v[2][32];
                tmem_ld32(lanes + u * 192 + j * 64, v[0]);
                tmem_ld32(lanes + u * 192 + j * 64 + 32, v[1]);
                tmem_ld_wait();
                float* dst = p.partial + (first + slice) * 8192u + static_cast<size_t>(q * 16 * 32 + lane) * 4;
#pragma unroll
                for (int g = 0; g < 16; ++g)
                    *reinterpret_cast<uint4*>(dst + static_cast<size_t>(g) * 128) =
                        make_uint4(v[g >> 3][4 * (g & 7)], v[g >> 3][4 * (g & 7) + 1], v[g >> 3][4 * (g & 7) + 2], v[g >> 3][4 * (g & 7) + 3]);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tmem_dealloc(tmem, 512);
    }
}

// ------------------------------------------------------------------------------ dX, and the sums of the slices
constexpr int kDxThreads = 480;              // 0 loads windows, 1 MMAs, 2..9 epilogue, 10 loads U, 11..14 sums (without dX 2..9 too)
constexpr int kDxRows = 256;                 // positions of a tile: two row tiles
constexpr int kDxMaxStages = 8;
constexpr uint32_t kDxStage = 16384;         // one tap of U^T: 128 channels x 64 ranks
struct DxCtl {
    uint64_t a_full[2], a_empty[2], full[kDxMaxStages], empty[kDxMaxStages], acc_full[2], acc_empty[2];
    uint32_t tmem_base, abort;
};
// kFull: more than 48 ranks, i.e. four steps of 16 (a loop of p.ksteps steps issues the MMAs at half the pace of the tensor cores: 42.7 us
// by ncu at 128 x 32 x 32, 256 -> 64 -> 256, 36.2 unrolled).
template <bool kFull>
__global__ void __launch_bounds__(kDxThreads, 1)
tc_conv_dx_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const __grid_constant__ DxParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t* smem = smem_raw + (((raw + 1023u) & ~1023u) - raw);
    DxCtl* ctl = reinterpret_cast<DxCtl*>(smem);
    const uint32_t base = smem_u32(smem);
    const uint32_t abuf = base + p.a_off, ring = base + p.ring_off;
    volatile uint32_t* abort_flag = &ctl->abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t NS = static_cast<uint32_t>(p.num_stages);
    const int step = p.step, first = static_cast<int>(blockIdx.x) < step ? static_cast<int>(blockIdx.x) : p.tiles;

    if (threadIdx.x == 0) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&ctl->a_full[b]), 1);
            mbar_init(smem_u32(&ctl->a_empty[b]), 1);
            mbar_init(smem_u32(&ctl->acc_full[b]), 1);
            mbar_init(smem_u32(&ctl->acc_empty[b]), 8);
        }
        for (uint32_t s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&ctl->full[s]), 1);
            mbar_init(smem_u32(&ctl->empty[s]), 1);
        }
        ctl->abort = 0;
        fence_barrier_init();
        fence_proxy_async_smem();
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
    }
    if (warp == 1) tmem_alloc(smem_u32(&ctl->tmem_base), 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp != 10) {           // (U was complete long before)
        pdl_wait();
        pdl_launch_dependents();
    }
    const uint32_t tmem = ctl->tmem_base;
    const FlatImage& f = p.f;
    // Warps of a block that add up slices: without dX the epilogue's join where four have more than a unit each (backward of 128 x 32 x 32, 256 -> 64 -> 256
    // 57.7 -> 54.9 us, of 64 x 28 x 28, 320 -> 40 -> 320 58.2 -> 50.0; with fewer units they would leave the blocks that end early nothing to end early
    // with, and the next call's first launch starts on those: 60 x 28 x 28, 80 -> 40 -> 80 33.0, 35.8 with twelve).
    const int own_sums = p.tiles == 0 && p.sum.tiles * 64 > 4 * static_cast<int>(gridDim.x) ? 12 : 4;
    auto first_unit = [&](int q0) { return floor_div(q0 - f.Wp - 1, f.unit_rows); };

    if (warp == 0) {
        if (elect_one()) {
            uint32_t b = 0, ph = 1;
            for (int t = first; t < p.tiles; t += step) {
                const int q0 = t * kDxRows, u0 = first_unit(q0), count = floor_div(q0 + kDxRows + f.Wp, f.unit_rows) - u0 + 1;
                if (!mbar_wait(smem_u32(&ctl->a_empty[b]), ph, abort_flag, p.status)) break;
                const uint32_t full = smem_u32(&ctl->a_full[b]);
                mbar_expect_tx(full, static_cast<uint32_t>(count * f.unit_rows) * 128u);
                load_window(f, &tmA, abuf + b * p.a_bytes, full, u0, count, 0);
                b ^= 1u;
                if (b == 0) ph ^= 1u;
            }
        }
    } else if (warp == 10) {
        if (elect_one()) {
            uint32_t s = 0, ph = 1;
            bool ok = true;
            for (int t = first; t < p.tiles && ok; t += step)
                for (int j = 0; j < p.nblk && ok; ++j)
                    for (int tap = 0; tap < 9; ++tap) {
                        ok = mbar_wait(smem_u32(&ctl->empty[s]), ph, abort_flag, p.status);
                        if (!ok) break;
                        const uint32_t full = smem_u32(&ctl->full[s]);
                        mbar_expect_tx(full, kDxStage);
                        tma_load_2d(ring + s * kDxStage, &tmB, full, 0, tap * p.C + j * 128);      // (rows past a tap's C: columns past C)
                        if (++s == NS) { s = 0; ph ^= 1u; }
                    }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            const uint32_t idesc = make_idesc_bf16(128, 128, 0, 0), full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
            const uint64_t u_desc = make_smem_desc(ring, 16, 1024);
            const uint32_t hi = desc_hi(u_desc), u0 = desc_lo(u_desc);       // (A's tiles have the same strides)
            const int ksteps = p.ksteps;
            uint32_t u = u0, s = 0, ph = 0, b = 0, bph = 0, use = 0;
            bool ok = true;
            for (int t = first; t < p.tiles && ok; t += step) {
                const int q0 = t * kDxRows, row0 = q0 - first_unit(q0) * f.unit_rows;
                ok = mbar_wait(smem_u32(&ctl->a_full[b]), bph, abort_flag, p.status);
                if (!ok) break;
                const uint32_t a0 = desc_lo(make_smem_desc(abuf + b * p.a_bytes, 16, 1024)) + static_cast<uint32_t>(row0) * 8u;
                for (int j = 0; j < p.nblk && ok; ++j, ++use) {
                    ok = mbar_wait(smem_u32(&ctl->acc_empty[use & 1u]), ((use >> 1) & 1u) ^ 1u, abort_flag, p.status);
                    if (!ok) break;
                    const uint32_t d = tmem + (use & 1u) * 256u;
                    int o = f.Wp + 1;                        // tap (0, 0) takes dT from one row and one column further
                    for (int tap = 0; tap < 9; ++tap) {
                        ok = mbar_wait(full0 + 8 * s, ph, abort_flag, p.status);
                        if (!ok) break;
                        tc_fence_after();
                        const uint32_t a = a0 + static_cast<uint32_t>(o * 8);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            if (!kFull && k >= ksteps) break;
                            const uint32_t acc = tap + k > 0 ? 1u : 0u;
                            tc_mma_bf16_words(d, a + 2 * k, hi, u + 2 * k, hi, idesc, acc);
                            tc_mma_bf16_words(d + 128, a + 1024 + 2 * k, hi, u + 2 * k, hi, idesc, acc);
                        }
                        tc_commit(empty0 + 8 * s);
                        u += kDxStage >> 4;
                        if (++s == NS) { s = 0; u = u0; ph ^= 1u; }
                        o -= tap == 2 || tap == 5 ? f.Wp - 2 : 1;
                    }
                    if (ok) tc_commit(smem_u32(&ctl->acc_full[use & 1u]));
                }
                if (!ok) break;
                tc_commit(smem_u32(&ctl->a_empty[b]));
                b ^= 1u;
                if (b == 0) bph ^= 1u;
            }
        }
    } else if (warp < 10 && own_sums == 4) {
        const int m = (warp - 2) >> 2, q4 = warp & 3;
        const uint32_t lanes = tmem + (static_cast<uint32_t>(q4 * 32) << 16) + static_cast<uint32_t>(m) * 128u;
        const uint32_t panel = base + p.stg_off + static_cast<uint32_t>(warp - 2) * 4096u;
        uint32_t use = 0;
        bool ok = true;
        for (int t = first; t < p.tiles && ok; t += step) {
            const int pix = pixel_of(f, t * kDxRows + m * 128 + q4 * 32 + lane);
            for (int j = 0; j < p.nblk; ++j, ++use) {
                ok = mbar_wait_warp(smem_u32(&ctl->acc_full[use & 1u]), (use >> 1) & 1u, abort_flag, p.status);
                tc_fence_after();
                if (!ok) break;
                store_block(lanes + (use & 1u) * 256u, panel, lane, pix, p.out, p.C, j * 128, p.C, &ctl->acc_empty[use & 1u]);
            }
        }
    } else {
        // (blocks without a tile are not kept waiting: they take their share of the sums first)
        const int unit = static_cast<int>(gridDim.x - 1 - blockIdx.x) * own_sums + (warp > 10 ? warp - 11 : warp + 2), units = static_cast<int>(gridDim.x) * own_sums;
        if (__any_sync(0xffffffffu, sum_slices<true>(p.sum, unit, units, lane))) mend_sums(p, unit, units, lane);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tmem_dealloc(tmem, 512);
    }
}

// ------------------------------------------------------------------------------ host
struct FlatBwd {
    FlatImage f;
    ConvTiling ct;               // of dU's contraction
    int wx;                      // columns of x's blocks
    int tb, split[2], per[2], grid_v, pairs;
    int v_stages, x_stages;
    uint32_t a_bytes;
    size_t smem_v, smem_x, bytes_u, bytes_v;
};
bool flat_bwd_plan(int N, int H, int W, int C, int R, int O, int kh, int kw, int stride, int pad, FlatBwd* b) {
    if (kh != 3 || kw != 3 || stride != 1 || pad != 1 || R > 64 || R % 8 || C % 8 || O % 8 || O > 512 || C > 1024 || W > 63 || N < 1) return false;
    const int64_t P = static_cast<int64_t>(N) * H * W;
    if (static_cast<int64_t>(N) * (H + 1) * (W + 1) >= (1 << 30)) return false;
    // dT and dV
    b->pairs = static_cast<int>(ceil_div(O, 128));
    // Blocks of the two reductions: one more shortens the blocks and lengthens the sums of the slices (a tile of dY takes a block about
    // 0.8 us, a block of positions 0.42, sixteen slices 1.5), so the best count grows with the root of the work.
    auto root = [](double v) { return static_cast<int>(std::ceil(std::sqrt(v))); };
    const int64_t tiles_v = ceil_div(P, 128), want_v = std::min<int64_t>(std::min<int64_t>(tiles_v, num_sms()), root(12.0 * static_cast<double>(tiles_v)));
    b->grid_v = static_cast<int>(ceil_div(tiles_v, ceil_div(tiles_v, want_v)));
    const size_t fixed = 1024 + 2 * kPanel + 4 * 4096 + static_cast<size_t>(ceil_div(O, 64)) * 8192, limit = 226 * 1024;
    b->v_stages = static_cast<int>(std::min<size_t>(kStreamMaxStages, (limit - fixed) / kStreamStage));
    b->smem_v = 1024 + fixed + b->v_stages * kStreamStage;
    b->bytes_v = align_up(static_cast<size_t>(b->pairs) * b->grid_v * 32768, 256);
    // dU
    b->wx = W % 16 == 0 ? W : W + 1;
    b->ct = conv_tiling(N, H, b->wx, 64);
    b->tb = static_cast<int>(ceil_div(C, 128));
    if (b->tb == 1) {
        b->split[0] = num_sms() * 2 / 3;
        b->split[1] = num_sms() - b->split[0];
    } else {
        b->split[0] = b->split[1] = num_sms() / (b->tb + static_cast<int>(ceil_div(b->tb, 2)));
    }
    const int want_u = root(4.5 * static_cast<double>(b->ct.blocks));
    b->split[0] = std::min(b->split[0], want_u);
    b->split[1] = std::min(b->split[1], b->tb == 1 ? (want_u + 1) / 2 : want_u);
    for (int i = 0; i < 2; ++i) {
        b->per[i] = static_cast<int>(ceil_div(b->ct.blocks, b->split[i]));
        b->split[i] = static_cast<int>(ceil_div(b->ct.blocks, b->per[i]));
    }
    b->bytes_u = align_up((static_cast<size_t>(6) * b->split[0] + static_cast<size_t>(3) * b->split[1]) * b->tb * 32768, 256);
    // dX
    b->f = flat_image(N, H, W);
    b->a_bytes = static_cast<uint32_t>(align_up(static_cast<size_t>(window_rows(b->f, kDxRows + 2 * b->f.Wp + 2)) * 128, 1024));
    const size_t before = 1024 + 2 * static_cast<size_t>(b->a_bytes) + 32768;
    if (before + 3 * kDxStage > limit) return false;
    b->x_stages = static_cast<int>(std::min<size_t>(kDxMaxStages, (limit - before) / kDxStage));
    b->smem_x = 1024 + before + b->x_stages * kDxStage;
    return true;
}
}  // namespace

// Against the launches that fetch pixels per tap (those / here, passes over buffers that do not fit L2; both with dT at a pitch of whole
// lines).  Rows of dT and U that straddle lines are what those suffer from, so at ranks of 24, 40 or 56 these pay early: 160 -> 40 -> 160 of 12544
// pixels 37.8 / 31.9 us, 50176 107.0 / 56.1; 64 -> 24 -> 64 of 12544 21.4 / 26.2, 25088 32.3 / 29.9; 448 -> 56 -> 448 of 12544 48.9 / 45.9; wide
// y later: 320 -> 56 -> 512 of 15680 42.0 / 46.6, 320 -> 24 -> 512 of 9200 39.3 / 40.5.  At 48: 192 -> 48 -> 192 of 12544 23.9 / 28.4, 25088
// 37.3 / 33.5.  Elsewhere the starts of three launches and the sums of the slices (10 to 20 us) want more: 256 -> 64 -> 256 of 25088
// 32.0 / 33.4, 50176 51.0 / 47.7, 131072 111.4 / 85.6; 128 -> 32 -> 128 of 25088 24.5 / 26.5, 100352 64.4 / 47.5; an expected time decides, fitted to an earlier
// state of these kernels, so it keeps to the other form up to 12 % beyond the crossing (512 -> 64 -> 512 of 25088 56.2 / 51.3).
// Without dX the other form has two launches and these still three, of which dX's share was the larger gain, so the line is a work of
// reductions (pixels times channels), less where rows straddle lines or the other form works most for padding, more where a block of 128
// channels is half empty: 192 -> 48 -> 192 of 25088 23.3 / 27.6, 50176 34.5 / 34.7, 75264 45.4 / 40.8; 256 -> 64 -> 256 of 25088 25.0 / 28.0, 50176 37.6 / 34.8; 128 ->
// 32 -> 128 of 50176 25.8 / 28.8, 100352 40.1 / 37.9; 64 -> 32 -> 64 of 131072 34.6 / 39.0; 128 -> 16 -> 128 of 62720 32.3 / 31.6, 128 -> 16 -> 256 of 86016 43.2 / 38.5; 64 ->
// 24 -> 64 of 50176 30.2 / 30.1, 75264 36.6 / 35.1; 160 -> 24 -> 160 of 26656 36.9 / 32.8; 160 -> 40 -> 160 of 12544 23.0 / 23.0, 25088 35.2 / 31.5; 320 ->
// 40 -> 320 of 12544 31.4 / 27.9; 256 -> 8 -> 256 of 15680 29.3 / 27.5.  Channels that leave a block of 64 ragged cost the other form more: 96 -> 48 -> 96 of
// 79968 40.2 / 35.0, 352 -> 56 -> 352 of 21952 37.9 / 31.3, 160 -> 64 -> 160 of 48608 32.2 / 33.9, 61152 37.4 / 37.0.
namespace {
bool flat_bwd_wanted(const ConvArgs& a, bool dX) {
    if (a.kh != 3 || a.stride != 1 || a.R > 64) return false;       // (most calls of other kinds: no plan is made for them)
    const double c = a.C / 100.0, p = static_cast<double>(a.N) * a.H * a.W / 1000.0, pc = p * c, po = p * a.O / 100.0;
    if (!dX) {
        if (a.R == 8 || a.R == 16 || a.R == 40) return pc >= (a.R == 8 ? 36.0 : a.R == 16 ? 76.0 : 16.0 + 5.0 * c);
        if (a.R == 24) return pc >= (a.C > 64 ? 33.0 + 2.0 * c : 44.0);
        return pc >= (a.C <= 64 ? 260.0 : a.R == 32 ? std::max(100.0, 125.0 - 13.0 * c) : 114.0) * (a.C % 64 == 0 ? 1.0 : 64 % a.R == 0 ? 0.8 : 0.66);
    }
    if (64 % a.R != 0) return a.R % 16 != 0 ? p >= (a.C >= 160 ? (a.O > a.C ? 18.0 : 11.0) : a.C >= 96 ? 16.0 : 25.0) : p >= (a.C >= 160 ? 20.0 : 50.0);
    return p >= 2.0 && 14.6 + 3.58 * c + 0.23 * p + 0.07 * pc + 0.05 * po < (a.R > 32 ? 0.9 : 1.05) * (12.35 + 0.07 * c + 0.16 * p + 0.19 * pc + 0.07 * po);
}
bool flat_bwd_plan(const ConvArgs& a, FlatBwd* b) { return flat_bwd_plan(a.N, a.H, a.W, a.C, a.R, a.O, a.kh, a.kw, a.stride, a.pad, b); }
}  // namespace

bool conv_flat_bwd_pays(const ConvArgs& a, bool dX) {
    FlatBwd b;
    return flat_bwd_wanted(a, dX) && flat_bwd_plan(a, &b);
}
size_t conv_flat_bwd_workspace(const ConvArgs& a) {
    FlatBwd b;
    return (flat_bwd_wanted(a, true) || flat_bwd_wanted(a, false)) && flat_bwd_plan(a, &b) ? b.bytes_u + b.bytes_v : 0;
}

// T: the stash, or x * U as a launch before left it.
int conv_flat_bwd(const ConvArgs& a, const void* T, const void* U, int64_t ldu, char* ws, bool early, const Before& before) {
    FlatBwd b;
    if (encode_fn() == nullptr || !flat_bwd_plan(a, &b)) return PF_ERR_UNSUPPORTED;
    const int64_t P = static_cast<int64_t>(a.N) * a.H * a.W;
    const int64_t ldt = conv_dt_pitch(a.R);
    float* pu = reinterpret_cast<float*>(ws);
    float* pv = reinterpret_cast<float*>(ws + b.bytes_u);
    unsigned int* status = device_status_ptr();
    CUtensorMap y, t, v, ux, ut, xa, xb;
    const bool ok = cached_map_2d(&y, a.dY, P, a.O, a.O, 128) && cached_map_2d(&t, T, P, a.R, a.R, 128) && cached_map_2d(&v, a.V, a.O, a.R, a.R, 64) &&
                    cached_map_nhwc(&ux, a.x, a.N, a.H, a.W, a.C, b.wx, b.ct.bh, b.ct.nb, 1) &&
                    cached_map_nhwc(&ut, a.ws_G, a.N, a.H, a.W, a.R, a.W + 1, b.ct.bh, b.ct.nb, 1, ldt) && window_map(&xa, b.f, a.ws_G, a.R, ldt) &&
                    cached_map_2d(&xb, U, static_cast<int64_t>(9) * a.C, a.R, ldu, 128);
    if (!ok) return PF_ERR_UNSUPPORTED;
    DtDvParams sp = {};
    sp.rows = static_cast<int>(P); sp.R = a.R;
    sp.tiles = static_cast<int>(ceil_div(P, 128));
    sp.panels = static_cast<int>(ceil_div(a.O, 64)); sp.pairs = b.pairs;
    sp.num_stages = b.v_stages;
    sp.dT = reinterpret_cast<__nv_bfloat16*>(a.ws_G);
    sp.ldt = static_cast<int>(ldt);
    sp.early = early;
    sp.partial = pv; sp.status = status;
    DuParams up = {};
    up.C = a.C; up.tb = b.tb;
    up.blocks = static_cast<int>(b.ct.blocks);
    for (int i = 0; i < 2; ++i) { up.split[i] = b.split[i]; up.per[i] = b.per[i]; }
    up.bh = b.ct.bh; up.nb = b.ct.nb; up.tpi = b.ct.tpi;
    up.kpix_x = b.ct.pixels;
    up.kpix_t = b.ct.nb * b.ct.bh * (a.W + 1);
    up.ksteps = static_cast<int>(ceil_div(b.ct.pixels, 16));
    up.steps_row = b.wx == a.W ? a.W / 16 : 1 << 20;
    up.partial = pu; up.status = status;
    DxParams xp = {};
    xp.f = b.f;
    xp.tiles = a.dX ? static_cast<int>(ceil_div(static_cast<int64_t>(b.f.N) * b.f.Hp * b.f.Wp, kDxRows)) : 0;
    xp.C = a.C; xp.nblk = static_cast<int>(ceil_div(a.C, 128)); xp.ksteps = static_cast<int>(ceil_div(a.R, 16));
    xp.out = static_cast<__nv_bfloat16*>(a.dX);
    xp.x = static_cast<const __nv_bfloat16*>(a.x); xp.dT = sp.dT; xp.ldt = sp.ldt;
    xp.a_bytes = b.a_bytes; xp.a_off = 1024; xp.stg_off = 1024 + 2 * b.a_bytes; xp.ring_off = xp.stg_off + 32768;
    xp.num_stages = b.x_stages;
    // (straight into the caller's matrices, whatever they hold: one more launch would read every slice again)
    const ConvArgs::Gradients* g = a.gradients;
    auto part = [&](const float* slices, void* plain, void* user) {
        SumPart s = {};
        s.partial = slices;
        s.out = g ? user : plain;
        s.f32 = g && g->f32; s.accumulate = g && g->accumulate;
        s.plain = !s.f32 && !s.accumulate && (reinterpret_cast<uintptr_t>(s.out) & 15) == 0;
        s.R = a.R;
        return s;
    };
    xp.sum = part(pu, a.dU, g ? g->dU : nullptr);
    xp.sum.tiles = 9 * b.tb; xp.sum.per_tap = b.tb; xp.sum.rows = a.C;
    xp.sum.split[0] = b.split[0]; xp.sum.split[1] = b.split[1]; xp.sum.tail = 6 * b.tb;
    up.sum = part(pv, a.dV, g ? g->dV : nullptr);
    up.sum.tiles = up.sum.tail = b.pairs; up.sum.rows = a.O;
    up.sum.split[0] = up.sum.split[1] = b.grid_v;
    xp.status = status;
    auto* dx_kernel = a.R > 48 ? tc_conv_dx_kernel<true> : tc_conv_dx_kernel<false>;
    const size_t smem_u = 1024 + 1024 + kDuStages * kDuStage;
    if (allow_smem(tc_conv_dt_dv_kernel, 227 * 1024) != cudaSuccess || allow_smem(tc_conv_du_kernel, smem_u) != cudaSuccess ||
        allow_smem(dx_kernel, 227 * 1024) != cudaSuccess)
        return PF_ERR_UNSUPPORTED;
    const int st = before();
    if (st != PF_OK) return st;
    if (launch_overlapped(tc_conv_dt_dv_kernel, dim3(static_cast<unsigned>(b.grid_v)), dim3(kStreamThreads), b.smem_v, a.stream, y, t, v, sp) != cudaSuccess) return PF_ERR_CUDA;
    count_launch();
    const int du_blocks = b.tb * b.split[0] + static_cast<int>(ceil_div(b.tb, 2)) * b.split[1];
    if (launch_overlapped(tc_conv_du_kernel, dim3(static_cast<unsigned>(du_blocks)), dim3(kDuThreads), smem_u, a.stream, ux, ut, up) != cudaSuccess) return PF_ERR_CUDA;
    count_launch();
    // (every SM has a block for the sums; tiles go round by an even number of blocks)
    xp.step = xp.tiles > 0 ? even_grid(xp.tiles) : 1;
    if (launch_overlapped(dx_kernel, dim3(static_cast<unsigned>(num_sms())), dim3(kDxThreads), b.smem_x, a.stream, xa, xb, xp) != cudaSuccess) return PF_ERR_CUDA;
    count_launch();
    if (a.gradients) a.gradients->written = true;
    return PF_OK;
}

}  // namespace tc
}  // namespace pf
