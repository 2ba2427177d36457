// 3 x 3, stride-1 convolutions (padding 1) whose image tile stays in shared memory while all nine taps read it.
//
// The implicit GEMM that fetches a tile's pixels once per tap is bound by its SM's load path (a 128-pixel tile of
// 256 channels pulls 864 KB through it, 112-116 KB/us, while the tensor cores idle half the time).  Here the image
// is seen as one flat sequence of positions
//     q = (n (H + 1) + h)(W + 1) + w ,      0 <= h <= H, 0 <= w <= W,
// in which column W and row H of every image are zeros (TMA's out-of-range fill): they are the right neighbour of one
// row and the left neighbour of the next, the bottom of one image and the top of the next.  In that sequence tap
// (dy, dx) of EVERY position is the position dy (W + 1) + dx further, so with positions as rows of a 128-byte-
// swizzled tile (64 channels each) the operand of a tap is the same tile read from another row on: a descriptor
// whose start address is a number of rows further (the swizzle is a function of the address, so any row will do;
// rows arrive by one box per image row, or per image when images are small).  A window of 256 + 2 (W + 2) positions
// serves 9 taps x 2 row tiles of 128 positions; the positions in column W and row H are computed and not stored.
// Per 64 channels of 256 positions at 32 x 32: 45 KB of image + 72 KB of factor instead of 432 KB.
//
// Forward: T = taps(x, U), then per 128 output channels y = T V^T with T (bf16) in shared memory; software-pipelined:
// the first product of tile t + 1 is issued before the second of tile t.  What bounds it now is shared-memory
// bandwidth (a 128 x 64 x 16 MMA reads 6 KB in 48 clocks; at 128 x 32 x 32 the MMAs' reads take 63 % of the data pipe's
// cycles and the epilogue's accesses 25 %, the tensor pipe is busy 35 %).  128 x 32 x 32, 256 -> 64 -> 256: 65.5 -> 55.3 us;
// 256 x 14 x 14: 37.8 -> 30.6; 32 x 56 x 56, 64 -> 16 -> 64: 32.3 -> 19.5 (back to back, caches warm, images after
// max(0, .); with a cold L2 60.4, 35.8 and 25.6).
//
// Warps: 0 = producer of image windows (two buffers), 1 = MMA issue, 2..9 = epilogue (four per row tile), 10 =
// producer of factor tiles (ring).  Persistent, one CTA per SM.  Every wait is bounded.
#include <cuda.h>

#include <algorithm>

#include "pf_tc_conv_flat.cuh"

namespace pf {
namespace tc {
namespace {

constexpr int kResThreads = 352;
constexpr int kResRows = 256;              // positions per tile: two row tiles of 128
constexpr int kResMaxStages = 12;

struct ResParams {
    FlatImage f;
    int tiles;               // of kResRows positions
    int cblks;               // 64-channel blocks of the window's image
    int ragged;              // C is not a multiple of 64, the factor map is [taps][C][R]
    int C;                   // channels per tap of U
    int R;                   // ranks (T's row length)
    int nblk;                // 128-column blocks of the output
    int Nout;                // output channels (row length of out)
    __nv_bfloat16 *out, *T;  // T: the stash or null
    uint32_t a_bytes;        // one window buffer
    uint32_t a_off, t_off, ring_off, stg_off;      // from the 1 KB-aligned base
    int num_stages;
    unsigned int* status;
};

struct ResCtl {
    uint64_t a_full[2], a_empty[2];
    uint64_t full[kResMaxStages], empty[kResMaxStages];
    uint64_t t_full[2], t_ready;         // accumulators of T complete / T is in shared memory
    uint64_t acc_full[2], acc_empty[2];  // output accumulator of a row tile
    uint32_t tmem_base, abort;
};

__global__ void __launch_bounds__(kResThreads, 1)
tc_conv_res_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB1, const __grid_constant__ CUtensorMap tmB2,
                   const __grid_constant__ ResParams p) {
    constexpr uint32_t kStage = 8192;          // one tap of U, or half a 128-column tile of V, 64 channels / columns deep
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t* smem = smem_raw + (((raw + 1023u) & ~1023u) - raw);
    ResCtl* ctl = reinterpret_cast<ResCtl*>(smem);
    const uint32_t base = smem_u32(smem);
    const uint32_t abuf = base + p.a_off, ring = base + p.ring_off;
    volatile uint32_t* abort_flag = &ctl->abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t NS = static_cast<uint32_t>(p.num_stages);
    const int nt = static_cast<int>(blockIdx.x) < p.tiles ? (p.tiles - static_cast<int>(blockIdx.x) + static_cast<int>(gridDim.x) - 1) / static_cast<int>(gridDim.x) : 0;

    if (threadIdx.x == 0) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&ctl->a_full[b]), 1);
            mbar_init(smem_u32(&ctl->a_empty[b]), 1);
            mbar_init(smem_u32(&ctl->t_full[b]), 1);
            mbar_init(smem_u32(&ctl->acc_full[b]), 1);
            mbar_init(smem_u32(&ctl->acc_empty[b]), 4);
        }
        for (uint32_t s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&ctl->full[s]), 1);
            mbar_init(smem_u32(&ctl->empty[s]), 1);
        }
        mbar_init(smem_u32(&ctl->t_ready), 8);
        ctl->abort = 0;
        fence_barrier_init();
        fence_proxy_async_smem();
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB1);
        tma_prefetch_desc(&tmB2);
    }
    if (warp == 1) tmem_alloc(smem_u32(&ctl->tmem_base), 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_wait();
    pdl_launch_dependents();
    const uint32_t tmem = ctl->tmem_base;
    const FlatImage& f = p.f;
    // first box of a tile's window, and the window's row of the tile's first position
    auto first_unit = [&](int q0) { return floor_div(q0 - f.Wp - 1, f.unit_rows); };

    if (warp == 0) {
        if (elect_one()) {
            uint32_t b = 0, ph = 1;
            bool ok = true;
            for (int i = 0; i < nt && ok; ++i) {
                const int q0 = (static_cast<int>(blockIdx.x) + i * static_cast<int>(gridDim.x)) * kResRows;
                const int u0 = first_unit(q0), count = floor_div(q0 + kResRows + f.Wp, f.unit_rows) - u0 + 1;
                for (int cb = 0; cb < p.cblks; ++cb) {
                    ok = mbar_wait(smem_u32(&ctl->a_empty[b]), ph, abort_flag, p.status);
                    if (!ok) break;
                    const uint32_t full = smem_u32(&ctl->a_full[b]);
                    mbar_expect_tx(full, static_cast<uint32_t>(count * f.unit_rows) * 128u);
                    load_window(f, &tmA, abuf + b * p.a_bytes, full, u0, count, cb * 64);
                    b ^= 1u;
                    if (b == 0) ph ^= 1u;
                }
            }
        }
    } else if (warp == 10) {
        if (elect_one()) {
            uint32_t s = 0, ph = 1;
            bool ok = true;
            auto slot = [&](auto&& issue) {
                ok = mbar_wait(smem_u32(&ctl->empty[s]), ph, abort_flag, p.status);
                if (!ok) return;
                const uint32_t full = smem_u32(&ctl->full[s]);
                mbar_expect_tx(full, kStage);
                issue(ring + s * kStage, full);
                if (++s == NS) { s = 0; ph ^= 1u; }
            };
            for (int t = 0; t <= nt && ok; ++t) {
                if (t < nt)
                    for (int cb = 0; cb < p.cblks && ok; ++cb)
                        for (int tap = 0; tap < 9 && ok; ++tap)
                            slot([&](uint32_t dst, uint32_t full) {
                                if (p.ragged) tma_load_3d(dst, &tmB1, full, 0, cb * 64, tap);
                                else tma_load_2d(dst, &tmB1, full, 0, tap * p.C + cb * 64);
                            });
                if (t >= 1)
                    for (int h = 0; h < 2 * p.nblk && ok; ++h)
                        slot([&](uint32_t dst, uint32_t full) { tma_load_2d(dst, &tmB2, full, 0, h * 64); });
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            uint32_t s = 0, ph = 0, b = 0, bph = 0;
            uint32_t use = 0;                       // accumulator uses so far
            bool ok = true;
            // the nine taps of one window buffer, into d0 (first row tile) and d1
            const uint64_t b_desc = make_smem_desc(ring, 8192, 1024);
            const uint32_t a_hi = desc_hi(make_smem_desc(abuf, 16, 1024)), b_hi = desc_hi(b_desc), b_lo = desc_lo(b_desc);
            const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
            auto taps = [&](uint32_t buf, int row0, uint32_t d0, uint32_t d1, uint32_t idesc, bool fresh) {
                const uint32_t a0 = desc_lo(make_smem_desc(abuf + buf * p.a_bytes, 16, 1024)) + static_cast<uint32_t>(row0) * 8u;
                int o = -f.Wp - 1;                       // tap (0, 0)
                for (int tap = 0; tap < 9; ++tap) {
                    ok = mbar_wait(full0 + 8 * s, ph, abort_flag, p.status);
                    if (!ok) return;
                    tc_fence_after();
                    const uint32_t a = a0 + static_cast<uint32_t>(o * 8), bd = b_lo + s * (kStage >> 4);
                    const uint32_t acc = (fresh && tap == 0) ? 0u : 1u;
#pragma unroll
                    for (int m = 0; m < 2; ++m) {
                        const uint32_t d = m ? d1 : d0;
                        const uint32_t am = a + m * 128u * 8u;
                        tc_mma_bf16_words(d, am, a_hi, bd, b_hi, idesc, acc);
                        tc_mma_bf16_words(d, am + 2, a_hi, bd + 128, b_hi, idesc, 1u);
                        tc_mma_bf16_words(d, am + 4, a_hi, bd + 256, b_hi, idesc, 1u);
                        tc_mma_bf16_words(d, am + 6, a_hi, bd + 384, b_hi, idesc, 1u);
                    }
                    tc_commit(empty0 + 8 * s);
                    if (++s == NS) { s = 0; ph ^= 1u; }
                    o += tap == 2 || tap == 5 ? f.Wp - 2 : 1;
                }
            };
            const uint32_t idesc1 = make_idesc_bf16(128, 64, 0, 1), idesc2 = make_idesc_bf16(128, 64, 0, 0);
            const uint64_t t_desc = make_smem_desc(base + p.t_off, 16, 1024);
            for (int t = 0; t <= nt && ok; ++t) {
                if (t < nt) {
                    const int q0 = (static_cast<int>(blockIdx.x) + t * static_cast<int>(gridDim.x)) * kResRows;
                    const int row0 = q0 - first_unit(q0) * f.unit_rows;
                    const uint32_t d = tmem + static_cast<uint32_t>(t & 1) * 128u;
                    for (int cb = 0; cb < p.cblks && ok; ++cb) {
                        ok = mbar_wait(smem_u32(&ctl->a_full[b]), bph, abort_flag, p.status);
                        if (!ok) break;
                        taps(b, row0, d, d + 64, idesc1, cb == 0);
                        if (!ok) break;
                        tc_commit(smem_u32(&ctl->a_empty[b]));
                        b ^= 1u;
                        if (b == 0) bph ^= 1u;
                    }
                    if (!ok) break;
                    tc_commit(smem_u32(&ctl->t_full[t & 1]));
                }
                if (t >= 1) {
                    const int u = t - 1;
                    ok = mbar_wait(smem_u32(&ctl->t_ready), static_cast<uint32_t>(u) & 1u, abort_flag, p.status);
                    if (!ok) break;
                    tc_fence_after();
                    for (int j = 0; j < p.nblk && ok; ++j, ++use) {
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            ok = mbar_wait(smem_u32(&ctl->full[s]), ph, abort_flag, p.status);
                            if (!ok) break;
                            const uint64_t bd = make_smem_desc(ring + s * kStage, 16, 1024);
                            for (int m = 0; m < 2; ++m) {
                                if (h == 0) ok = ok && mbar_wait(smem_u32(&ctl->acc_empty[m]), (use & 1u) ^ 1u, abort_flag, p.status);
                                tc_fence_after();
                                const uint32_t d = tmem + 256u + m * 128u + h * 64u;
                                const uint64_t am = t_desc + m * 1024u;
                                tc_mma_bf16(d, am, bd, idesc2, 0u);
                                tc_mma_bf16(d, am + 2, bd + 2, idesc2, 1u);
                                tc_mma_bf16(d, am + 4, bd + 4, idesc2, 1u);
                                tc_mma_bf16(d, am + 6, bd + 6, idesc2, 1u);
                            }
                            if (!ok) break;
                            tc_commit(smem_u32(&ctl->empty[s]));
                            if (++s == NS) { s = 0; ph ^= 1u; }
                        }
                        if (!ok) break;
                        tc_commit(smem_u32(&ctl->acc_full[0]));
                        tc_commit(smem_u32(&ctl->acc_full[1]));
                    }
                }
            }
        }
    } else {
        const int m = (warp - 2) >> 2, q4 = warp & 3;
        const uint32_t lanes = tmem + (static_cast<uint32_t>(q4 * 32) << 16);
        const uint32_t panel = base + p.stg_off + static_cast<uint32_t>(warp - 2) * 4096u;
        auto pixel = [&](int i) {
            return pixel_of(f, (static_cast<int>(blockIdx.x) + i * static_cast<int>(gridDim.x)) * kResRows + m * 128 + q4 * 32 + lane);
        };
        uint32_t use = 0;
        bool ok = true;
        const uint32_t t_rows = base + p.t_off + static_cast<uint32_t>(m) * 16384u + static_cast<uint32_t>(q4 * 32) * 128u;
        int pix = -1;
        for (int t = 0; t <= nt && ok; ++t) {
            if (t >= 1) {
                for (int j = 0; j < p.nblk; ++j, ++use) {
                    ok = mbar_wait_warp(smem_u32(&ctl->acc_full[m]), use & 1u, abort_flag, p.status);
                    tc_fence_after();
                    if (!ok) break;
                    store_block(lanes + 256 + m * 128, panel, lane, pix, p.out, p.Nout, j * 128, p.Nout, &ctl->acc_empty[m]);
                }
            }
            if (t < nt && ok) {
                // T(t): the second product of t - 1 has read T's buffer (its last accumulator was complete above)
                ok = mbar_wait_warp(smem_u32(&ctl->t_full[t & 1]), static_cast<uint32_t>(t >> 1) & 1u, abort_flag, p.status);
                tc_fence_after();
                if (!ok) break;
                uint32_t v0[32], v1[32];
                const uint32_t acc = lanes + static_cast<uint32_t>(t & 1) * 128u + static_cast<uint32_t>(m) * 64u;
                tmem_ld32(acc, v0);
                tmem_ld32(acc + 32, v1);
                tmem_ld_wait();
                const uint32_t own = t_rows + static_cast<uint32_t>(lane) * 128u;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const uint32_t* v = e < 4 ? v0 + 8 * e : v1 + 8 * (e - 4);
                    st_shared_v4(own + ((static_cast<uint32_t>(e) ^ static_cast<uint32_t>(lane & 7)) << 4),
                                 make_uint4(pack_bf16x2(__uint_as_float(v[0]), __uint_as_float(v[1])), pack_bf16x2(__uint_as_float(v[2]), __uint_as_float(v[3])),
                                            pack_bf16x2(__uint_as_float(v[4]), __uint_as_float(v[5])), pack_bf16x2(__uint_as_float(v[6]), __uint_as_float(v[7]))));
                }
                tc_fence_before();
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&ctl->t_ready));
                pix = pixel(t);
                if (p.T) {
                    const int sub = lane >> 3, piece = lane & 7;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int rr = i * 4 + sub;
                        const int px = __shfl_sync(0xffffffffu, pix, rr);
                        const uint4 w = ld_shared_v4(t_rows + static_cast<uint32_t>(rr) * 128u + ((static_cast<uint32_t>(piece) ^ static_cast<uint32_t>(rr & 7)) << 4));
                        if (px >= 0 && piece * 8 < p.R) *reinterpret_cast<uint4*>(p.T + static_cast<size_t>(px) * p.R + piece * 8) = w;
                    }
                }
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

// ------------------------------------------------------------------------------ host
bool res_shape(const ConvArgs& a) {
    return a.kh == 3 && a.kw == 3 && a.stride == 1 && a.pad == 1 && a.R <= 64 && a.R % 8 == 0 && a.C % 8 == 0 && a.O % 8 == 0 && a.W <= 128 &&
           static_cast<int64_t>(a.N) * (a.H + 1) * (a.W + 1) < (1 << 30) && static_cast<int64_t>(9) * a.C < (1 << 24) && encode_fn() != nullptr;
}
struct ResLayout {
    uint32_t a_bytes, a_off, t_off, stg_off, ring_off;
    int stages;
    size_t smem;
};
bool res_layout(const FlatImage& f, ResLayout* l) {
    const uint32_t stage = 8192, limit = 226 * 1024;
    l->a_bytes = static_cast<uint32_t>(align_up(static_cast<size_t>(window_rows(f, kResRows + 2 * f.Wp + 2)) * 128, 1024));
    uint32_t off = 1024;
    l->a_off = off; off += 2 * l->a_bytes;
    l->t_off = off; off += 32768;
    l->stg_off = off; off += 32768;
    l->ring_off = off;
    if (off + 3 * stage > limit) return false;
    l->stages = std::min<int>(kResMaxStages, static_cast<int>((limit - off) / stage));
    l->smem = off + static_cast<size_t>(l->stages) * stage + 1024;
    return true;
}
void fill(ResParams* p, const FlatImage& f, const ResLayout& l, const ConvArgs& a) {
    p->f = f;
    p->tiles = static_cast<int>(ceil_div(static_cast<int64_t>(f.N) * f.Hp * f.Wp, kResRows));
    p->C = a.C; p->R = a.R;
    p->ragged = a.C % 64 != 0;
    p->a_bytes = l.a_bytes; p->a_off = l.a_off; p->t_off = l.t_off; p->ring_off = l.ring_off; p->stg_off = l.stg_off;
    p->num_stages = l.stages;
    p->status = device_status_ptr();
}
}  // namespace

int conv_res_fwd(const ConvArgs& a, int64_t ldf, const Before& before) {
    if (!res_shape(a)) return PF_ERR_UNSUPPORTED;
    const FlatImage f = flat_image(a.N, a.H, a.W);
    ResLayout l;
    if (!res_layout(f, &l)) return PF_ERR_UNSUPPORTED;
    // Per 64 channels a tile of 256 positions takes 3.05 us here, a tile of up to 128 pixels in the kernel that fetches
    // them per tap 1.86 us while the grid fits one wave and 2.2 beyond; the coarser tiles lose where there are few.
    const int64_t rounds = ceil_div(ceil_div(static_cast<int64_t>(f.N) * f.Hp * f.Wp, kResRows), num_sms());
    const int64_t other = ceil_div(conv_tiling(a.N, a.Ho, a.Wo, 128).blocks, num_sms());
    if (3.05 * static_cast<double>(rounds) >= (other > 1 ? 2.2 : 1.86) * static_cast<double>(other)) return PF_ERR_UNSUPPORTED;
    ResParams p = {};
    fill(&p, f, l, a);
    p.cblks = static_cast<int>(ceil_div(a.C, 64));
    p.nblk = static_cast<int>(ceil_div(a.O, 128));
    p.Nout = a.O;
    p.out = static_cast<__nv_bfloat16*>(a.y);
    p.T = static_cast<__nv_bfloat16*>(a.T);
    CUtensorMap ta, tb1, tb2;
    const bool ok = window_map(&ta, f, a.x, a.C) &&
                    (p.ragged ? cached_map_planes(&tb1, a.U, 9, a.C, a.R, a.C, 64, ldf) : cached_map_2d(&tb1, a.U, static_cast<int64_t>(9) * a.C, a.R, ldf, 64)) &&
                    cached_map_2d(&tb2, a.V, a.O, a.R, ldf, 64);
    if (!ok || allow_smem(tc_conv_res_kernel, 227 * 1024) != cudaSuccess) return PF_ERR_CUDA;
    const int st = before();
    if (st != PF_OK) return st;
    if (launch_overlapped(tc_conv_res_kernel, dim3(static_cast<unsigned>(even_grid(p.tiles))), dim3(kResThreads), l.smem, a.stream, ta, tb1, tb2, p) != cudaSuccess)
        return PF_ERR_CUDA;
    count_launch();
    return PF_OK;
}

}  // namespace tc
}  // namespace pf
