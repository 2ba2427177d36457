// fp32 layers on the tensor cores: host side of the kernel in pf_tc_f32_kernel.cuh.  Forward: T = x U (or the thin
// convolution), then y = T V^T with the bias / activation epilogue.  Backward: G = dY V beside dV = dY^T T, then
// dU = x^T G beside dX = G U^T.  Contractions that are long for the number of tiles are cut into slices.
#include "pf_tc.h"

#include <cuda.h>

#include <algorithm>

#include "pf_tc_f32_kernel.cuh"
#include "pf_tc_host.h"

namespace pf {
namespace tc {
namespace {

int64_t f32_pitch(int64_t v, bool tight = false) { return v > 16 && !tight ? (v + 31) / 32 * 32 : (v + 3) / 4 * 4; }      // whole 128-byte lines, as row_pitch
bool f32_tma_ok(const void* p, int64_t ld) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && ld % 4 == 0 && ld * 4 < (1LL << 40); }

// fp32 tensor maps with boxes of 32 columns (128 bytes): rank 2 = [rows, cols], rank 3 = [planes][rows][cols]
// (contiguous), rank 4 = NHWC image (see cached_map_nhwc).
bool f32_encode(EncodeTiledFn fn, CUtensorMap* map, const void* p, int rank, const cuuint64_t* dims, const cuuint64_t* strides,
                const cuuint32_t* box, const cuuint32_t* estr) {
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, static_cast<cuuint32_t>(rank), const_cast<void*>(p), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
bool f32_map_2d(CUtensorMap* map, const void* p, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
    return cached_map(map, MapKey{p, {rows, cols, ld, box_rows, -2, -4, -4, -4}}, [&](EncodeTiledFn fn) {
        const cuuint64_t dims[2] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows)};
        const cuuint64_t strides[1] = {static_cast<cuuint64_t>(ld) * 4};
        const cuuint32_t box[2] = {32u, static_cast<cuuint32_t>(box_rows)}, estr[2] = {1u, 1u};
        return f32_encode(fn, map, p, 2, dims, strides, box, estr);
    });
}
bool f32_map_planes(CUtensorMap* map, const void* p, int64_t planes, int64_t rows, int64_t cols, int box_rows) {
    return cached_map(map, MapKey{p, {planes, rows, cols, box_rows, -3, -4, -4, -4}}, [&](EncodeTiledFn fn) {
        const cuuint64_t dims[3] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows), static_cast<cuuint64_t>(planes)};
        const cuuint64_t strides[2] = {static_cast<cuuint64_t>(cols) * 4, static_cast<cuuint64_t>(rows) * cols * 4};
        const cuuint32_t box[3] = {32u, static_cast<cuuint32_t>(box_rows), 1u}, estr[3] = {1u, 1u, 1u};
        return f32_encode(fn, map, p, 3, dims, strides, box, estr);
    });
}
bool f32_map_nhwc(CUtensorMap* map, const void* p, int64_t N, int64_t H, int64_t W, int64_t C, int box_w, int box_h, int box_n, int stride) {
    return cached_map(map, MapKey{p, {N, H * 4096 + W, C, box_w, box_h, box_n, stride, -5}}, [&](EncodeTiledFn fn) {
        const cuuint64_t dims[4] = {static_cast<cuuint64_t>(C), static_cast<cuuint64_t>(W), static_cast<cuuint64_t>(H), static_cast<cuuint64_t>(N)};
        const cuuint64_t strides[3] = {static_cast<cuuint64_t>(C) * 4, static_cast<cuuint64_t>(W) * C * 4, static_cast<cuuint64_t>(H) * W * C * 4};
        const cuuint32_t box[4] = {32u, static_cast<cuuint32_t>(box_w * stride), static_cast<cuuint32_t>(box_h * stride),
                                   static_cast<cuuint32_t>(box_n)};
        const cuuint32_t estr[4] = {1u, static_cast<cuuint32_t>(stride), static_cast<cuuint32_t>(stride), 1u};
        return f32_encode(fn, map, p, 4, dims, strides, box, estr);
    });
}

struct F32Op {
    const void* p;
    int64_t ld;
    bool mn;                 // stored [K, MN] (the M / N index contiguous)
    bool early = false;      // see kEarlyA in pf_tc_prims.cuh
};
struct F32Conv {
    int mode = 0;            // as F32Params::mode
    int N = 0, H = 0, W = 0, C = 0, R = 0, Ho = 0, Wo = 0, kh = 0, kw = 0, pad = 0, stride = 1;
};
// One product of a launch: sizes and geometry (plan), then tensor maps and addresses (prepare).
struct F32Work {
    int64_t M = 0, N = 0, K = 0;
    F32Conv cv;
    ConvTiling ct;           // blocks of pixels: rows of a tile (modes 1, 3) or of a k-block (mode 2)
    int wblk = 1, bw = 0;    // mode 2: blocks per image row and their width
    int64_t tiles_x = 0, tiles_y = 0, nkb = 0;
    int bn = 0, splits = 1;
    int64_t tiles() const { return tiles_x * tiles_y; }
    size_t partial_bytes() const { return splits > 1 ? align_up(static_cast<size_t>(tiles()) * splits * 128 * bn * 4, 256) : 0; }
};

// Blocks of at most 32 output pixels for the contraction of dU: an image row is cut into equal parts when it is longer.
void du_blocks(F32Work* w) {
    const F32Conv& c = w->cv;
    w->wblk = static_cast<int>(ceil_div(c.Wo, 32));
    w->bw = static_cast<int>(ceil_div(c.Wo, w->wblk));
    if (w->wblk == 1) {
        w->ct = conv_tiling(c.N, c.Ho, c.Wo, 32);
    } else {
        w->ct.nb = 1; w->ct.bh = 1; w->ct.tpi = c.Ho; w->ct.pixels = w->bw;
        w->ct.blocks = static_cast<int64_t>(c.N) * c.Ho;
    }
}
void f32_tiles(F32Work* w, int bn) {
    w->bn = bn;
    w->tiles_y = ceil_div(w->N, bn);
}
F32Work f32_work(int64_t M, int64_t N, int64_t K, const F32Conv* cv = nullptr) {
    F32Work w;
    w.M = M; w.N = N; w.K = K;
    w.tiles_x = ceil_div(M, 128);
    w.nkb = ceil_div(K, 32);
    if (cv) {
        w.cv = *cv;
        const int taps = cv->kh * cv->kw;
        if (cv->mode == 2) {
            du_blocks(&w);
            w.tiles_x = ceil_div(static_cast<int64_t>(taps) * ceil_div(cv->C, 32), 4);
            w.nkb = w.ct.blocks * w.wblk;
        } else if (cv->mode == 1) {
            w.ct = conv_tiling(cv->N, static_cast<int>(ceil_div(cv->H, cv->stride)), static_cast<int>(ceil_div(cv->W, cv->stride)), 128);
            w.tiles_x = w.ct.blocks * cv->stride * cv->stride;
            w.nkb = static_cast<int64_t>(taps) * ceil_div(cv->R, 32);
        } else {
            // (a box spans stride input rows per output row, and TMA boxes are at most 256 high)
            w.ct = conv_tiling(cv->N, cv->Ho, cv->Wo, std::min(128, 256 / cv->stride * cv->Wo));
            w.tiles_x = w.ct.blocks;
            w.nkb = static_cast<int64_t>(taps) * ceil_div(cv->C, 32);
        }
    }
    // narrow tiles where 128-column ones would leave half of the machine idle (f32_split looks at both)
    f32_tiles(&w, (N <= 64 || w.tiles_x * ceil_div(N, 128) * 2 <= num_sms()) ? 64 : 128);
    return w;
}
// Slice counts of the products of one launch (`can` = which may be split): every block should carry about the same
// number of k-blocks and all of them fit the machine at once.  A slice sum costs about as much as 12 k-blocks
// (5 us of L2 round trips), so contractions shorter than that stay whole.
void f32_slices(F32Work* const* w, const bool* can, int count) {
    int64_t work = 0, longest = 0;
    for (int i = 0; i < count; ++i) {
        work += w[i]->tiles() * w[i]->nkb;
        longest = std::max(longest, w[i]->nkb);
        w[i]->splits = 1;
    }
    for (int64_t target = std::max<int64_t>(4, ceil_div(work, num_sms())); target < longest; target += 1 + target / 16) {
        int64_t split_blocks = 0;
        for (int i = 0; i < count; ++i) {
            int64_t s = can[i] && w[i]->nkb > 12 ? ceil_div(w[i]->nkb, target) : 1;
            if (s > 64) s = 64;
            s = ceil_div(w[i]->nkb, ceil_div(w[i]->nkb, s));       // every slice gets k-blocks
            w[i]->splits = static_cast<int>(s);
            if (s > 1) split_blocks += w[i]->tiles() * s;
        }
        if (split_blocks <= num_sms()) return;
    }
    for (int i = 0; i < count; ++i) w[i]->splits = 1;
}

// Expected microseconds of the launch: 5 of start and end, a k-block of a 128-column tile 0.95 and of a 64-column one 0.67,
// 5 for a sum of slices; one block per SM at a time.
double f32_us(F32Work* const* w, int count) {
    double blocks = 0, load = 0, longest = 0;
    for (int i = 0; i < count; ++i) {
        const double n = static_cast<double>(w[i]->tiles() * w[i]->splits);
        const double us = 5.0 + (w[i]->bn == 64 ? 0.67 : 0.95) * static_cast<double>(ceil_div(w[i]->nkb, w[i]->splits)) + (w[i]->splits > 1 ? 5.0 : 0.0);
        blocks += n;
        load += n * us;
        longest = std::max(longest, us);
    }
    return blocks <= num_sms() ? longest : count == 1 ? longest * static_cast<double>(ceil_div(static_cast<int64_t>(blocks), num_sms()))
                                                      : std::max(longest, 1.1 * load / num_sms());
}
// Slices, and the widths of the tiles: 128 columns do in one k-block of 0.95 us what two 64-column tiles do in 1.34, so long
// contractions are better cut into more slices of wide tiles: backward of 2048 x 512 -> 128 -> 2048: 45.7 -> 37.3 us, of 1000 x 1024 ->
// 256 -> 1024: 43.1 -> 31.9; forward of 2048 x 2048 -> 128 -> 512: 26.1 -> 23.3.
// tight: less room, not less time (the slices of wide tiles take up to twice the bytes).
void f32_split(F32Work* const* w, const bool* can, int count, bool tight = false) {
    f32_slices(w, can, count);
    if (tight) return;
    F32Work wide[2];
    F32Work* pw[2] = {&wide[0], &wide[1]};
    bool other = false;
    for (int i = 0; i < count; ++i) {
        wide[i] = *w[i];
        if (w[i]->bn == 64 && w[i]->N > 64) {
            f32_tiles(&wide[i], 128);
            other = true;
        }
    }
    if (!other) return;
    f32_slices(pw, can, count);
    if (f32_us(pw, count) < f32_us(w, count))
        for (int i = 0; i < count; ++i) *w[i] = wide[i];
}

size_t f32_smem(int bn, int stages) { return 2048 + 3 * static_cast<size_t>(bn) * 128 + static_cast<size_t>(stages) * (16384 + static_cast<size_t>(bn) * 128); }
int f32_stages(int bn) { return bn == 64 ? 8 : 5; }

bool f32_prepare(const F32Work& w, const F32Op& A, const F32Op& B, float* C, int64_t ldc, float* partial, CUtensorMap* ta, CUtensorMap* tb,
                 F32Params* p) {
    const F32Conv& c = w.cv;
    bool ok = true;
    *p = F32Params();
    if (c.mode == 0) {
        ok = A.mn ? f32_map_2d(ta, A.p, w.K, w.M, A.ld, 32) : f32_map_2d(ta, A.p, w.M, w.K, A.ld, 128);
        ok = ok && (B.mn ? f32_map_2d(tb, B.p, w.K, w.N, B.ld, 32) : f32_map_2d(tb, B.p, w.N, w.K, B.ld, w.bn));
    } else if (c.mode == 1) {            // A = dT, B = U as (taps * C) x R
        ok = f32_map_nhwc(ta, A.p, c.N, c.Ho, c.Wo, c.R, static_cast<int>(ceil_div(c.W, c.stride)), w.ct.bh, w.ct.nb, 1) &&
             f32_map_2d(tb, B.p, static_cast<int64_t>(c.kh) * c.kw * c.C, c.R, c.R, w.bn);
    } else if (c.mode == 2) {            // A = x, B = dT
        ok = f32_map_nhwc(ta, A.p, c.N, c.H, c.W, c.C, w.bw, w.ct.bh, w.ct.nb, c.stride) &&
             f32_map_nhwc(tb, B.p, c.N, c.Ho, c.Wo, c.R, w.bw, w.ct.bh, w.ct.nb, 1);
    } else {                             // A = x, B = U
        ok = f32_map_nhwc(ta, A.p, c.N, c.H, c.W, c.C, c.Wo, w.ct.bh, w.ct.nb, c.stride);
        ok = ok && (c.C % 32 ? f32_map_planes(tb, B.p, static_cast<int64_t>(c.kh) * c.kw, c.C, c.R, 32)
                             : f32_map_2d(tb, B.p, static_cast<int64_t>(c.kh) * c.kw * c.C, c.R, c.R, 32));
    }
    if (!ok) return false;
    p->M = static_cast<int>(w.M); p->N = static_cast<int>(w.N);
    p->a_mn = A.mn; p->b_mn = B.mn;
    p->bn = w.bn;
    p->nkb = static_cast<int>(w.nkb);
    p->kb_per_split = static_cast<int>(ceil_div(w.nkb, w.splits));
    p->splits = w.splits;
    p->num_stages = f32_stages(w.bn);
    p->mode = c.mode;
    p->tiles_x = static_cast<int>(w.tiles_x); p->tiles_y = static_cast<int>(w.tiles_y);
    p->A = static_cast<const float*>(A.p); p->B = static_cast<const float*>(B.p);
    p->lda = A.ld; p->ldb = B.ld;
    p->K = static_cast<int>(w.K);
    p->cv_H = c.mode == 1 ? c.Ho : c.H; p->cv_W = c.mode == 1 ? c.Wo : c.W; p->cv_R = c.R;
    p->C = C; p->ldc = ldc;
    p->partial = partial;
    p->counters = w.splits > 1 ? split_counters() : nullptr;
    if (w.splits > 1 && !p->counters) return false;
    p->status = device_status_ptr();
    p->cv_blks = static_cast<int>(ceil_div(c.mode == 1 ? c.R : c.C, 32));
    p->cv_kw = c.kw; p->cv_kh = c.kh; p->cv_pad = c.pad; p->cv_stride = c.stride; p->cv_C = c.C;
    p->cv_bh = w.ct.bh; p->cv_nb = w.ct.nb; p->cv_tpi = w.ct.tpi; p->cv_N = c.N;
    p->cv_bw = c.mode == 1 ? static_cast<int>(ceil_div(c.W, c.stride)) : c.mode == 2 ? w.bw : std::max(1, c.Wo);
    p->cv_inv_bw = 65535 / p->cv_bw + 1;
    p->cv_inv_bh = 65535 / std::max(1, w.ct.bh) + 1;
    p->cv_tiles_class = static_cast<int>(std::max<int64_t>(1, w.ct.blocks));
    p->out_h = c.mode == 1 ? c.H : c.Ho;
    p->out_w = c.mode == 1 ? c.W : c.Wo;
    p->step = c.mode == 1 ? c.stride : 1;
    p->cv_blocks = c.kh * c.kw * p->cv_blks;
    p->cv_wblk = w.wblk;
    p->rows_tile = w.ct.pixels;
    p->kpix = w.ct.pixels;
    p->ragged = c.C % 32 != 0;
    p->early = (A.early ? kEarlyA : 0) | (B.early ? kEarlyB : 0);
    return true;
}

// Split products first: their blocks wait for one another and must be resident together.
int f32_launch(F32Launch* a, int count, cudaStream_t stream) {
    if (count == 2 && a->p[0].splits <= 1 && a->p[1].splits > 1) {
        std::swap(a->ta[0], a->ta[1]);
        std::swap(a->tb[0], a->tb[1]);
        std::swap(a->p[0], a->p[1]);
    }
    size_t smem = 0;
    int total = 0;
    bool conv = false;
    for (int i = 0; i < 3; ++i) {
        if (i < count) {
            total += a->p[i].tiles_x * a->p[i].tiles_y * a->p[i].splits;
            smem = std::max(smem, f32_smem(a->p[i].bn, a->p[i].num_stages));
            conv = conv || a->p[i].mode != 0;
        } else {
            a->ta[i] = a->ta[0]; a->tb[i] = a->tb[0]; a->p[i] = a->p[0];
        }
        a->end[i] = total;
    }
    cudaError_t e;
    if (conv) {
        e = launch_f32_conv(total, smem, stream, *a);
    } else {
        e = allow_smem(tc_f32_kernel<false>, 227 * 1024);
        if (e == cudaSuccess) e = launch_overlapped(tc_f32_kernel<false>, dim3(static_cast<unsigned>(total)), dim3(kF32Threads), smem, stream, *a);
    }
    if (e != cudaSuccess) return PF_ERR_CUDA;
    count_launch();
    return PF_OK;
}

// A matrix that TMA must read: as it is, or (ragged widths) copied to scratch at a pitch of whole 16-byte pieces.  The
// copy kernel moves 2-byte units.
struct Staged32 {
    const void* p;
    int64_t ld;
};
bool f32_stage(const void* p, int64_t ld, int64_t rows, int64_t cols, char*& scratch, Staged32* out, RepackJob* jobs, int* count, bool tight = false) {
    *out = Staged32{p, ld};
    if (f32_tma_ok(p, ld)) return true;
    if (cols % 4 == 0) return false;      // the workspace query reserves repack room only for ragged widths
    const int64_t ldp = f32_pitch(cols, tight);
    jobs[(*count)++] = RepackJob{p, 2 * ld, scratch, 2 * ldp, rows, 2 * cols};
    *out = Staged32{scratch, ldp};
    scratch += align_up(static_cast<size_t>(rows) * ldp * 4, 256);
    return true;
}
size_t f32_mat(int64_t rows, int64_t cols, bool tight = false) { return align_up(static_cast<size_t>(rows) * f32_pitch(cols, tight) * 4, 256); }
size_t f32_room(int64_t rows, int64_t cols, bool tight = false) { return cols % 4 == 0 ? 0 : f32_mat(rows, cols, tight); }

// The products of the two layers in the order they are launched, planned from the sizes alone.
struct F32Fwd {
    F32Work t, y;
};
F32Fwd f32_plan_fwd(const F32Work& t, const F32Work& y, bool tight = false) {
    F32Fwd f{t, y};
    F32Work* w = &f.t;
    const bool can = true;
    f32_split(&w, &can, 1, tight);
    return f;
}
struct F32Bwd {
    F32Work t, g, dv, du, dx;
};
F32Bwd f32_plan_bwd(const F32Work& t, const F32Work& g, const F32Work& dv, const F32Work& du, const F32Work& dx) {
    F32Bwd b{t, g, dv, du, dx};
    const bool can[2] = {true, true}, first[2] = {true, false};
    F32Work *wt = &b.t, *wa[2] = {&b.g, &b.dv}, *wb[2] = {&b.du, &b.dx};
    f32_split(&wt, can, 1);
    f32_split(wa, can, 2);
    f32_split(wb, first, 2);
    return b;
}
F32Fwd linear_plan_fwd(int64_t m, int64_t k, int64_t n, int64_t r, bool tight) { return f32_plan_fwd(f32_work(m, r, k), f32_work(m, n, r), tight); }
F32Bwd linear_plan_bwd(int64_t m, int64_t k, int64_t n, int64_t r) {
    return f32_plan_bwd(f32_work(m, r, k), f32_work(m, r, n), f32_work(n, r, m), f32_work(k, r, m), f32_work(m, k, r));
}
F32Conv f32_conv(const ConvArgs& a, int mode) {
    F32Conv c;
    c.mode = mode; c.N = a.N; c.H = a.H; c.W = a.W; c.C = a.C; c.R = a.R; c.Ho = a.Ho; c.Wo = a.Wo; c.kh = a.kh; c.kw = a.kw; c.pad = a.pad;
    c.stride = a.stride;
    return c;
}
F32Fwd conv_plan_fwd(const ConvArgs& a) {
    const int64_t P = static_cast<int64_t>(a.N) * a.Ho * a.Wo;
    const F32Conv c = f32_conv(a, 3);
    return f32_plan_fwd(f32_work(P, a.R, 0, &c), f32_work(P, a.O, a.R));
}
F32Bwd conv_plan_bwd(const ConvArgs& a) {
    const int64_t P = static_cast<int64_t>(a.N) * a.Ho * a.Wo, Keff = static_cast<int64_t>(a.kh) * a.kw * a.C;
    const F32Conv c3 = f32_conv(a, 3), c2 = f32_conv(a, 2), c1 = f32_conv(a, 1);
    return f32_plan_bwd(f32_work(P, a.R, 0, &c3), f32_work(P, a.R, a.O), f32_work(a.O, a.R, P), f32_work(Keff, a.R, 0, &c2),
                        f32_work(static_cast<int64_t>(a.N) * a.H * a.W, a.C, 0, &c1));
}

bool sizes_ok(int64_t m, int64_t k, int64_t n, int64_t r) {
    return m <= (1 << 30) && k <= (1 << 22) && n <= (1 << 22) && r <= (1 << 20) && m * std::max({k, n, r}) < (1LL << 38);
}
bool tiles_ok(const F32Work& w) { return w.tiles() * w.splits < (1LL << 30) && w.nkb < (1LL << 28); }
}  // namespace

size_t f32_linear_workspace(int64_t m, int64_t k, int64_t n, int64_t r, bool bwd, bool tight) {
    if (!sizes_ok(m, k, n, r) || m < 1) return 0;
    size_t b = f32_room(m, k, tight) + f32_room(k, r, tight) + f32_room(n, r, tight) + f32_mat(m, r, tight);      // x, U, V, T
    if (!bwd) return b + linear_plan_fwd(m, k, n, r, tight).t.partial_bytes();
    const F32Bwd p = linear_plan_bwd(m, k, n, r);
    return b + f32_room(m, n) + f32_mat(m, r) + std::max(p.t.partial_bytes(), p.g.partial_bytes()) + p.dv.partial_bytes() + p.du.partial_bytes();
}

int f32_linear_fwd(const LinearArgs& a, int* handled, size_t room) {
    *handled = 0;
    if (encode_fn() == nullptr || !sizes_ok(a.m, a.k, a.n, a.r) || f32_linear_workspace(a.m, a.k, a.n, a.r, false, a.tight) > room) return PF_OK;
    const F32Fwd f = linear_plan_fwd(a.m, a.k, a.n, a.r, a.tight);
    if (!tiles_ok(f.t) || !tiles_ok(f.y)) return PF_OK;
    char* ws = a.ws;
    Staged32 x, U, V;
    RepackJob jobs[3];
    int nj = 0;
    if (!f32_stage(a.x, a.ldx, a.m, a.k, ws, &x, jobs, &nj, a.tight) || !f32_stage(a.U, a.ldu, a.k, a.r, ws, &U, jobs, &nj, a.tight) ||
        !f32_stage(a.V, a.ldv, a.n, a.r, ws, &V, jobs, &nj, a.tight))
        return PF_OK;
    // T: the stash itself when TMA can read it back, else scratch; the first product then writes the stash beside it
    const bool direct = a.T && f32_tma_ok(a.T, a.ldt);
    float* T = direct ? static_cast<float*>(a.T) : reinterpret_cast<float*>(ws);
    const int64_t ldT = direct ? a.ldt : f32_pitch(a.r, a.tight);
    ws += f32_mat(a.m, a.r, a.tight);
    F32Launch l1, l2;
    if (!f32_prepare(f.t, {x.p, x.ld, false}, {U.p, U.ld, true}, T, ldT, reinterpret_cast<float*>(ws), &l1.ta[0], &l1.tb[0], &l1.p[0]) ||
        !f32_prepare(f.y, {T, ldT, false}, {V.p, V.ld, false, true}, static_cast<float*>(a.y), a.ldy, nullptr, &l2.ta[0], &l2.tb[0], &l2.p[0]))
        return PF_ERR_CUDA;
    if (a.T && !direct) { l1.p[0].C2 = static_cast<float*>(a.T); l1.p[0].ldc2 = a.ldt; }
    l2.p[0].bias = static_cast<const float*>(a.bias);
    l2.p[0].act = a.act;
    *handled = 1;
    if (nj > 0 && repack_rows_bf16_multi(jobs, nj, a.stream) != cudaSuccess) return PF_ERR_CUDA;
    const int st = f32_launch(&l1, 1, a.stream);
    return st != PF_OK ? st : f32_launch(&l2, 1, a.stream);
}

int f32_linear_bwd(const LinearArgs& a, int* handled) {
    *handled = 0;
    if (encode_fn() == nullptr || !sizes_ok(a.m, a.k, a.n, a.r)) return PF_OK;
    const F32Bwd b = linear_plan_bwd(a.m, a.k, a.n, a.r);
    if (!tiles_ok(b.t) || !tiles_ok(b.g) || !tiles_ok(b.dv) || !tiles_ok(b.du) || !tiles_ok(b.dx)) return PF_OK;
    char* ws = a.ws;
    Staged32 x, U, V, dY, T{nullptr, 0};
    RepackJob jobs[5];
    int nj = 0;
    if (!f32_stage(a.x, a.ldx, a.m, a.k, ws, &x, jobs, &nj) || !f32_stage(a.U, a.ldu, a.k, a.r, ws, &U, jobs, &nj) ||
        !f32_stage(a.V, a.ldv, a.n, a.r, ws, &V, jobs, &nj) || !f32_stage(a.dY, a.lddy, a.m, a.n, ws, &dY, jobs, &nj))
        return PF_OK;
    char* Tbuf = ws;
    ws += f32_mat(a.m, a.r);
    if (a.T) {
        if (f32_tma_ok(a.T, a.ldt)) {
            T = Staged32{a.T, a.ldt};
        } else {
            jobs[nj++] = RepackJob{a.T, 2 * a.ldt, Tbuf, 2 * f32_pitch(a.r), a.m, 2 * a.r};
            T = Staged32{Tbuf, f32_pitch(a.r)};
        }
    } else {
        T = Staged32{Tbuf, f32_pitch(a.r)};
    }
    float* G = reinterpret_cast<float*>(ws);
    const int64_t ldG = f32_pitch(a.r);
    ws += f32_mat(a.m, a.r);
    float* p1 = reinterpret_cast<float*>(ws);
    ws += std::max(b.t.partial_bytes(), b.g.partial_bytes());
    float* pv = reinterpret_cast<float*>(ws);
    ws += b.dv.partial_bytes();
    float* pu = reinterpret_cast<float*>(ws);
    F32Launch lt, la, lb;
    bool ok = true;
    if (!a.T)
        ok = f32_prepare(b.t, {x.p, x.ld, false}, {U.p, U.ld, true}, reinterpret_cast<float*>(Tbuf), f32_pitch(a.r), p1, &lt.ta[0], &lt.tb[0], &lt.p[0]);
    // (the launch before is the recomputed T, this call's re-pitch copies, or one of an earlier call)
    const bool early = !a.T;
    ok = ok && f32_prepare(b.g, {dY.p, dY.ld, false, early}, {V.p, V.ld, true, early}, G, ldG, p1, &la.ta[0], &la.tb[0], &la.p[0]) &&
         f32_prepare(b.dv, {dY.p, dY.ld, true, early}, {T.p, T.ld, true}, static_cast<float*>(a.dV), a.lddv, pv, &la.ta[1], &la.tb[1], &la.p[1]) &&
         f32_prepare(b.du, {x.p, x.ld, true, true}, {G, ldG, true}, static_cast<float*>(a.dU), a.lddu, pu, &lb.ta[0], &lb.tb[0], &lb.p[0]);
    if (ok && a.dX)
        ok = f32_prepare(b.dx, {G, ldG, false}, {U.p, U.ld, false, true}, static_cast<float*>(a.dX), a.lddx, nullptr, &lb.ta[1], &lb.tb[1], &lb.p[1]);
    if (!ok) return PF_ERR_CUDA;
    *handled = 1;
    if (nj > 0 && repack_rows_bf16_multi(jobs, nj, a.stream) != cudaSuccess) return PF_ERR_CUDA;
    int st = PF_OK;
    if (!a.T) st = f32_launch(&lt, 1, a.stream);
    if (st == PF_OK) st = f32_launch(&la, 2, a.stream);
    if (st == PF_OK) st = f32_launch(&lb, a.dX ? 2 : 1, a.stream);
    return st;
}

// The convolution on the same kernel: channel counts that are multiples of 4 (TMA pitches), output rows of at most 128
// pixels, and for a strided backward at least one tap per pixel class.
static bool f32_conv_ok(const ConvArgs& a, bool bwd) {
    if (encode_fn() == nullptr || a.kh != a.kw || a.C % 4 != 0 || a.R % 4 != 0 || a.O % 4 != 0 || a.stride > 4) return false;
    if (a.Wo > 128 || a.stride * a.Wo > 256 || a.H > 4095 || a.W > 4095) return false;
    if (bwd && (a.kh < a.stride || ceil_div(a.W, a.stride) > 128)) return false;
    const int64_t in = static_cast<int64_t>(a.N) * a.H * a.W, out = static_cast<int64_t>(a.N) * a.Ho * a.Wo;
    if (in > 0x3fffffff || out > 0x3fffffff || static_cast<int64_t>(a.kh) * a.kw * a.C > 0x3fffffff) return false;
    for (const void* p : {a.x, a.U, a.V, a.dY, static_cast<const void*>(a.T)})
        if (p && (reinterpret_cast<uintptr_t>(p) & 15) != 0) return false;
    return true;
}

size_t f32_conv_workspace(const ConvArgs& a, bool bwd) {
    if (!f32_conv_ok(a, bwd) || a.N < 1 || a.Ho < 1 || a.Wo < 1) return 0;
    if (!bwd) return conv_plan_fwd(a).t.partial_bytes();
    const F32Bwd b = conv_plan_bwd(a);
    return std::max(b.t.partial_bytes(), b.g.partial_bytes()) + b.dv.partial_bytes() + b.du.partial_bytes();
}

int f32_conv_fwd(const ConvArgs& a, int* handled) {
    *handled = 0;
    if (!f32_conv_ok(a, false)) return PF_OK;
    const F32Fwd f = conv_plan_fwd(a);
    if (!tiles_ok(f.t) || !tiles_ok(f.y)) return PF_OK;
    float* T = static_cast<float*>(a.T ? a.T : a.ws_T);
    F32Launch l1, l2;
    if (!f32_prepare(f.t, {a.x, 0, false}, {a.U, a.R, true}, T, a.R, reinterpret_cast<float*>(a.ws), &l1.ta[0], &l1.tb[0], &l1.p[0]) ||
        !f32_prepare(f.y, {T, a.R, false}, {a.V, a.R, false, true}, static_cast<float*>(a.y), a.O, nullptr, &l2.ta[0], &l2.tb[0], &l2.p[0]))
        return PF_ERR_CUDA;
    *handled = 1;
    const int st = f32_launch(&l1, 1, a.stream);
    return st != PF_OK ? st : f32_launch(&l2, 1, a.stream);
}

int f32_conv_bwd(const ConvArgs& a, int* handled) {
    *handled = 0;
    if (!f32_conv_ok(a, true)) return PF_OK;
    const F32Bwd b = conv_plan_bwd(a);
    if (!tiles_ok(b.t) || !tiles_ok(b.g) || !tiles_ok(b.dv) || !tiles_ok(b.du) || !tiles_ok(b.dx)) return PF_OK;
    const float* T = static_cast<const float*>(a.T ? a.T : a.ws_T);
    float* dT = reinterpret_cast<float*>(a.ws_G);
    char* ws = a.ws;
    float* p1 = reinterpret_cast<float*>(ws);
    ws += std::max(b.t.partial_bytes(), b.g.partial_bytes());
    float* pv = reinterpret_cast<float*>(ws);
    ws += b.dv.partial_bytes();
    float* pu = reinterpret_cast<float*>(ws);
    F32Launch lt, la, lb;
    bool ok = true;
    if (!a.T) ok = f32_prepare(b.t, {a.x, 0, false}, {a.U, a.R, true}, reinterpret_cast<float*>(a.ws_T), a.R, p1, &lt.ta[0], &lt.tb[0], &lt.p[0]);
    ok = ok && f32_prepare(b.g, {a.dY, a.O, false}, {a.V, a.R, true}, dT, a.R, p1, &la.ta[0], &la.tb[0], &la.p[0]) &&
         f32_prepare(b.dv, {a.dY, a.O, true}, {T, a.R, true}, static_cast<float*>(a.dV), a.R, pv, &la.ta[1], &la.tb[1], &la.p[1]) &&
         f32_prepare(b.du, {a.x, 0, true, true}, {dT, 0, true}, static_cast<float*>(a.dU), a.R, pu, &lb.ta[0], &lb.tb[0], &lb.p[0]);
    if (ok && a.dX) ok = f32_prepare(b.dx, {dT, 0, false}, {a.U, a.R, false, true}, static_cast<float*>(a.dX), a.C, nullptr, &lb.ta[1], &lb.tb[1], &lb.p[1]);
    if (!ok) return PF_ERR_CUDA;
    *handled = 1;
    int st = PF_OK;
    if (!a.T) st = f32_launch(&lt, 1, a.stream);
    if (st == PF_OK) st = f32_launch(&la, 2, a.stream);
    if (st == PF_OK) st = f32_launch(&lb, a.dX ? 2 : 1, a.stream);
    return st;
}

}  // namespace tc
}  // namespace pf
