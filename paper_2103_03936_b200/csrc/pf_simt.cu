// FMA (CUDA-core) GEMM with implicit-matrix views.
//
// Serves every shape and layout outside the tensor-core envelopes (odd row pitches on even widths,
// channel counts that are not multiples of 8 in bf16 or 4 in fp32).  One kernel, templated on
// how operand A is addressed: plain strided, im2col of an NHWC image (convolution forward
// and dU), or the gather form of the transposed convolution (dX).  Products accumulate in
// fp32; a reduction split over K writes fp32 partials that a second kernel sums in a fixed
// order, so results are bit-reproducible run to run.
#include <algorithm>

#include "pf_internal.h"

namespace pf {
namespace {

constexpr int BM = 64, BN = 64, BK = 16, NT = 256;

template <typename T> __device__ __forceinline__ float ldf(const void* p, int64_t idx);
template <> __device__ __forceinline__ float ldf<float>(const void* p, int64_t idx) {
    return __ldg(reinterpret_cast<const float*>(p) + idx);
}
template <> __device__ __forceinline__ float ldf<__nv_bfloat16>(const void* p, int64_t idx) {
    const unsigned short raw = __ldg(reinterpret_cast<const unsigned short*>(p) + idx);
    return __uint_as_float(static_cast<unsigned int>(raw) << 16);
}
template <typename T> __device__ __forceinline__ void stf(void* p, int64_t idx, float v);
template <> __device__ __forceinline__ void stf<float>(void* p, int64_t idx, float v) {
    reinterpret_cast<float*>(p)[idx] = v;
}
template <> __device__ __forceinline__ void stf<__nv_bfloat16>(void* p, int64_t idx, float v) {
    reinterpret_cast<__nv_bfloat16*>(p)[idx] = __float2bfloat16_rn(v);
}

template <typename T, int AK>
__device__ __forceinline__ float load_a(const MatA& A, int64_t i, int64_t l) {
    if (AK == A_PLAIN) {
        return ldf<T>(A.p, i * A.s_row + l * A.s_col);
    } else if (AK == A_IM2COL || AK == A_IM2COL_T) {
        const int64_t pix = (AK == A_IM2COL) ? i : l;
        const int64_t q = (AK == A_IM2COL) ? l : i;
        const ConvGeom& g = A.g;
        const int c = static_cast<int>(q % g.C);
        const int tap = static_cast<int>(q / g.C);
        const int b = tap % g.kw, a = tap / g.kw;
        const int wo = static_cast<int>(pix % g.Wo);
        const int64_t t = pix / g.Wo;
        const int ho = static_cast<int>(t % g.Ho);
        const int64_t n = t / g.Ho;
        const int h = ho * g.st - g.pad + a, w = wo * g.st - g.pad + b;
        if (h < 0 || h >= g.H || w < 0 || w >= g.W) return 0.f;
        return ldf<T>(A.p, ((n * g.H + h) * g.W + w) * g.C + c);
    } else {  // A_COL2IM
        const ConvGeom& g = A.g;
        const int j = static_cast<int>(l % g.R);
        const int tap = static_cast<int>(l / g.R);
        const int b = tap % g.kw, a = tap / g.kw;
        const int w = static_cast<int>(i % g.W);
        const int64_t t = i / g.W;
        const int h = static_cast<int>(t % g.H);
        const int64_t n = t / g.H;
        const int hn = h + g.pad - a, wn = w + g.pad - b;
        if (hn < 0 || wn < 0 || hn % g.st != 0 || wn % g.st != 0) return 0.f;
        const int ho = hn / g.st, wo = wn / g.st;
        if (ho >= g.Ho || wo >= g.Wo) return 0.f;
        return ldf<T>(A.p, ((n * g.Ho + ho) * g.Wo + wo) * g.R + j);
    }
}

template <typename T, int BKD>
__device__ __forceinline__ float load_b(const MatB& B, int64_t l, int64_t j) {
    if (BKD == B_PLAIN) return ldf<T>(B.p, l * B.s_row + j * B.s_col);
    const int64_t tap = l / B.R, q = l % B.R;
    return ldf<T>(B.p, tap * B.CR + j * B.R + q);
}

template <typename T, int AK, int BKD>
__global__ void __launch_bounds__(NT)
simt_gemm_kernel(const SimtGemm g) {
    __shared__ float As[BK][BM + 1];
    __shared__ float Bs[BK][BN + 1];
    const int tid = threadIdx.x;
    const int tx = tid % 16, ty = tid / 16;
    const int64_t i0 = static_cast<int64_t>(blockIdx.x) * BM;
    const int64_t j0 = static_cast<int64_t>(blockIdx.y) * BN;
    const int64_t kchunk = (g.K + g.splits - 1) / g.splits;
    const int64_t kbeg = static_cast<int64_t>(blockIdx.z) * kchunk;
    const int64_t kend = kbeg + kchunk < g.K ? kbeg + kchunk : g.K;

    float acc[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = 0.f;

    for (int64_t l0 = kbeg; l0 < kend; l0 += BK) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            int li, ii;
            if (g.A.l_fast) { li = tid % BK; ii = tid / BK + (NT / BK) * q; }
            else            { ii = tid % BM; li = tid / BM + (NT / BM) * q; }
            const int64_t gi = i0 + ii, gl = l0 + li;
            As[li][ii] = (gi < g.M && gl < kend) ? load_a<T, AK>(g.A, gi, gl) : 0.f;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            int li, ji;
            if (g.B.l_fast) { li = tid % BK; ji = tid / BK + (NT / BK) * q; }
            else            { ji = tid % BN; li = tid / BN + (NT / BN) * q; }
            const int64_t gj = j0 + ji, gl = l0 + li;
            Bs[li][ji] = (gj < g.N && gl < kend) ? load_b<T, BKD>(g.B, gl, gj) : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int l = 0; l < BK; ++l) {
            float a[4], b[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) a[u] = As[l][ty * 4 + u];
#pragma unroll
            for (int v = 0; v < 4; ++v) b[v] = Bs[l][tx * 4 + v];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(a[u], b[v], acc[u][v]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int64_t gi = i0 + ty * 4 + u;
        if (gi >= g.M) continue;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int64_t gj = j0 + tx * 4 + v;
            if (gj >= g.N) continue;
            if (g.splits > 1) g.partial[(static_cast<int64_t>(blockIdx.z) * g.M + gi) * g.N + gj] = acc[u][v];
            else stf<T>(g.C, gi * g.ldc + gj, acc[u][v]);
        }
    }
}

template <typename T>
__global__ void __launch_bounds__(256)
splitk_reduce_kernel(const float* __restrict__ partial, void* C, int64_t ldc, int64_t M, int64_t N,
                     int splits) {
    const int64_t total = M * N;
    for (int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < total;
         e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        float s = 0.f;
        for (int z = 0; z < splits; ++z) s += partial[static_cast<int64_t>(z) * total + e];
        stf<T>(C, (e / N) * ldc + (e % N), s);
    }
}

template <typename T>
cudaError_t launch_typed(const SimtGemm& g, cudaStream_t stream) {
    dim3 grid(static_cast<unsigned>(ceil_div(g.M, BM)), static_cast<unsigned>(ceil_div(g.N, BN)),
              static_cast<unsigned>(g.splits));
    if (g.A.kind == A_PLAIN && g.B.kind == B_PLAIN)
        simt_gemm_kernel<T, A_PLAIN, B_PLAIN><<<grid, NT, 0, stream>>>(g);
    else if (g.A.kind == A_IM2COL && g.B.kind == B_PLAIN)
        simt_gemm_kernel<T, A_IM2COL, B_PLAIN><<<grid, NT, 0, stream>>>(g);
    else if (g.A.kind == A_IM2COL_T && g.B.kind == B_PLAIN)
        simt_gemm_kernel<T, A_IM2COL_T, B_PLAIN><<<grid, NT, 0, stream>>>(g);
    else if (g.A.kind == A_COL2IM && g.B.kind == B_TAPSPLIT)
        simt_gemm_kernel<T, A_COL2IM, B_TAPSPLIT><<<grid, NT, 0, stream>>>(g);
    else
        return cudaErrorInvalidValue;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    count_launch();
    if (g.splits > 1) {
        const int64_t total = g.M * g.N;
        const int blocks = static_cast<int>(ceil_div(total, 256) < 4 * num_sms() ? ceil_div(total, 256)
                                                                                : 4 * num_sms());
        splitk_reduce_kernel<T><<<blocks, 256, 0, stream>>>(g.partial, g.C, g.ldc, g.M, g.N, g.splits);
        e = cudaGetLastError();
        if (e == cudaSuccess) count_launch();
    }
    return e;
}

__global__ void __launch_bounds__(256)
repack_rows_kernel(const unsigned short* __restrict__ src, int64_t ld_src,
                   unsigned short* __restrict__ dst, int64_t ld_dst, int64_t rows, int64_t cols,
                   int64_t cols_padded) {
    const int64_t total = rows * cols_padded;
    for (int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < total;
         e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t rr = e / cols_padded, cc = e % cols_padded;
        dst[rr * ld_dst + cc] = cc < cols ? src[rr * ld_src + cc] : static_cast<unsigned short>(0);
    }
}

// Several re-pitch copies in one launch.  A work item is one 16-byte piece (8 elements) of a
// destination row: the destination is 16-byte aligned with a pitch that is a multiple of 8
// elements, the source may start at any element.  Pure streaming (4 bytes per element), so both sides move
// 16 bytes per access: a whole piece is assembled from the two aligned source vectors that cover it with a
// funnel shift; a row's last piece takes the vectors that hold at least one of its bytes and masks what lies behind the
// row.  (Bytes beside the source inside an aligned vector are read, never used.)
// A job may cover several matrices (groups) a fixed stride apart, which land one after the other.
// Launched with programmatic dependent launch: its start hides behind the previous kernel's tail, and the
// product that reads the copies starts its own prologue meanwhile.
// Bytes [4 q + bit / 8, + 16) of the window lo:hi.
__device__ __forceinline__ uint4 shifted_vector(const uint4 o, const uint4 h, unsigned q, unsigned bit) {
    const bool q1 = q & 1, q2 = q & 2;
    const unsigned x0 = q2 ? o.z : o.x, x1 = q2 ? o.w : o.y, x2 = q2 ? h.x : o.z, x3 = q2 ? h.y : o.w, x4 = q2 ? h.z : h.x, x5 = q2 ? h.w : h.y;
    const unsigned w0 = q1 ? x1 : x0, w1 = q1 ? x2 : x1, w2 = q1 ? x3 : x2, w3 = q1 ? x4 : x3, w4 = q1 ? x5 : x4;
    return make_uint4(__funnelshift_r(w0, w1, bit), __funnelshift_r(w1, w2, bit), __funnelshift_r(w2, w3, bit), __funnelshift_r(w3, w4, bit));
}
// kDeep: pieces of a thread in flight together.
template <int kDeep>
__global__ void __launch_bounds__(256)
repack_multi_kernel(const __grid_constant__ RepackBatchArgs a) {
    const unsigned int total = a.item_end[a.count - 1], step = gridDim.x * blockDim.x;
    const unsigned short* sp[kDeep];
    unsigned short* to[kDeep];
    int left[kDeep];                      // elements of the row from the piece on, 0: no piece
    auto place = [&](unsigned int first) {
#pragma unroll
        for (int u = 0; u < kDeep; ++u) {
            const unsigned int it = first + u * step;
            left[u] = 0;
            if (it >= total) continue;
            int j = 0;
            while (j + 1 < a.count && it >= a.item_end[j]) ++j;
            const unsigned int local = it - (j > 0 ? a.item_end[j - 1] : 0u), ppr = static_cast<unsigned int>(a.pieces_per_row[j]);
            const unsigned int row = local / ppr;
            const int c0 = static_cast<int>(local - row * ppr) * 8;
            const unsigned int g = a.gs_src[j] ? row / static_cast<unsigned int>(a.rows[j]) : 0u;
            sp[u] = a.src[j] + g * a.gs_src[j] + (row - g * static_cast<unsigned int>(a.rows[j])) * a.ld_src[j] + c0;
            to[u] = a.dst[j] + row * a.ld_dst[j] + c0;
            left[u] = a.cols[j] - c0;
        }
    };
    unsigned int first = blockIdx.x * blockDim.x + threadIdx.x;
    place(first);                         // (reads the kernel's parameters only: beside the previous kernel's tail)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    while (first < total) {
        // the aligned vectors that hold at least one byte of each piece, all of them in flight together
        uint4 lo[kDeep], hi[kDeep];
        unsigned int sh[kDeep];
#pragma unroll
        for (int u = 0; u < kDeep; ++u) {
            sh[u] = static_cast<unsigned int>(reinterpret_cast<uintptr_t>(sp[u])) & 15u;
            const uint4* v = reinterpret_cast<const uint4*>(reinterpret_cast<uintptr_t>(sp[u]) - sh[u]);
            lo[u] = hi[u] = make_uint4(0u, 0u, 0u, 0u);
            if (left[u] > 0) lo[u] = __ldg(v);
            if (left[u] > 0 && static_cast<int>(sh[u]) + 2 * min(left[u], 8) > 16) hi[u] = __ldg(v + 1);
        }
#pragma unroll
        for (int u = 0; u < kDeep; ++u) {
            if (left[u] <= 0) continue;
            uint4 o = shifted_vector(lo[u], hi[u], sh[u] >> 2, (sh[u] & 3u) * 8u);
            if (left[u] < 8) {            // zeros behind the row's end
                auto keep = [&](int e) { return (e < left[u] ? 0xffffu : 0u) | (e + 1 < left[u] ? 0xffff0000u : 0u); };
                o.x &= keep(0); o.y &= keep(2); o.z &= keep(4); o.w &= keep(6);
            }
            *reinterpret_cast<uint4*>(to[u]) = o;
        }
        if (total - first <= kDeep * step) break;
        first += kDeep * step;
        place(first);
    }
}

}  // namespace

int simt_pick_splits(int64_t M, int64_t N, int64_t K) {
    const int64_t tiles = ceil_div(M, BM) * ceil_div(N, BN);
    int64_t s = ceil_div(2 * num_sms(), tiles);
    const int64_t max_by_k = ceil_div(K, 8 * BK);
    if (s > max_by_k) s = max_by_k;
    if (s > 64) s = 64;
    if (s < 1) s = 1;
    return static_cast<int>(s);
}

cudaError_t splitk_reduce(const float* partial, void* C, int64_t ldc, int64_t M, int64_t N, int splits,
                          int dtype, cudaStream_t stream) {
    const int64_t total = M * N;
    if (total <= 0) return cudaSuccess;
    const int blocks = static_cast<int>(ceil_div(total, 256) < 4 * num_sms() ? ceil_div(total, 256) : 4 * num_sms());
    if (dtype == PF_BF16) splitk_reduce_kernel<__nv_bfloat16><<<blocks, 256, 0, stream>>>(partial, C, ldc, M, N, splits);
    else splitk_reduce_kernel<float><<<blocks, 256, 0, stream>>>(partial, C, ldc, M, N, splits);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) count_launch();
    return e;
}

cudaError_t simt_gemm(const SimtGemm& g, cudaStream_t stream) {
    if (g.M <= 0 || g.N <= 0) return cudaSuccess;
    if (ceil_div(g.N, BN) > 65535 || ceil_div(g.M, BM) > 2147483647LL) return cudaErrorInvalidConfiguration;
    return g.dtype == PF_BF16 ? launch_typed<__nv_bfloat16>(g, stream) : launch_typed<float>(g, stream);
}

// acc[rows, cols] (fp32, dense) = (first ? 0 : acc) + src (storage dtype, pitch ld_src); and its
// counterpart that rounds the sums to the storage dtype once.  They add up the per-group input
// gradients of a grouped layer whose groups share one input, on the path that runs group by group.
template <typename T>
__global__ void accumulate_kernel(float* acc, const T* src, int64_t ld_src, int64_t rows, int64_t cols, int first) {
    const int64_t total = rows * cols;
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < total;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t rr = i / cols, cc = i - rr * cols;
        const float v = static_cast<float>(src[rr * ld_src + cc]);
        acc[i] = first ? v : acc[i] + v;
    }
}
template <typename T>
__global__ void round_out_kernel(const float* acc, T* dst, int64_t ld_dst, int64_t rows, int64_t cols) {
    const int64_t total = rows * cols;
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < total;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t rr = i / cols, cc = i - rr * cols;
        dst[rr * ld_dst + cc] = static_cast<T>(acc[i]);
    }
}
// out = (accumulate ? out : 0) + src, the sum taken in fp32 and rounded once to out's type.
template <typename TO, typename TS>
__global__ void grad_combine_kernel(TO* out, int64_t ld_out, const TS* src, int64_t ld_src, int64_t rows, int64_t cols,
                                    int accumulate) {
    const int64_t total = rows * cols;
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < total;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t rr = i / cols, cc = i - rr * cols;
        float v = static_cast<float>(src[rr * ld_src + cc]);
        if (accumulate) v += static_cast<float>(out[rr * ld_out + cc]);
        out[rr * ld_out + cc] = static_cast<TO>(v);
    }
}
cudaError_t grad_combine(void* out, int64_t ld_out, int out_dtype, const void* src, int64_t ld_src, int src_dtype,
                         int64_t rows, int64_t cols, bool accumulate, cudaStream_t stream) {
    const int64_t total = rows * cols;
    if (total <= 0) return cudaSuccess;
    const int blocks = static_cast<int>(ceil_div(total, 256) < 8 * num_sms() ? ceil_div(total, 256) : 8 * num_sms());
    const int acc = accumulate ? 1 : 0;
    if (out_dtype == PF_F32 && src_dtype == PF_BF16)
        grad_combine_kernel<<<blocks, 256, 0, stream>>>(static_cast<float*>(out), ld_out, static_cast<const __nv_bfloat16*>(src), ld_src, rows, cols, acc);
    else if (out_dtype == PF_F32)
        grad_combine_kernel<<<blocks, 256, 0, stream>>>(static_cast<float*>(out), ld_out, static_cast<const float*>(src), ld_src, rows, cols, acc);
    else
        grad_combine_kernel<<<blocks, 256, 0, stream>>>(static_cast<__nv_bfloat16*>(out), ld_out, static_cast<const __nv_bfloat16*>(src), ld_src, rows, cols, acc);
    count_launch();
    return cudaGetLastError();
}

// The fp32 slices a split tensor-core reduction left in the workspace, summed once more in slice order
// (the very sums the reduction rounded to bf16) and written unrounded to an fp32 matrix and / or added to
// the old contents.  Slice layout: [tile][slice][32-row quadrant][4-column group][row][4 floats], tile = column
// tile * tiles_x + row tile.
struct SliceSumJob {
    const float* partial;
    void* out;
    long long ld;
    int M, N, S, bn, tiles_x, tiles_y, out_f32, accumulate, conv_c;
};
__global__ void __launch_bounds__(256) slices_to_gradients_kernel(const SliceSumJob j0, const SliceSumJob j1, int blocks0) {
    const bool first = static_cast<int>(blockIdx.x) < blocks0;
    const SliceSumJob& j = first ? j0 : j1;
    const int b = first ? blockIdx.x : blockIdx.x - blocks0;
    const int nb = first ? blocks0 : gridDim.x - blocks0;
    const int pieces = j.bn / 4;
    const long long total = static_cast<long long>(j.tiles_x) * j.tiles_y * 128 * pieces;
    for (long long i = static_cast<long long>(b) * blockDim.x + threadIdx.x; i < total; i += static_cast<long long>(nb) * blockDim.x) {
        const int in = static_cast<int>(i % (128 * pieces)), tile = static_cast<int>(i / (128 * pieces));
        const int pc = (in >> 5) % pieces, rin = (in >> 5) / pieces * 32 + (in & 31);
        const int bx = tile % j.tiles_x, by = tile / j.tiles_x;
        const int col = by * j.bn + pc * 4;
        int row = bx * 128 + rin;
        if (j.conv_c > 0) {      // pairs of 64-channel blocks, ceil(C / 64) blocks per tap
            const int blks = (j.conv_c + 63) / 64, blk = row >> 6, tap = blk / blks, c = (blk - tap * blks) * 64 + (row & 63);
            row = c < j.conv_c ? tap * j.conv_c + c : j.M;
        }
        if (row >= j.M || col >= j.N) continue;
        const float* src = j.partial + static_cast<size_t>(tile) * j.S * 128 * j.bn + static_cast<size_t>(in) * 4;
        float4 acc = *reinterpret_cast<const float4*>(src);
        for (int s = 1; s < j.S; ++s) {
            const float4 w = *reinterpret_cast<const float4*>(src + static_cast<size_t>(s) * 128 * j.bn);
            acc.x += w.x; acc.y += w.y; acc.z += w.z; acc.w += w.w;
        }
        const float sums[4] = {acc.x, acc.y, acc.z, acc.w};
        const size_t at = static_cast<size_t>(row) * j.ld + col;
        for (int e = 0; e < 4 && col + e < j.N; ++e) {
            if (j.out_f32) {
                float* o = static_cast<float*>(j.out) + at + e;
                *o = j.accumulate ? *o + sums[e] : sums[e];
            } else {
                __nv_bfloat16* o = static_cast<__nv_bfloat16*>(j.out) + at + e;
                *o = __float2bfloat16_rn(j.accumulate ? __bfloat162float(*o) + sums[e] : sums[e]);
            }
        }
    }
}
cudaError_t slices_to_gradients(const SliceSums* jobs, int count, cudaStream_t stream) {
    if (count < 1 || count > 2) return cudaErrorInvalidValue;
    SliceSumJob j[2];
    int blocks[2] = {0, 0};
    for (int i = 0; i < 2; ++i) {
        const SliceSums& s = jobs[i < count ? i : 0];
        j[i] = SliceSumJob{s.partial, s.out, s.ld, s.M, s.N, s.splits, s.bn, s.tiles_x, s.tiles_y, s.out_f32 ? 1 : 0, s.accumulate ? 1 : 0, s.conv_c};
        if (i < count) {
            const long long total = static_cast<long long>(s.tiles_x) * s.tiles_y * 128 * (s.bn / 4);
            blocks[i] = static_cast<int>(std::min<long long>(ceil_div(total, 256), 4LL * num_sms()));
            if (blocks[i] < 1) blocks[i] = 1;
        }
    }
    slices_to_gradients_kernel<<<blocks[0] + blocks[1], 256, 0, stream>>>(j[0], j[1], blocks[0]);
    count_launch();
    return cudaGetLastError();
}

// Backward of y = act(z + bias): dZ = dY where y > 0 (act = max(0, .)) or everywhere (identity), written
// over dY; partial column sums of dZ per chunk of rows go to `part` [chunks, cols] (fp32), summed in chunk
// order by the second kernel into db (deterministic).
// Bound by memory: a lane reads kVec consecutive columns (16 bytes where pitch and pointers allow) of every eighth
// row of the chunk, four rows in flight.
template <typename T, int kVec>
struct alignas(sizeof(T) * kVec) Pack {
    T v[kVec];
};
template <typename T, int kVec>
__global__ void __launch_bounds__(256) act_bwd_kernel(const T* y, int64_t ldy, T* dY, int64_t lddy, int64_t rows,
                                                      int64_t cols, int act, float* part, int rows_per_chunk) {
    using P = Pack<T, kVec>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t col = (static_cast<int64_t>(blockIdx.x) * 32 + lane) * kVec;
    const int64_t r_beg = static_cast<int64_t>(blockIdx.y) * rows_per_chunk;
    const int64_t r_end = r_beg + rows_per_chunk < rows ? r_beg + rows_per_chunk : rows;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    float sum[kVec];
#pragma unroll
    for (int e = 0; e < kVec; ++e) sum[e] = 0.f;
    if (col < cols) {
        auto one = [&](int64_t r, P g, const P& yv) {
            if (act == 1) {
                bool cut = false;
#pragma unroll
                for (int e = 0; e < kVec; ++e)
                    if (!(static_cast<float>(yv.v[e]) > 0.f)) { g.v[e] = static_cast<T>(0.f); cut = true; }
                if (cut) *reinterpret_cast<P*>(dY + r * lddy + col) = g;
            }
#pragma unroll
            for (int e = 0; e < kVec; ++e) sum[e] += static_cast<float>(g.v[e]);
        };
        int64_t r = r_beg + warp;
        for (; r + 24 < r_end; r += 32) {
            P g[4], yv[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) g[u] = *reinterpret_cast<const P*>(dY + (r + 8 * u) * lddy + col);
            if (act == 1)
#pragma unroll
                for (int u = 0; u < 4; ++u) yv[u] = *reinterpret_cast<const P*>(y + (r + 8 * u) * ldy + col);
#pragma unroll
            for (int u = 0; u < 4; ++u) one(r + 8 * u, g[u], act == 1 ? yv[u] : g[u]);
        }
        for (; r < r_end; r += 8) {
            const P g = *reinterpret_cast<const P*>(dY + r * lddy + col);
            one(r, g, act == 1 ? *reinterpret_cast<const P*>(y + r * ldy + col) : g);
        }
    }
    if (!part) return;
    __shared__ float red[8][32 * kVec + 1];
#pragma unroll
    for (int e = 0; e < kVec; ++e) red[warp][lane * kVec + e] = sum[e];
    __syncthreads();
    for (int c = threadIdx.x; c < 32 * kVec; c += 256) {
        const int64_t cc = static_cast<int64_t>(blockIdx.x) * 32 * kVec + c;
        if (cc >= cols) break;
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) s += red[w][c];
        part[static_cast<int64_t>(blockIdx.y) * cols + cc] = s;
    }
}
// Eight warps per 32 columns: warp w adds chunks w, w + 8, ..., then the eight sums are added in warp order.
template <typename T>
__global__ void __launch_bounds__(256) act_bwd_bias_kernel(const float* part, int chunks, int64_t cols, T* db) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t col = static_cast<int64_t>(blockIdx.x) * 32 + lane;
    float s = 0.f;
    if (col < cols)
#pragma unroll 8
        for (int c = warp; c < chunks; c += 8) s += part[static_cast<int64_t>(c) * cols + col];
    __shared__ float red[8][32];
    red[warp][lane] = s;
    __syncthreads();
    if (warp == 0 && col < cols) {
        for (int w = 1; w < 8; ++w) s += red[w][lane];
        db[col] = static_cast<T>(s);
    }
}
// The same pass with db in one launch: the blocks of a cluster share a panel of columns, each sums its rows, and the
// first adds the blocks' sums in block order (deterministic).  A panel is 128 bytes wide where 16-byte accesses fit
// (eight lanes to a row, four rows to a warp access), so that a batch of a few hundred rows is one trip to memory and a
// layer of a few columns still gets a cluster of blocks.  Bound by latency: the launch, one to four trips to memory, the
// sums' way through shared memory.
constexpr int kColThreads = 512, kColBlocks = 8;      // blocks of a cluster: the largest portable size
template <typename T, int kVec>
constexpr int kColLanes = kVec * sizeof(T) == 16 ? 8 : kVec * sizeof(T) == 8 ? 16 : 32;      // lanes to a row
template <typename T, int kVec, bool kRelu>
__global__ void __launch_bounds__(kColThreads) act_bwd_sum_kernel(const T* y, int64_t ldy, T* dY, int64_t lddy, int64_t rows,
                                                                  int64_t cols, T* db, int64_t rows_per_block) {
    using P = Pack<T, kVec>;
    constexpr int kLanes = kColLanes<T, kVec>, kPanel = kLanes * kVec, kWarps = kColThreads / 32;
    constexpr int kStep = kWarps * (32 / kLanes), kDeep = 4;
    __shared__ float red[kWarps][kPanel];
    __shared__ float sums[kColBlocks][kPanel];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t col = static_cast<int64_t>(blockIdx.x) * kPanel + (lane % kLanes) * kVec;
    const int64_t r_beg = static_cast<int64_t>(blockIdx.y) * rows_per_block;
    const int64_t r_end = r_beg + rows_per_block < rows ? r_beg + rows_per_block : rows;
    asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");      // (waited for before the sums travel: every block runs by then)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    float sum[kVec];
#pragma unroll
    for (int e = 0; e < kVec; ++e) sum[e] = 0.f;
    if (col < cols) {
        auto one = [&](int64_t r, P g, const P& yv) {
            if (kRelu) {
                bool cut = false;
#pragma unroll
                for (int e = 0; e < kVec; ++e)
                    if (!(static_cast<float>(yv.v[e]) > 0.f)) { g.v[e] = static_cast<T>(0.f); cut = true; }
                if (cut) *reinterpret_cast<P*>(dY + r * lddy + col) = g;
            }
#pragma unroll
            for (int e = 0; e < kVec; ++e) sum[e] += static_cast<float>(g.v[e]);
        };
        int64_t r = r_beg + warp * (32 / kLanes) + lane / kLanes;
        for (; r + (kDeep - 1) * kStep < r_end; r += kDeep * kStep) {
            P g[kDeep], yv[kRelu ? kDeep : 1];
#pragma unroll
            for (int u = 0; u < kDeep; ++u) g[u] = *reinterpret_cast<const P*>(dY + (r + u * kStep) * lddy + col);
            if (kRelu)
#pragma unroll
                for (int u = 0; u < kDeep; ++u) yv[u] = *reinterpret_cast<const P*>(y + (r + u * kStep) * ldy + col);
#pragma unroll
            for (int u = 0; u < kDeep; ++u) one(r + u * kStep, g[u], yv[kRelu ? u : 0]);
        }
#pragma unroll 4
        for (; r < r_end; r += kStep) {
            const P g = *reinterpret_cast<const P*>(dY + r * lddy + col);
            one(r, g, kRelu ? *reinterpret_cast<const P*>(y + r * ldy + col) : g);
        }
    }
#pragma unroll
    for (int e = 0; e < kVec; ++e) {
#pragma unroll
        for (int o = kLanes; o < 32; o *= 2) sum[e] += __shfl_xor_sync(0xffffffffu, sum[e], o);
        if (lane < kLanes) red[warp][lane * kVec + e] = sum[e];
    }
    __syncthreads();
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    const int c = threadIdx.x;
    if (c < kPanel) {
        float s = red[0][c];
#pragma unroll
        for (int w = 1; w < kWarps; ++w) s += red[w][c];
        uint32_t to;
        asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(to) : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(&sums[blockIdx.y][c]))));
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(to), "f"(s) : "memory");
    }
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    const int64_t cc = static_cast<int64_t>(blockIdx.x) * kPanel + c;
    if (blockIdx.y == 0 && c < kPanel && cc < cols) {
        float s = sums[0][c];
        for (unsigned b = 1; b < gridDim.y; ++b) s += sums[b][c];
        db[cc] = static_cast<T>(s);
    }
}
int act_bwd_chunks(int64_t rows) {
    const int64_t c = ceil_div(rows, 128);
    return static_cast<int>(c < 1 ? 1 : (c > 64 ? 64 : c));
}
template <typename... KArgs, typename... Args>
static cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, cudaStream_t stream, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = dim3(256); cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
    if (e == cudaSuccess) count_launch();
    return e;
}
// One launch up to 4096 rows: beyond, eight blocks to a panel are fewer than memory wants and the second launch of the
// chunks' form costs less.  Training steps with a bias, chunks -> cluster: 64 x 64 -> 256: 20.6 -> 17.6 us; 2048 x 512 -> 2048:
// 36.6 -> 34.6; 4096 x 512 -> 2048: 42.2 -> 41.0; 8192 x 512 -> 2048: 54.8 -> 56.2; 16384 x 256 -> 1024: 57.3 -> 64.0.
constexpr int64_t kColRows = 4096;
template <typename T, int kVec>
static cudaError_t launch_col_sum(const T* y, int64_t ldy, T* dY, int64_t lddy, T* db, int64_t rows, int64_t cols, int act, cudaStream_t stream) {
    constexpr int kPanel = kColLanes<T, kVec> * kVec, kStep = kColThreads / kColLanes<T, kVec>;
    // a block has at least one full access of every thread
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>(kColBlocks, ceil_div(rows, kStep)));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(ceil_div(cols, kPanel)), static_cast<unsigned>(blocks));
    cfg.blockDim = dim3(kColThreads); cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1; attr[1].val.clusterDim.y = static_cast<unsigned>(blocks); attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 2;
    auto* kernel = act == 1 ? act_bwd_sum_kernel<T, kVec, true> : act_bwd_sum_kernel<T, kVec, false>;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, y, ldy, dY, lddy, rows, cols, db, ceil_div(rows, blocks));
    if (e == cudaSuccess) count_launch();
    return e;
}
template <typename T>
static cudaError_t act_bwd_typed(const T* y, int64_t ldy, T* dY, int64_t lddy, T* db, int64_t rows, int64_t cols, int act, float* part,
                                 cudaStream_t stream) {
    const int chunks = act_bwd_chunks(rows);
    const int rpc = static_cast<int>(ceil_div(rows, chunks));
    float* pp = db ? part : nullptr;
    // the widest access that keeps every row aligned and whole
    constexpr int64_t kSize = sizeof(T);
    int64_t unit = static_cast<int64_t>(reinterpret_cast<uintptr_t>(dY)) | (lddy * kSize) | (cols * kSize) | 16;
    if (act == 1) unit |= static_cast<int64_t>(reinterpret_cast<uintptr_t>(y)) | (ldy * kSize);
    const int vec = static_cast<int>((unit & -unit) / kSize);
    auto grid = [&](int v) { return dim3(static_cast<unsigned>(ceil_div(cols, 32 * v)), static_cast<unsigned>(chunks)); };
    cudaError_t e;
    if (db && rows <= kColRows) {
        if (vec >= 8) return launch_col_sum<T, static_cast<int>(16 / kSize)>(y, ldy, dY, lddy, db, rows, cols, act, stream);
        if (vec >= 4) return launch_col_sum<T, 4>(y, ldy, dY, lddy, db, rows, cols, act, stream);
        if (vec >= 2) return launch_col_sum<T, 2>(y, ldy, dY, lddy, db, rows, cols, act, stream);
        return launch_col_sum<T, 1>(y, ldy, dY, lddy, db, rows, cols, act, stream);
    }
    if (vec >= 8) e = launch_pdl(act_bwd_kernel<T, static_cast<int>(16 / kSize)>, grid(8), stream, y, ldy, dY, lddy, rows, cols, act, pp, rpc);
    else if (vec >= 4) e = launch_pdl(act_bwd_kernel<T, 4>, grid(4), stream, y, ldy, dY, lddy, rows, cols, act, pp, rpc);
    else if (vec >= 2) e = launch_pdl(act_bwd_kernel<T, 2>, grid(2), stream, y, ldy, dY, lddy, rows, cols, act, pp, rpc);
    else e = launch_pdl(act_bwd_kernel<T, 1>, grid(1), stream, y, ldy, dY, lddy, rows, cols, act, pp, rpc);
    if (e != cudaSuccess || !db) return e;
    return launch_pdl(act_bwd_bias_kernel<T>, dim3(static_cast<unsigned>(ceil_div(cols, 32))), stream, part, chunks, cols, db);
}
cudaError_t act_bwd(const void* y, int64_t ldy, void* dY, int64_t lddy, void* db, int64_t rows, int64_t cols, int act,
                    int dtype, float* part, cudaStream_t stream) {
    if (rows <= 0 || cols <= 0) return cudaSuccess;
    if (dtype == PF_BF16)
        return act_bwd_typed(static_cast<const __nv_bfloat16*>(y), ldy, static_cast<__nv_bfloat16*>(dY), lddy, static_cast<__nv_bfloat16*>(db),
                             rows, cols, act, part, stream);
    return act_bwd_typed(static_cast<const float*>(y), ldy, static_cast<float*>(dY), lddy, static_cast<float*>(db), rows, cols, act, part, stream);
}

// y = act(y + bias) in place (the paths that do not fuse the epilogue into the producing kernel).
template <typename T>
__global__ void bias_act_kernel(T* y, int64_t ld, int64_t rows, int64_t cols, const T* bias, int act) {
    const int64_t total = rows * cols;
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < total;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t rr = i / cols, cc = i - rr * cols;
        float v = static_cast<float>(y[rr * ld + cc]);
        if (bias) v += static_cast<float>(bias[cc]);
        if (act == 1) v = fmaxf(v, 0.f);
        y[rr * ld + cc] = static_cast<T>(v);
    }
}
cudaError_t bias_act_inplace(void* y, int64_t ld, int64_t rows, int64_t cols, const void* bias, int act, int dtype,
                             cudaStream_t stream) {
    const int64_t total = rows * cols;
    if (total <= 0 || (!bias && !act)) return cudaSuccess;
    const int blocks = static_cast<int>(ceil_div(total, 256) < 8 * num_sms() ? ceil_div(total, 256) : 8 * num_sms());
    if (dtype == PF_BF16)
        bias_act_kernel<<<blocks, 256, 0, stream>>>(static_cast<__nv_bfloat16*>(y), ld, rows, cols,
                                                    static_cast<const __nv_bfloat16*>(bias), act);
    else
        bias_act_kernel<<<blocks, 256, 0, stream>>>(static_cast<float*>(y), ld, rows, cols, static_cast<const float*>(bias), act);
    count_launch();
    return cudaGetLastError();
}
cudaError_t accumulate_f32(float* acc, const void* src, int64_t ld_src, int64_t rows, int64_t cols, int dtype, bool first,
                           cudaStream_t stream) {
    const int64_t total = rows * cols;
    if (total <= 0) return cudaSuccess;
    const int blocks = static_cast<int>(ceil_div(total, 256) < 8 * num_sms() ? ceil_div(total, 256) : 8 * num_sms());
    if (dtype == PF_BF16)
        accumulate_kernel<<<blocks, 256, 0, stream>>>(acc, static_cast<const __nv_bfloat16*>(src), ld_src, rows, cols, first ? 1 : 0);
    else
        accumulate_kernel<<<blocks, 256, 0, stream>>>(acc, static_cast<const float*>(src), ld_src, rows, cols, first ? 1 : 0);
    count_launch();
    return cudaGetLastError();
}
cudaError_t round_out_f32(const float* acc, void* dst, int64_t ld_dst, int64_t rows, int64_t cols, int dtype,
                          cudaStream_t stream) {
    const int64_t total = rows * cols;
    if (total <= 0) return cudaSuccess;
    const int blocks = static_cast<int>(ceil_div(total, 256) < 8 * num_sms() ? ceil_div(total, 256) : 8 * num_sms());
    if (dtype == PF_BF16)
        round_out_kernel<<<blocks, 256, 0, stream>>>(acc, static_cast<__nv_bfloat16*>(dst), ld_dst, rows, cols);
    else
        round_out_kernel<<<blocks, 256, 0, stream>>>(acc, static_cast<float*>(dst), ld_dst, rows, cols);
    count_launch();
    return cudaGetLastError();
}

cudaError_t repack_rows_bf16(const void* src, int64_t ld_src, void* dst, int64_t ld_dst,
                             int64_t rows, int64_t cols, int64_t cols_padded, cudaStream_t stream) {
    const int64_t total = rows * cols_padded;
    if (total <= 0) return cudaSuccess;
    const int blocks = static_cast<int>(ceil_div(total, 256) < 8 * num_sms() ? ceil_div(total, 256)
                                                                            : 8 * num_sms());
    repack_rows_kernel<<<blocks, 256, 0, stream>>>(static_cast<const unsigned short*>(src), ld_src,
                                                   static_cast<unsigned short*>(dst), ld_dst, rows, cols,
                                                   cols_padded);
    count_launch();
    return cudaGetLastError();
}

// One launch holds kRepackJobs runs of rows and counts its pieces in 32 bits; what is more goes into further launches.
cudaError_t repack_rows_bf16_multi(const RepackJob* jobs, int count, cudaStream_t stream) {
    constexpr long long kMostPieces = 0x7fffffffLL;
    RepackBatchArgs a = {};
    long long total = 0;
    auto launch = [&]() -> cudaError_t {
        if (a.count == 0) return cudaSuccess;
        cudaLaunchConfig_t cfg = {};
        // Copies of 7.3 to 9.7 MB are a trip and a half to memory with one piece of a thread in flight (twelve to sixteen blocks for an SM that
        // holds eight): four pieces, in one wave of blocks (four to an SM).  Training steps, one piece / four: 700 x 1500 -> 375 -> 6000 49.4 / 47.8 us, 900 of them
        // 58.2 / 56.4, 600 x 1996 -> 375 -> 6000 49.9 / 48.1, 1200 x 1500 -> 375 -> 3000 53.1 / 52.2; a forward or backward by itself 1 to 2 % longer.  Smaller
        // ones fit a wave either way and pay for the longer start (3000 x 1004 -> 252 -> 1004, 7.1 MB, forward 19.8 / 20.1; backward of 2048 x 500 -> 125 -> 2000 22.1
        // / 22.6, of 1024 x 2044 -> 128 -> 512 14.8 / 15.6); larger ones stream, for which twice the threads do better (8 x (700 x 1500 -> 375 ->
        // 1500), 20 and 41 MB, 102.5 / 104.6).
        const bool deep = total > 12 * 256 * num_sms() && total <= 16 * 256 * num_sms();
        cfg.gridDim = dim3(static_cast<unsigned>(deep ? std::min<int64_t>(ceil_div(total, 256), 4 * num_sms()) : std::min<int64_t>(ceil_div(total, 256), 16 * num_sms())));
        cfg.blockDim = dim3(256);
        cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
        const cudaError_t e = cudaLaunchKernelEx(&cfg, deep ? repack_multi_kernel<4> : repack_multi_kernel<1>, a);
        if (e == cudaSuccess) count_launch();
        a.count = 0;
        total = 0;
        return e;
    };
    // rows of one matrix or of `groups` matrices gs elements apart (0: one run of rows), `first` rows into the destination
    auto add = [&](const RepackJob& j, const unsigned short* src, int64_t first, int64_t rows, int64_t groups, int64_t gs) {
        const int k = a.count++;
        a.src[k] = src;
        a.dst[k] = static_cast<unsigned short*>(j.dst) + first * j.ld_dst;
        a.ld_src[k] = j.ld_src; a.ld_dst[k] = j.ld_dst;
        a.gs_src[k] = gs;
        a.cols[k] = static_cast<int>(j.cols);
        a.rows[k] = static_cast<int>(rows);
        a.pieces_per_row[k] = static_cast<int>((j.cols + 7) / 8);
        total += rows * groups * a.pieces_per_row[k];
        a.item_end[k] = static_cast<unsigned int>(total);
    };
    for (int i = 0; i < count; ++i) {
        const RepackJob& j = jobs[i];
        const int64_t pieces = (j.cols + 7) / 8;
        if (j.rows <= 0 || j.groups <= 0 || j.cols <= 0) continue;
        if (pieces > kMostPieces) return cudaErrorInvalidValue;
        const unsigned short* src = static_cast<const unsigned short*>(j.src);
        const bool apart = j.groups > 1 && j.gs_src != j.rows * j.ld_src;
        if (apart && a.count < kRepackJobs && total + j.rows * j.groups * pieces <= kMostPieces) {
            add(j, src, 0, j.rows, j.groups, j.gs_src);
            continue;
        }
        const int64_t runs = apart ? j.groups : 1, rows = apart ? j.rows : j.rows * j.groups;
        for (int64_t g = 0; g < runs; ++g) {
            for (int64_t r = 0; r < rows;) {
                const int64_t n = a.count < kRepackJobs ? std::min<int64_t>(rows - r, (kMostPieces - total) / pieces) : 0;
                if (n == 0) {
                    const cudaError_t e = launch();
                    if (e != cudaSuccess) return e;
                    continue;
                }
                add(j, src + g * j.gs_src + r * j.ld_src, g * rows + r, n, 1, 0);
                r += n;
            }
        }
    }
    return launch();
}

}  // namespace pf
