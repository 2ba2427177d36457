// Layers with few rows (a time step of a recurrent layer, generation, the smallest batches): forward on any
// layout, without re-pitch copies.
//
// With a few dozen rows the factors are the work: every element of U and V is read once and used m times, so the
// layer is bound by getting them through the SMs, and in practice by latencies: a tcgen05 tile of 128 rows pays
// its set-up, TMA round trips and slice sums (three launches, 18 us for 20 x 1500 -> 6000 at r 375) for rows
// that do not exist.  Here the factor takes the 128-row side of nothing: warps multiply 16 x 16 blocks of it by
// all m rows of the batch with mma.sync (m16n8k16, fp32 accumulation), which needs no descriptors, takes any
// alignment and starts as soon as its operands are in registers.
//   small_reduce_kernel   T[m, r] = A[m, K] B[K, r]     (A, B) = (x, U): long contraction, few outputs; a CTA owns 16
//                         columns of r and a cluster of CTAs shares the contraction (sum through distributed
//                         shared memory, in rank order).
//   small_out_kernel      y[m, n] = act(T[m, r] V[n, r]^T + bias): a CTA owns 32 rows of V, which it stages BEFORE
//                         waiting for the kernel that produces T (that kernel does not write V).
#include <cuda_bf16.h>

#include <algorithm>

#include "pf_tc.h"
#include "pf_tc_host.h"

namespace pf {
namespace small {
namespace {

constexpr int kThreads = 512;

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pair(unsigned short lo, unsigned short hi) { return lo | (static_cast<uint32_t>(hi) << 16); }

struct ReduceParams {
    const unsigned short *A, *B;     // bf16
    unsigned short* C;
    long long lda, ldb, ldc;
    int m, K, r;
    int k_per_rank;                  // multiple of 16
};

// kTiles: blocks of 8 batch rows.  kPairs: rows of A are 4-byte aligned and K is even.
template <int kTiles, bool kPairs>
__global__ void __launch_bounds__(kThreads) small_reduce_kernel(const ReduceParams p) {
    constexpr int kWarps = kThreads / 32;
    __shared__ float part[kWarps][16][kTiles * 8 + 1];
    __shared__ float sums[16][kTiles * 8 + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int r0 = blockIdx.x * 16;
    const int k_beg = blockIdx.y * p.k_per_rank, k_end = min(p.K, k_beg + p.k_per_rank);
    const int k_pair = p.K - 2;
    pdl_wait();
    pdl_launch_dependents();
    float acc[kTiles][4];
#pragma unroll
    for (int j = 0; j < kTiles; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[j][e] = 0.f;
    // loads are unconditional (addresses clamped, values masked afterwards)
    const unsigned short* bcol0 = p.B + min(r0 + g, p.r - 1);
    const unsigned short* bcol1 = p.B + min(r0 + g + 8, p.r - 1);
    const unsigned short* xrow[kTiles];
#pragma unroll
    for (int j = 0; j < kTiles; ++j) xrow[j] = p.A + static_cast<long long>(min(j * 8 + g, p.m - 1)) * p.lda;
#pragma unroll 1
    for (int k0 = k_beg + warp * 16; k0 < k_end; k0 += kWarps * 16) {
        uint32_t a[4], b[kTiles][2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = k0 + 2 * t + 8 * h;
            const int ka = min(k, k_end - 1), kb = min(k + 1, k_end - 1);
            // a0: (r g, k 2t, 2t+1), a1: (r g + 8, same k), a2 / a3: k + 8
            const unsigned short u0 = bcol0[ka * p.ldb], u1 = bcol0[kb * p.ldb], v0 = bcol1[ka * p.ldb], v1 = bcol1[kb * p.ldb];
#pragma unroll
            for (int j = 0; j < kTiles; ++j) {
                if constexpr (kPairs) b[j][h] = *reinterpret_cast<const uint32_t*>(xrow[j] + min(k, k_pair));
                else b[j][h] = pair(xrow[j][ka], xrow[j][kb]);
            }
            a[2 * h] = pair(u0, u1);
            a[2 * h + 1] = pair(v0, v1);
            // contraction past the end: zero on both sides (0 * Inf would not be zero)
            const uint32_t keep = (k < k_end ? 0xffffu : 0u) | (k + 1 < k_end ? 0xffff0000u : 0u);
            a[2 * h] &= keep;
            a[2 * h + 1] &= keep;
#pragma unroll
            for (int j = 0; j < kTiles; ++j) b[j][h] &= keep;
        }
#pragma unroll
        for (int j = 0; j < kTiles; ++j) mma16816(acc[j], a, b[j][0], b[j][1]);
    }
    // c0, c1: (r g, rows 2t, 2t + 1); c2, c3: r g + 8
#pragma unroll
    for (int j = 0; j < kTiles; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) part[warp][g + 8 * (e >> 1)][j * 8 + 2 * t + (e & 1)] = acc[j][e];
    __syncthreads();
    constexpr int kOut = 16 * kTiles * 8;
    for (int i = threadIdx.x; i < kOut; i += kThreads) {
        const int c = i & 15, row = i >> 4;
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) s += part[w][c][row];
        sums[c][row] = s;
    }
    const int ranks = gridDim.y;
    if (ranks > 1) {
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    } else {
        __syncthreads();
    }
    // each rank stores a share of the outputs: the sums of all ranks, added in rank order
    const int rank = blockIdx.y;
    for (int i = rank * kThreads + threadIdx.x; i < kOut; i += ranks * kThreads) {
        const int c = i & 15, row = i >> 4;
        float s = 0.f;
        if (ranks > 1) {
            const uint32_t local = static_cast<uint32_t>(__cvta_generic_to_shared(&sums[c][row]));
            for (int q = 0; q < ranks; ++q) {
                uint32_t addr;
                float v;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(local), "r"(q));
                asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
                s += v;
            }
        } else {
            s = sums[c][row];
        }
        if (row < p.m && r0 + c < p.r) p.C[row * p.ldc + r0 + c] = __bfloat16_as_ushort(__float2bfloat16_rn(s));
    }
    if (ranks > 1) {        // nobody leaves while its sums may still be read
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    }
}

// Copies `rows` rows of `cols` bf16 (any element alignment and pitch) into shared memory rows of `pitch` bytes (a
// multiple of 16), zero-filled to whole 16-byte pieces up to `pieces` per row.  Both sides move 16 bytes: a piece is
// assembled from the two aligned source vectors that cover it (each holds at least one of its bytes).
// Four pieces per thread at a time, loads before uses; one copy of the code for both operands (these kernels run for
// two or three microseconds, of which cold instructions are a part).
__device__ __noinline__ void stage_rows(uint8_t* dst, uint32_t pitch, int pieces, const unsigned short* src, long long ld, int rows, int cols) {
    constexpr int kBatch = 4;
    const int total = rows * pieces;
    for (int base = threadIdx.x; base < total; base += kBatch * kThreads) {
        uint4 lo[kBatch], hi[kBatch];
        uint32_t at[kBatch], sh[kBatch];
        int left_[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const int i = min(base + u * kThreads, total - 1);          // (a clamped piece is written twice, alike)
            const int row = i / pieces, pc = i - row * pieces, left = cols - pc * 8;
            const unsigned short* sp = src + row * ld + pc * 8;
            at[u] = static_cast<uint32_t>(row) * pitch + static_cast<uint32_t>(pc) * 16u;
            sh[u] = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(sp)) & 15u;
            lo[u] = hi[u] = make_uint4(0, 0, 0, 0);
            // aligned vectors that hold at least one byte of the piece (of what the row has of it)
            const uint4* v = reinterpret_cast<const uint4*>(reinterpret_cast<uintptr_t>(sp) - sh[u]);
            left_[u] = min(left, 8);
            if (left > 0) lo[u] = v[0];
            if (left > 0 && static_cast<int>(sh[u]) + 2 * left_[u] > 16) hi[u] = v[1];
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const uint32_t q = sh[u] >> 2, bit = (sh[u] & 3u) * 8u;
            const uint4 o = lo[u], h = hi[u];
            const bool q1 = q & 1, q2 = q & 2;
            // words q .. q + 4 of the window lo:hi
            const uint32_t x0 = q2 ? o.z : o.x, x1 = q2 ? o.w : o.y, x2 = q2 ? h.x : o.z, x3 = q2 ? h.y : o.w, x4 = q2 ? h.z : h.x, x5 = q2 ? h.w : h.y;
            const uint32_t w0 = q1 ? x1 : x0, w1 = q1 ? x2 : x1, w2 = q1 ? x3 : x2, w3 = q1 ? x4 : x3, w4 = q1 ? x5 : x4;
            uint4 r = make_uint4(__funnelshift_r(w0, w1, bit), __funnelshift_r(w1, w2, bit), __funnelshift_r(w2, w3, bit), __funnelshift_r(w3, w4, bit));
            if (left_[u] < 8) {            // zeros behind the row's end
                auto keep = [&](int e) { return (e < left_[u] ? 0xffffu : 0u) | (e + 1 < left_[u] ? 0xffff0000u : 0u); };
                r.x &= keep(0); r.y &= keep(2); r.z &= keep(4); r.w &= keep(6);
            }
            *reinterpret_cast<uint4*>(dst + at[u]) = r;
        }
    }
}

struct OutParams {
    const unsigned short *T, *V, *bias;
    unsigned short* y;
    long long ldt, ldv, ldy;
    int m, n, r, act;
    int steps;                       // 16-element steps of the contraction
    uint32_t pitch;                  // bytes of a staged row: 16 modulo 128, so that fragment loads do not conflict
};

// Sixteen warps: two blocks of 16 rows of V times eight parts of the contraction.
template <int kTiles>
__global__ void __launch_bounds__(kThreads) small_out_kernel(const OutParams p) {
    extern __shared__ uint4 smem4[];
    uint8_t* sV = reinterpret_cast<uint8_t*>(smem4);
    uint8_t* sT = sV + 32 * p.pitch;
    __shared__ float part[8][32][kTiles * 8 + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int n0 = blockIdx.x * 32, rows = min(32, p.n - n0);
    stage_rows(sV, p.pitch, p.steps * 2, p.V + n0 * p.ldv, p.ldv, rows, p.r);
    for (int i = threadIdx.x; i < (32 - rows) * p.steps * 2; i += kThreads)
        *reinterpret_cast<uint4*>(sV + (rows + i / (p.steps * 2)) * p.pitch + (i % (p.steps * 2)) * 16) = make_uint4(0, 0, 0, 0);
    pdl_wait();
    pdl_launch_dependents();
    stage_rows(sT, p.pitch, p.steps * 2, p.T, p.ldt, p.m, p.r);
    for (int i = threadIdx.x; i < (kTiles * 8 - p.m) * p.steps * 2; i += kThreads)
        *reinterpret_cast<uint4*>(sT + (p.m + i / (p.steps * 2)) * p.pitch + (i % (p.steps * 2)) * 16) = make_uint4(0, 0, 0, 0);
    __syncthreads();
    const int block = warp & 1, part_k = warp >> 1;
    float acc[kTiles][4];
#pragma unroll
    for (int j = 0; j < kTiles; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[j][e] = 0.f;
    const uint8_t* va = sV + (block * 16 + g) * p.pitch + t * 4;
    const uint8_t* tb = sT + g * p.pitch + t * 4;
#pragma unroll 1
    for (int s = part_k; s < p.steps; s += 8) {
        uint32_t a[4];
        a[0] = *reinterpret_cast<const uint32_t*>(va + s * 32);
        a[1] = *reinterpret_cast<const uint32_t*>(va + 8 * p.pitch + s * 32);
        a[2] = *reinterpret_cast<const uint32_t*>(va + s * 32 + 16);
        a[3] = *reinterpret_cast<const uint32_t*>(va + 8 * p.pitch + s * 32 + 16);
#pragma unroll
        for (int j = 0; j < kTiles; ++j) {
            const uint8_t* tj = tb + j * 8 * p.pitch + s * 32;
            mma16816(acc[j], a, *reinterpret_cast<const uint32_t*>(tj), *reinterpret_cast<const uint32_t*>(tj + 16));
        }
    }
#pragma unroll
    for (int j = 0; j < kTiles; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) part[part_k][block * 16 + g + 8 * (e >> 1)][j * 8 + 2 * t + (e & 1)] = acc[j][e];
    __syncthreads();
    const int c = lane;
    const bool in = n0 + c < p.n;
    const float b = p.bias && in ? __uint_as_float(static_cast<uint32_t>(p.bias[n0 + c]) << 16) : 0.f;
    for (int row = warp; row < p.m; row += kThreads / 32) {
        float v = part[0][c][row];
#pragma unroll
        for (int q = 1; q < 8; ++q) v += part[q][c][row];
        v += b;
        if (p.act == PF_ACT_RELU) v = fmaxf(v, 0.f);
        if (in) p.y[row * p.ldy + n0 + c] = __bfloat16_as_ushort(__float2bfloat16_rn(v));
    }
}

cudaError_t launch_reduce(void (*kernel)(const ReduceParams), dim3 grid, cudaStream_t stream, const ReduceParams& p) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = dim3(kThreads); cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1; attr[1].val.clusterDim.y = grid.y; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 2;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, p);
    if (e == cudaSuccess) count_launch();
    return e;
}

// Blocks of 8 batch rows that the kernels are compiled for.
int tiles_of(int64_t m) {
    const int t = static_cast<int>(ceil_div(m, 8));
    return t;
}
size_t out_smem(int64_t m, int64_t r) {
    const size_t row = static_cast<size_t>(ceil_div(r, 16)) * 32;
    return (32 + static_cast<size_t>(tiles_of(m)) * 8) * ((row + 111) / 128 * 128 + 16);
}

template <int kTiles>
int forward(const tc::LinearArgs& a, void* T, int64_t ldt) {
    ReduceParams q;
    q.A = static_cast<const unsigned short*>(a.x); q.B = static_cast<const unsigned short*>(a.U); q.C = static_cast<unsigned short*>(T);
    q.lda = a.ldx; q.ldb = a.ldu; q.ldc = ldt;
    q.m = static_cast<int>(a.m); q.K = static_cast<int>(a.k); q.r = static_cast<int>(a.r);
    const bool pairs = (reinterpret_cast<uintptr_t>(a.x) & 3) == 0 && a.ldx % 2 == 0 && a.k % 2 == 0;
    // as many ranks as keep at least one 16-element step per warp, while the grid fits the machine
    const int64_t blocks = ceil_div(a.r, 16);
    int ranks = 1;
    while (ranks < 8 && blocks * ranks * 2 <= num_sms() && a.k > 16 * (kThreads / 32) * ranks) ranks *= 2;
    q.k_per_rank = static_cast<int>(ceil_div(ceil_div(a.k, ranks), 16) * 16);
    if (launch_reduce(pairs ? small_reduce_kernel<kTiles, true> : small_reduce_kernel<kTiles, false>, dim3(static_cast<unsigned>(blocks), static_cast<unsigned>(ranks)), a.stream, q) != cudaSuccess) return PF_ERR_CUDA;
    OutParams o;
    o.T = static_cast<const unsigned short*>(T); o.V = static_cast<const unsigned short*>(a.V); o.bias = static_cast<const unsigned short*>(a.bias);
    o.y = static_cast<unsigned short*>(a.y);
    o.ldt = ldt; o.ldv = a.ldv; o.ldy = a.ldy;
    o.m = q.m; o.n = static_cast<int>(a.n); o.r = q.r; o.act = a.act;
    o.steps = static_cast<int>(ceil_div(a.r, 16));
    o.pitch = static_cast<uint32_t>((o.steps * 32 + 111) / 128 * 128 + 16);
    const size_t smem = out_smem(a.m, a.r);
    if (tc::allow_smem(small_out_kernel<kTiles>, 190 * 1024) != cudaSuccess ||
        tc::launch_overlapped(small_out_kernel<kTiles>, dim3(static_cast<unsigned>(ceil_div(a.n, 32))), dim3(kThreads), smem, a.stream, o) != cudaSuccess)
        return PF_ERR_CUDA;
    count_launch();
    return PF_OK;
}
}  // namespace

bool linear_fwd_fits(int64_t m, int64_t k, int64_t n, int64_t r) {
    // beyond about 2^26 multiplications the 128-row tiles win (4096 x 4096, r 256: 11.2 against 13.0 us at 20 rows, 15.0
    // against 13.1 at 32; caches warm), beyond 2^27 where they need re-pitch copies; up to 8 rows never
    const int64_t most = (k % 8 || r % 8) ? 1LL << 27 : 1LL << 26;
    return m >= 1 && m <= 32 && k <= (1 << 24) && n <= (1 << 24) && r <= (1 << 16) && out_smem(m, r) <= 190 * 1024 &&
           (m <= 8 || m * (k + n) * r < most);
}

// T [m, r]: the stash or scratch.
int linear_fwd(const tc::LinearArgs& a, void* T, int64_t ldt) {
    switch (tiles_of(a.m)) {
        case 1: return forward<1>(a, T, ldt);
        case 2: return forward<2>(a, T, ldt);
        case 3: return forward<3>(a, T, ldt);
        default: return forward<4>(a, T, ldt);
    }
}

// ------------------------------------------------------------------------------ fp32, small products
// The smallest fp32 layers (a few million multiplications per product) are all latency: the split-operand tensor-core
// kernel needs 6 us a launch for them (set-up, ring fill, splitting, drains).  Here a CTA computes a 16 x 32 tile of
// C with plain FMAs: all loads of 128 elements of the contraction are in flight at once, the next 128 while these
// are multiplied.  64 x 256 -> 256 at r 32, forward + backward: 25.8 -> 17.1 us (back to back, caches warm).
namespace {

constexpr int kF32Chunk = 128;
struct F32Product {
    const float *A, *B, *bias;
    float* C;
    long long a_row, a_l, b_l, b_col, ldc;      // A(i, l) = A[i a_row + l a_l], B(l, j) = B[l b_l + j b_col]
    int M, N, K, act, tiles_x;
};
struct F32Pair {
    F32Product p[2];
    int end0;
};

__global__ void __launch_bounds__(256) small_f32_kernel(const F32Pair both) {
    __shared__ float sA[16][kF32Chunk + 4];
    __shared__ float sB[kF32Chunk][34];
    const bool first = static_cast<int>(blockIdx.x) < both.end0;
    const F32Product& p = both.p[first ? 0 : 1];
    const int idx = blockIdx.x - (first ? 0 : both.end0);
    const int i0 = (idx % p.tiles_x) * 16, j0 = (idx / p.tiles_x) * 32, tid = threadIdx.x;
    pdl_wait();
    pdl_launch_dependents();
    // consecutive threads read consecutive addresses: along the contraction, or along the rows / columns
    const bool al = p.a_l == 1, bl = p.b_l == 1;
    const int ai = al ? tid >> 7 : tid & 15, ak = al ? tid & 127 : tid >> 4;
    const int bj = bl ? tid >> 7 : tid & 31, bk = bl ? tid & 127 : tid >> 5;
    const int ai_step = al ? 2 : 0, ak_step = al ? 0 : 16, bj_step = bl ? 2 : 0, bk_step = bl ? 0 : 8;
    float ra[8], rb[16];
    auto load = [&](int l0) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int i = i0 + ai + q * ai_step, l = l0 + ak + q * ak_step;
            ra[q] = i < p.M && l < p.K ? __ldg(p.A + i * p.a_row + l * p.a_l) : 0.f;
        }
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const int j = j0 + bj + q * bj_step, l = l0 + bk + q * bk_step;
            rb[q] = j < p.N && l < p.K ? __ldg(p.B + l * p.b_l + j * p.b_col) : 0.f;
        }
    };
    const int ti = tid >> 4, tj = (tid & 15) * 2;
    float c0 = 0.f, c1 = 0.f;
    load(0);
    for (int l0 = 0; l0 < p.K; l0 += kF32Chunk) {
#pragma unroll
        for (int q = 0; q < 8; ++q) sA[ai + q * ai_step][ak + q * ak_step] = ra[q];
#pragma unroll
        for (int q = 0; q < 16; ++q) sB[bk + q * bk_step][bj + q * bj_step] = rb[q];
        __syncthreads();
        if (l0 + kF32Chunk < p.K) load(l0 + kF32Chunk);
        const int left = min(kF32Chunk, p.K - l0);
#pragma unroll 4
        for (int l = 0; l < left; l += 4) {           // (zeros behind the end)
            const float4 a = *reinterpret_cast<const float4*>(&sA[ti][l]);
            const float2 b0 = *reinterpret_cast<const float2*>(&sB[l][tj]), b1 = *reinterpret_cast<const float2*>(&sB[l + 1][tj]);
            const float2 b2 = *reinterpret_cast<const float2*>(&sB[l + 2][tj]), b3 = *reinterpret_cast<const float2*>(&sB[l + 3][tj]);
            c0 = fmaf(a.x, b0.x, c0); c1 = fmaf(a.x, b0.y, c1);
            c0 = fmaf(a.y, b1.x, c0); c1 = fmaf(a.y, b1.y, c1);
            c0 = fmaf(a.z, b2.x, c0); c1 = fmaf(a.z, b2.y, c1);
            c0 = fmaf(a.w, b3.x, c0); c1 = fmaf(a.w, b3.y, c1);
        }
        __syncthreads();
    }
    const int i = i0 + ti, j = j0 + tj;
    if (i >= p.M) return;
    if (p.bias) {
        if (j < p.N) c0 += __ldg(p.bias + j);
        if (j + 1 < p.N) c1 += __ldg(p.bias + j + 1);
    }
    if (p.act == PF_ACT_RELU) { c0 = fmaxf(c0, 0.f); c1 = fmaxf(c1, 0.f); }
    float* dst = p.C + i * p.ldc + j;
    if (j < p.N) dst[0] = c0;
    if (j + 1 < p.N) dst[1] = c1;
}

F32Product f32_product(const void* A, int64_t a_row, int64_t a_l, const void* B, int64_t b_l, int64_t b_col, void* C, int64_t ldc, int64_t M,
                       int64_t N, int64_t K) {
    F32Product p = {};
    p.A = static_cast<const float*>(A); p.B = static_cast<const float*>(B); p.C = static_cast<float*>(C);
    p.a_row = a_row; p.a_l = a_l; p.b_l = b_l; p.b_col = b_col; p.ldc = ldc;
    p.M = static_cast<int>(M); p.N = static_cast<int>(N); p.K = static_cast<int>(K);
    p.tiles_x = static_cast<int>(ceil_div(M, 16));
    return p;
}
int f32_run(const F32Product& a, const F32Product* b, cudaStream_t stream) {
    F32Pair both{{a, b ? *b : a}, static_cast<int>(a.tiles_x * ceil_div(a.N, 32))};
    const unsigned blocks = static_cast<unsigned>(both.end0 + (b ? b->tiles_x * ceil_div(b->N, 32) : 0));
    if (tc::launch_overlapped(small_f32_kernel, dim3(blocks), dim3(256), 0, stream, both) != cudaSuccess) return PF_ERR_CUDA;
    count_launch();
    return PF_OK;
}
}  // namespace

// ------------------------------------------------------------------------------ the smallest layers in one launch each way
// Up to 128 rows, k and n up to 256, r up to 32: every launch is a start, a trip to memory and a few dozen FMAs per thread,
// so the intermediate is computed where it is needed instead of by a launch of its own.
//   forward (fp32)  a CTA computes T of its 16 rows, whole, and then its 16 x 32 tile of y.
//   backward        a cluster of CTAs, 16 rows each, computes G = dY V, exchanges it through distributed shared memory and
//                   computes 32 columns of dX and 32 rows of dU; other clusters compute tiles of dV.
// 1024 threads, so that a whole contraction is one trip to memory and a quarter of it per thread.  bf16 operands are widened
// as they are staged, T and G rounded to bf16 as everywhere.  What bounds them is latency.
// 64 x 256 -> 32 -> 256, fp32: forward 8.6 -> 5.8 us, backward 8.8 -> 8.2, training step 17.1 -> 13.7 with two launches less;
// 36 x 64 -> 16 -> 64, bf16: backward 6.3 -> 5.5.
namespace {

constexpr int kTinyThreads = 1024, kTinyRows = 128, kTinyWide = 256, kTinyRank = 32;

__device__ __forceinline__ float widen(float v) { return v; }
__device__ __forceinline__ float widen(unsigned short v) { return __uint_as_float(static_cast<uint32_t>(v) << 16); }
__device__ __forceinline__ float rounded(float v, float) { return v; }
__device__ __forceinline__ float rounded(float v, unsigned short) { return __bfloat162float(__float2bfloat16_rn(v)); }
__device__ __forceinline__ void put(float* p, float v) { *p = v; }
__device__ __forceinline__ void put(unsigned short* p, float v) { *p = __bfloat16_as_ushort(__float2bfloat16_rn(v)); }

// A matrix as a contraction reads it: element (i, l) at p[i * si + l * sl], zero outside rows x len.
template <typename E>
struct Side {
    const E* p;
    long long si, sl;
    int rows, len;
};

struct TinyTiles {
    float a[16][kTinyWide + 4];
    float b[kTinyWide][34];
    float part[4][16][34];
};
// Element (tid / 32, tid % 32) of a 16 x 32 tile of A B, in the first 512 threads.
template <typename E>
__device__ __forceinline__ float tiny_product(TinyTiles& s, const Side<E>& A, int i0, const Side<E>& B, int j0) {
    const int tid = threadIdx.x;
    // consecutive threads read consecutive addresses: along the contraction, or along the rows / columns
    const bool al = A.sl == 1, bl = B.sl == 1;
    const int ai = al ? tid >> 8 : tid & 15, ak = al ? tid & 255 : tid >> 4, ai_step = al ? 4 : 0, ak_step = al ? 0 : 64;
    const int bj = bl ? tid >> 8 : tid & 31, bk = bl ? tid & 255 : tid >> 5, bj_step = bl ? 4 : 0, bk_step = bl ? 0 : 32;
    E ra[4], rb[8];                                   // (widened afterwards: all loads come first)
    const E *pa = A.p + (i0 + ai) * A.si + ak * A.sl, *pb = B.p + (j0 + bj) * B.si + bk * B.sl;
    const long long sa = ai_step * A.si + ak_step * A.sl, sb = bj_step * B.si + bk_step * B.sl;
#pragma unroll
    for (int q = 0; q < 4; ++q, pa += sa) ra[q] = i0 + ai + q * ai_step < A.rows && ak + q * ak_step < A.len ? __ldg(pa) : E(0);
#pragma unroll
    for (int q = 0; q < 8; ++q, pb += sb) rb[q] = j0 + bj + q * bj_step < B.rows && bk + q * bk_step < B.len ? __ldg(pb) : E(0);
#pragma unroll
    for (int q = 0; q < 4; ++q) s.a[ai + q * ai_step][ak + q * ak_step] = widen(ra[q]);
#pragma unroll
    for (int q = 0; q < 8; ++q) s.b[bk + q * bk_step][bj + q * bj_step] = widen(rb[q]);
    __syncthreads();
    const int group = tid >> 8, ti = (tid & 255) >> 4, tj = (tid & 15) * 2, l0 = group * 64, left = min(64, A.len - l0);
    float c0 = 0.f, c1 = 0.f;
#pragma unroll 4
    for (int l = l0; l < l0 + left; l += 4) {         // (zeros behind the end)
        const float4 a = *reinterpret_cast<const float4*>(&s.a[ti][l]);
        const float2 b0 = *reinterpret_cast<const float2*>(&s.b[l][tj]), b1 = *reinterpret_cast<const float2*>(&s.b[l + 1][tj]);
        const float2 b2 = *reinterpret_cast<const float2*>(&s.b[l + 2][tj]), b3 = *reinterpret_cast<const float2*>(&s.b[l + 3][tj]);
        c0 = fmaf(a.x, b0.x, c0); c1 = fmaf(a.x, b0.y, c1);
        c0 = fmaf(a.y, b1.x, c0); c1 = fmaf(a.y, b1.y, c1);
        c0 = fmaf(a.z, b2.x, c0); c1 = fmaf(a.z, b2.y, c1);
        c0 = fmaf(a.w, b3.x, c0); c1 = fmaf(a.w, b3.y, c1);
    }
    s.part[group][ti][tj] = c0;
    s.part[group][ti][tj + 1] = c1;
    __syncthreads();
    const int row = (tid >> 5) & 15, col = tid & 31;
    return (s.part[0][row][col] + s.part[1][row][col]) + (s.part[2][row][col] + s.part[3][row][col]);
}

struct TinyFwd {
    const float *x, *U, *V, *bias;
    float *y, *T;                     // T: the stash or null
    long long ldx, ldu, ldv, ldy, ldt;
    int m, k, n, r, act;
};
struct TinyFwdSmem {
    TinyTiles s;
    float t[16][kTinyRank + 1], v[kTinyRank][33];
};
__global__ void __launch_bounds__(kTinyThreads) tiny_fwd_kernel(const __grid_constant__ TinyFwd p) {
    extern __shared__ __align__(16) uint8_t tiny_smem[];
    TinyFwdSmem& s = *reinterpret_cast<TinyFwdSmem*>(tiny_smem);
    const int tid = threadIdx.x, row = tid >> 5, col = tid & 31, i0 = blockIdx.x * 16, j0 = blockIdx.y * 32, j = j0 + col;
    pdl_wait();
    pdl_launch_dependents();
    const float v = j0 + row < p.n && col < p.r ? __ldg(p.V + (j0 + row) * p.ldv + col) : 0.f;      // in flight beside the first product
    const float bias = p.bias && j < p.n ? __ldg(p.bias + j) : 0.f;
    const float t = tiny_product(s.s, Side<float>{p.x, p.ldx, 1, p.m, p.k}, i0, Side<float>{p.U, 1, p.ldu, p.r, p.k}, 0);
    s.v[col][row] = v;
    if (tid < 512) {
        s.t[row][col] = t;
        if (p.T && blockIdx.y == 0 && i0 + row < p.m && col < p.r) p.T[(i0 + row) * p.ldt + col] = t;
    }
    __syncthreads();
    if (tid >= 512 || i0 + row >= p.m || j >= p.n) return;
    float c = 0.f;
#pragma unroll 8
    for (int l = 0; l < p.r; ++l) c = fmaf(s.t[row][l], s.v[l][col], c);
    c += bias;
    if (p.act == PF_ACT_RELU) c = fmaxf(c, 0.f);
    p.y[(i0 + row) * p.ldy + j] = c;
}

struct TinyBwd {
    const void *x, *U, *V, *dY, *T;
    void *dX, *dU, *dV;               // dX may be null
    long long ldx, ldu, ldv, lddy, ldt, lddx, lddu, lddv;
    int m, k, n, r;
    int ranks, k_clusters;            // CTAs of a cluster; clusters that compute dX and dU
    int grads_f32, accumulate;
};
struct TinyBwdSmem {
    TinyTiles s;
    float g[kTinyRows][kTinyRank + 1];
    float u[kTinyRank][33];           // rows j0 .. j0 + 31 of U, by rank
    float x[2][kTinyRows][17];        // 16 columns of x per half of the threads
};
template <typename E>
__device__ __forceinline__ void put_grad(const TinyBwd& p, void* grad, long long at, float v) {
    if (p.grads_f32) {
        float* d = static_cast<float*>(grad) + at;
        *d = p.accumulate ? *d + v : v;
    } else {
        E* d = static_cast<E*>(grad) + at;
        put(d, p.accumulate ? widen(*d) + v : v);
    }
}
template <typename E>
__global__ void __launch_bounds__(kTinyThreads) tiny_bwd_kernel(const __grid_constant__ TinyBwd p) {
    extern __shared__ __align__(16) uint8_t tiny_smem[];
    TinyBwdSmem& s = *reinterpret_cast<TinyBwdSmem*>(tiny_smem);
    const int tid = threadIdx.x, half = tid >> 9, row = (tid >> 5) & 15, col = tid & 31;
    const int cluster = blockIdx.x / p.ranks, rank = blockIdx.x - cluster * p.ranks;
    const E *x = static_cast<const E*>(p.x), *U = static_cast<const E*>(p.U), *V = static_cast<const E*>(p.V), *dY = static_cast<const E*>(p.dY);
    const bool with_k = cluster < p.k_clusters;
    if (with_k) asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");      // (waited for before G travels: every CTA runs by then)
    pdl_wait();
    pdl_launch_dependents();
    if (!with_k) {                    // tiles of dV = dY^T T
        const int i0 = ((cluster - p.k_clusters) * p.ranks + rank) * 16;
        if (i0 >= p.n) return;
        const float v = tiny_product(s.s, Side<E>{dY, 1, p.lddy, p.n, p.m}, i0, Side<E>{static_cast<const E*>(p.T), 1, p.ldt, p.r, p.m}, 0);
        if (half == 0 && i0 + row < p.n && col < p.r) put_grad<E>(p, p.dV, (i0 + row) * p.lddv + col, v);
        return;
    }
    const int i0 = rank * 16, j0 = cluster * 32;
    // dU's two tiles of 16 rows: both on one CTA, a half of the threads each, or one on each of the first two ranks
    const int tile = p.ranks == 1 ? half : half == 0 ? rank : 2, r0 = j0 + tile * 16;
    const bool with_u = tile < 2 && r0 < p.k;
    // in flight beside the first product: U's rows and x's columns
    const E ru = p.dX && j0 + (tid >> 5) < p.k && col < p.r ? __ldg(U + (j0 + (tid >> 5)) * p.ldu + col) : E(0);
    E rx[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int i = tid & 15, l = ((tid & 511) >> 4) + 32 * q;
        rx[q] = with_u && l < p.m && r0 + i < p.k ? __ldg(x + l * p.ldx + r0 + i) : E(0);
    }
    const float sum = tiny_product(s.s, Side<E>{dY, p.lddy, 1, p.m, p.n}, i0, Side<E>{V, 1, p.ldv, p.r, p.n}, 0);
    const float g = i0 + row < p.m ? rounded(sum, E()) : 0.f;         // (zero times an infinity of V is no zero)
    s.u[col][tid >> 5] = widen(ru);
    if (with_u)
#pragma unroll
        for (int q = 0; q < 4; ++q) s.x[half][((tid & 511) >> 4) + 32 * q][tid & 15] = widen(rx[q]);
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    const uint32_t local = static_cast<uint32_t>(__cvta_generic_to_shared(&s.g[i0 + row][col]));
    for (int to = half; to < p.ranks; to += 2) {
        uint32_t addr;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(local), "r"(to));
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(g) : "memory");
    }
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    if (p.dX && half == 1 && i0 + row < p.m && j0 + col < p.k) {       // dX = G U^T: this rank's rows, 32 columns
        float c = 0.f;
#pragma unroll 8
        for (int l = 0; l < p.r; ++l) c = fmaf(s.g[i0 + row][l], s.u[l][col], c);
        put(static_cast<E*>(p.dX) + (i0 + row) * p.lddx + j0 + col, c);
    }
    if (with_u && r0 + row < p.k && col < p.r) {      // dU = x^T G
        float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
        for (int l = 0; l < p.m; l += 4)              // (rows of G behind the batch are zero, and so is x)
#pragma unroll
            for (int e = 0; e < 4; ++e) c[e] = fmaf(s.x[half][l + e][row], s.g[l + e][col], c[e]);
        put_grad<E>(p, p.dU, (r0 + row) * p.lddu + col, (c[0] + c[1]) + (c[2] + c[3]));
    }
}
}  // namespace

// bf16 only up to a width of 128: the backward of 128 x 256 -> 32 -> 256 takes 10.4 us here, 7.1 in two launches on the tensor
// cores; of 100 x 250 -> 30 -> 130 8.0 and 10.6.
bool tiny_fits(int64_t m, int64_t k, int64_t n, int64_t r, int dtype) {
    const int wide = dtype == PF_BF16 ? kTinyWide / 2 : kTinyWide;
    return m >= 1 && m <= kTinyRows && k <= wide && n <= wide && r <= kTinyRank;
}
// The whole backward in one launch, T given; gradients in fp32 and / or accumulated directly.
int tiny_bwd(const tc::LinearArgs& a, int dtype, bool grads_f32, bool accumulate) {
    TinyBwd p;
    p.x = a.x; p.U = a.U; p.V = a.V; p.dY = a.dY; p.T = a.T; p.dX = a.dX; p.dU = a.dU; p.dV = a.dV;
    p.ldx = a.ldx; p.ldu = a.ldu; p.ldv = a.ldv; p.lddy = a.lddy; p.ldt = a.ldt; p.lddx = a.lddx; p.lddu = a.lddu; p.lddv = a.lddv;
    p.m = static_cast<int>(a.m); p.k = static_cast<int>(a.k); p.n = static_cast<int>(a.n); p.r = static_cast<int>(a.r);
    p.ranks = (p.m + 15) / 16;                      // at most 8, the largest portable cluster
    p.k_clusters = (p.k + 31) / 32;
    p.grads_f32 = grads_f32; p.accumulate = accumulate;
    const int v_tiles = (p.n + 15) / 16;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>((p.k_clusters + (v_tiles + p.ranks - 1) / p.ranks) * p.ranks)); cfg.blockDim = dim3(kTinyThreads);
    cfg.dynamicSmemBytes = sizeof(TinyBwdSmem); cfg.stream = a.stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = static_cast<unsigned>(p.ranks); attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 2;
    auto* kernel = dtype == PF_BF16 ? tiny_bwd_kernel<unsigned short> : tiny_bwd_kernel<float>;
    if (tc::allow_smem(kernel, sizeof(TinyBwdSmem)) != cudaSuccess || cudaLaunchKernelEx(&cfg, kernel, p) != cudaSuccess) return PF_ERR_CUDA;
    count_launch();
    return PF_OK;
}

// Every product short (its contraction in two loads) and small.  Beyond, the tensor cores are as fast or faster
// (128 x 512 -> 512, r 64: 13.7 + 15.2 against 13.4 + 15.4 us; 512 x 512 -> 512, r 32: 14.0 against 16.4;
// caches warm).
bool f32_fits(int64_t m, int64_t k, int64_t n, int64_t r, bool bwd) {
    const int64_t longest = std::max({k, r, bwd ? std::max(n, m) : int64_t{1}});
    return longest <= 256 && n <= 4096 && m <= 4096 && m * r * std::max(k, n) <= (1 << 21);
}
int f32_linear_fwd(const tc::LinearArgs& a, void* T, int64_t ldt) {
    if (!a.group_member && tiny_fits(a.m, a.k, a.n, a.r, PF_F32)) {
        TinyFwd p;
        p.x = static_cast<const float*>(a.x); p.U = static_cast<const float*>(a.U); p.V = static_cast<const float*>(a.V);
        p.bias = static_cast<const float*>(a.bias);
        p.y = static_cast<float*>(a.y); p.T = static_cast<float*>(a.T);
        p.ldx = a.ldx; p.ldu = a.ldu; p.ldv = a.ldv; p.ldy = a.ldy; p.ldt = a.ldt;
        p.m = static_cast<int>(a.m); p.k = static_cast<int>(a.k); p.n = static_cast<int>(a.n); p.r = static_cast<int>(a.r); p.act = a.act;
        const dim3 grid(static_cast<unsigned>(ceil_div(a.m, 16)), static_cast<unsigned>(ceil_div(a.n, 32)));
        if (tc::allow_smem(tiny_fwd_kernel, sizeof(TinyFwdSmem)) != cudaSuccess ||
            tc::launch_overlapped(tiny_fwd_kernel, grid, dim3(kTinyThreads), sizeof(TinyFwdSmem), a.stream, p) != cudaSuccess)
            return PF_ERR_CUDA;
        count_launch();
        return PF_OK;
    }
    const int st = f32_run(f32_product(a.x, a.ldx, 1, a.U, a.ldu, 1, T, ldt, a.m, a.r, a.k), nullptr, a.stream);
    if (st != PF_OK) return st;
    F32Product y = f32_product(T, ldt, 1, a.V, 1, a.ldv, a.y, a.ldy, a.m, a.n, a.r);
    y.bias = static_cast<const float*>(a.bias);
    y.act = a.act;
    return f32_run(y, nullptr, a.stream);
}
// T: the stash, or ws_T to have it recomputed there.
int f32_linear_bwd(const tc::LinearArgs& a) {
    const void* T = a.T ? a.T : a.ws_T;
    const int64_t ldt = a.T ? a.ldt : a.r;
    int st = PF_OK;
    if (!a.T) st = f32_run(f32_product(a.x, a.ldx, 1, a.U, a.ldu, 1, a.ws_T, a.r, a.m, a.r, a.k), nullptr, a.stream);
    if (st != PF_OK) return st;
    const F32Product dv = f32_product(a.dY, 1, a.lddy, T, ldt, 1, a.dV, a.lddv, a.n, a.r, a.m);
    st = f32_run(f32_product(a.dY, a.lddy, 1, a.V, a.ldv, 1, a.ws_G, a.r, a.m, a.r, a.n), &dv, a.stream);
    if (st != PF_OK) return st;
    const F32Product dx = f32_product(a.ws_G, a.r, 1, a.U, 1, a.ldu, a.dX, a.lddx, a.m, a.k, a.r);
    return f32_run(f32_product(a.x, 1, a.ldx, a.ws_G, a.r, 1, a.dU, a.lddu, a.k, a.r, a.m), a.dX ? &dx : nullptr, a.stream);
}

}  // namespace small
}  // namespace pf
