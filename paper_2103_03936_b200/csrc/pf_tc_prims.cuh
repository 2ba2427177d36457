// Device-side primitives for the sm_100a tensor-core path: mbarriers with bounded waits, TMA
// tile loads, tensor-memory (TMEM) allocation, tcgen05 MMA issue / commit / accumulator loads,
// and the shared-memory matrix descriptors of the 128-byte-swizzled canonical layouts.
#ifndef PF_TC_PRIMS_CUH_
#define PF_TC_PRIMS_CUH_

#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace pf {
namespace tc {

constexpr unsigned int kStatusTimeout = 5;               // == PF_ERR_TIMEOUT
constexpr long long kWaitCycleLimit = 4000000000LL;      // about two seconds of SM clocks

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ bool elect_one() {
    uint32_t pred;
    asm volatile(
        "{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(pred));
    return pred != 0;
}

// ---------------------------------------------------------------- programmatic dependent launch
// A kernel launched with programmatic stream serialization may start while its predecessor in the
// stream is still running; pdl_wait() blocks until that predecessor has completed and its writes
// are visible (a no-op for an ordinary launch), pdl_launch_dependents() lets the successor start
// its own prologue early.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// Operands of a product that were complete before the preceding kernel of the stream got past its own wait, i.e. that
// neither that kernel writes nor a caller's kernel before it can still be writing: their producers do not wait for it.  Never in a
// call's first launch, which knows nothing of the kernel before.  Two kinds of blocks let their successor start without having waited: those
// of a product marked `independent` (others of its launch do wait, so the launch as a whole is like any) and the second half of the
// groups of a grouped forward (ChainParams::group_flags[1]).  Behind that half an operand is early only if it was complete before
// the first half got past its wait; today nothing in a call follows it.  (tests/host/launches.cu checks all this over drawn calls.)
constexpr int kEarlyA = 1, kEarlyB = 2;

// ---------------------------------------------------------------- mbarrier
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_barrier_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait: gives up after kWaitCycleLimit clocks (or as soon as another thread of the CTA
// has given up), records PF_ERR_TIMEOUT in the device status word and returns false; the caller
// then leaves its loop and falls through to the common teardown.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag,
                                          unsigned int* status) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
#pragma unroll 1
    for (uint32_t it = 1;; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 255u) == 0u) {
            if (*abort_flag) return false;
            if (clock64() - t0 > kWaitCycleLimit) break;
        }
    }
    *abort_flag = 1u;
    if (status) atomicExch(status, kStatusTimeout);
    return false;
}

// The same wait for a whole (converged) warp: lane 0 polls and broadcasts the verdict, so the
// barrier word is not hammered by 32 pollers and the warp leaves the wait converged (the
// elect.sync that usually follows needs all 32 lanes).
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag,
                                               unsigned int* status) {
    uint32_t ok = 1;
    if ((threadIdx.x & 31) == 0) ok = mbar_wait(bar, parity, abort_flag, status) ? 1u : 0u;
    return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

// ---------------------------------------------------------------- TMA
__device__ __forceinline__ void tma_prefetch_desc(const CUtensorMap* m) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(m) : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0,
                                            int c1) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1)
        : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0,
                                            int c1, int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}

// How L2 treats what a kernel streams through it: kL2Stream = first to go (an operand read for the last time or an output,
// both of more bytes than L2 holds), a fraction in (0, 1] = so much of it is kept (read again by the next launch), 0 = as ever.
constexpr float kL2Stream = -1.f;
constexpr double kL2Bytes = 126.0 * (1 << 20);      // of a B200
__device__ __forceinline__ uint64_t l2_policy(float keep) {
    uint64_t p;
    if (keep > 0.f) asm volatile("createpolicy.fractional.L2::evict_last.L2::evict_first.b64 %0, %1;" : "=l"(p) : "f"(keep));
    else if (keep < 0.f) asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    else asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "l"(policy)
        : "memory");
}

// Ask L2 to fetch one tile of a tensor (no shared-memory destination, no completion to wait for).
__device__ __forceinline__ void tma_prefetch_l2_2d(const CUtensorMap* map, int c0, int c1) {
    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(map), "r"(c0), "r"(c1)
                 : "memory");
}
__device__ __forceinline__ void tma_prefetch_l2_3d(const CUtensorMap* map, int c0, int c1, int c2) {
    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(map), "r"(c0), "r"(c1), "r"(c2)
                 : "memory");
}
// Shared -> global tile store (bulk async group); rows/columns outside the tensor are clipped.
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int c0, int c1) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                 ::"l"(map), "r"(src), "r"(c0), "r"(c1)
                 : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int c0, int c1, uint64_t policy) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group.L2::cache_hint [%0, {%2, %3}], [%1], %4;"
                 ::"l"(map), "r"(src), "r"(c0), "r"(c1), "l"(policy)
                 : "memory");
}
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, uint32_t src, int c0, int c1, int c2) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];"
                 ::"l"(map), "r"(src), "r"(c0), "r"(c1), "r"(c2)
                 : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// Wait until at most N of this thread's bulk groups still have shared-memory reads pending.
template <int N>
__device__ __forceinline__ void tma_store_wait_read() {
    asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint4 v) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
}

__device__ __forceinline__ uint4 ld_shared_v4(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}

// ---------------------------------------------------------------- TMEM
__device__ __forceinline__ void tmem_alloc(uint32_t smem_result, uint32_t ncols) {  // whole warp
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_result), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {  // whole warp
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// Arrive on an mbarrier once all tcgen05.mma issued so far by this thread have completed.
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}

// D[tmem] (+)= A[smem] * B[smem], bf16 inputs, fp32 accumulate, one CTA.
__device__ __forceinline__ void tc_mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// The same with the descriptors as words: a step along an operand changes the low one only (address and LBO; shared memory ends below
// its 14 bits of address), so loops carry that and the issuing thread adds 32 bits per operand.
__device__ __forceinline__ uint32_t desc_lo(uint64_t desc) { return static_cast<uint32_t>(desc); }
__device__ __forceinline__ uint32_t desc_hi(uint64_t desc) { return static_cast<uint32_t>(desc >> 32); }
__device__ __forceinline__ void tc_mma_bf16_words(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi, uint32_t idesc,
                                                  uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n .reg .b64 a, b;\n mov.b64 a, {%1, %2};\n mov.b64 b, {%3, %4};\n setp.ne.b32 p, %6, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, p;\n}\n"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
        : "memory");
}

// The same with A in tensor memory (row = lane, two bf16 contraction elements per 32-bit column).
__device__ __forceinline__ void tc_mma_bf16_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// 32 lanes x 8 consecutive columns: thread t of the warp writes row (lane base + t).
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&v)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(v[0]), "r"(v[1]),
                 "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t ld_shared_u32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}

// Counters in global memory through which blocks report finished work: the report makes what its thread has written, and
// what it has seen written (its warp's writes before a __syncwarp), visible to whoever reads it with the acquire load.
__device__ __forceinline__ void red_release_gpu(unsigned int* p, unsigned int v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned int ld_acquire_gpu(const unsigned int* p) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// 32 lanes x 32 consecutive fp32 columns: thread t of the warp receives row (lane base + t).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr)
        : "memory");
}
// 32 lanes x 16 consecutive columns.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// ---------------------------------------------------------------- descriptors
// Shared-memory matrix descriptor, 128-byte swizzle, descriptor version 1 (sm_100).
//   K-major operand (rows = M or N index, 64 contraction elements = 128 bytes per row):
//       8-row groups are 1024 bytes apart (SBO); LBO is fixed by the swizzle (encoded 1).
//   MN-major operand (rows = contraction index, 64 M/N elements = 128 bytes per row):
//       8-row groups (8 contraction steps) are 1024 bytes apart (SBO); the next 64 M/N
//       elements start LBO bytes further.
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
    uint64_t d = 0;
    d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
    d |= static_cast<uint64_t>((lbo_bytes >> 4) & 0x3FFFu) << 16;
    d |= static_cast<uint64_t>((sbo_bytes >> 4) & 0x3FFFu) << 32;
    d |= static_cast<uint64_t>(1) << 46;
    d |= static_cast<uint64_t>(2) << 61;
    return d;
}
// Instruction descriptor for kind::f16: bf16 x bf16 -> fp32, M x N tile, operand majors.
__host__ __device__ constexpr uint32_t make_idesc_bf16(int M, int N, int a_mn_major, int b_mn_major) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(a_mn_major) << 15) |
           (static_cast<uint32_t>(b_mn_major) << 16) | (static_cast<uint32_t>(N >> 3) << 17) |
           (static_cast<uint32_t>(M >> 4) << 24);
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

// Results whose rows TMA and 16-byte stores cannot take (any pitch, any alignment): a warp stages 32 rows x 64 columns as
// words, 33 to a row (free of bank conflicts both ways), and stores each row's whole 16-byte pieces of the DESTINATION,
// assembled from five words with a funnel shift, four rows to an instruction; what is left of a row in front and behind is
// stored by elements.  (One pair of columns per lane, a row per instruction: 700 x 1504 over 376, rows of even pitch 8.0 us,
// of odd pitch 8.7; this way 7.0 and 7.1, against 6.0 with 16-byte stores.)
constexpr int kRaggedWords = 33;
__device__ __forceinline__ void stage_ragged(uint32_t* stg, const uint32_t (&v0)[32], const uint32_t (&v1)[32], int lane) {
#pragma unroll
    for (int w = 0; w < 16; ++w) {
        stg[lane * kRaggedWords + w] = pack_bf16x2(__uint_as_float(v0[2 * w]), __uint_as_float(v0[2 * w + 1]));
        stg[lane * kRaggedWords + 16 + w] = pack_bf16x2(__uint_as_float(v1[2 * w]), __uint_as_float(v1[2 * w + 1]));
    }
}
// `row_of(r)`: row of C that staged row r goes to, negative = none; columns col0 .. col0 + 63, clipped at n.
template <typename RowOf>
__device__ __forceinline__ void store_ragged(const uint32_t* stg, __nv_bfloat16* C, long long ldc, int col0, int n, int lane, RowOf row_of) {
    const int p = lane & 7, count = min(64, n - col0);
#pragma unroll 2
    for (int i = 0; i < 8; ++i) {
        const int r = i * 4 + (lane >> 3), row = row_of(r);
        if (row < 0) continue;
        unsigned short* d = reinterpret_cast<unsigned short*>(C) + static_cast<long long>(row) * ldc + col0;
        const uint32_t* words = stg + r * kRaggedWords;
        const unsigned short* elems = reinterpret_cast<const unsigned short*>(words);
        const int head = static_cast<int>((0u - static_cast<uint32_t>(reinterpret_cast<uintptr_t>(d))) & 15u) >> 1;     // elements before the first whole piece
        const int e = head + 8 * p;
        if (e + 8 <= count) {
            const uint32_t* w = words + (e >> 1);
            const uint32_t bit = (e & 1) * 16;
            const uint32_t w0 = w[0], w1 = w[1], w2 = w[2], w3 = w[3], w4 = w[4];       // (the last one may be the row's padding word)
            *reinterpret_cast<uint4*>(d + e) = make_uint4(__funnelshift_r(w0, w1, bit), __funnelshift_r(w1, w2, bit), __funnelshift_r(w2, w3, bit),
                                                          __funnelshift_r(w3, w4, bit));
        }
        if (p < min(head, count)) d[p] = elems[p];
        const int t = count > head ? head + ((count - head) & ~7) + p : count;
        if (t < count) d[t] = elems[t];
    }
}

// Bias and activation (1 = max(0, .)) on 64 accumulator columns col .. col + 63 of a row, before the rounding: every
// lane fetches two of the columns' values (bf16), the columns take them from the lanes.
__device__ __forceinline__ void bias_act64(uint32_t (&v0)[32], uint32_t (&v1)[32], const void* bias, int act, int col, int n, int lane) {
    if (bias) {
        const unsigned short* b = reinterpret_cast<const unsigned short*>(bias);
        const float b0 = col + lane < n ? __uint_as_float(static_cast<uint32_t>(b[col + lane]) << 16) : 0.f;
        const float b1 = col + 32 + lane < n ? __uint_as_float(static_cast<uint32_t>(b[col + 32 + lane]) << 16) : 0.f;
#pragma unroll
        for (int e = 0; e < 32; ++e) {
            v0[e] = __float_as_uint(__uint_as_float(v0[e]) + __shfl_sync(0xffffffffu, b0, e));
            v1[e] = __float_as_uint(__uint_as_float(v1[e]) + __shfl_sync(0xffffffffu, b1, e));
        }
    }
    if (act == 1) {
#pragma unroll
        for (int e = 0; e < 32; ++e) {
            v0[e] = __float_as_uint(fmaxf(__uint_as_float(v0[e]), 0.f));
            v1[e] = __float_as_uint(fmaxf(__uint_as_float(v1[e]), 0.f));
        }
    }
}

}  // namespace tc
}  // namespace pf
#endif
