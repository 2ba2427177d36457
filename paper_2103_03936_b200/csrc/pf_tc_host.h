// Host-side helpers of the tensor-core path: TMA tensor-map encoding through the driver entry
// point (looked up at run time, so the library has no link-time dependency on libcuda).
#ifndef PF_TC_HOST_H_
#define PF_TC_HOST_H_

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>
#include <utility>

namespace pf {
namespace tc {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = [] {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return static_cast<EncodeTiledFn>(nullptr);
        return reinterpret_cast<EncodeTiledFn>(ptr);
    }();
    return fn;
}

// Encoding a tensor map costs a driver call of one to two microseconds, and a training step issues the
// same maps over and over, so encoded maps are kept in a small cache, one for each kind of map (the template is
// instantiated once for each `make`), keyed by everything the encoding depends on (the map holds no data, only
// addresses and shapes).  Four ways per set: a step uses some dozens of maps, and with a direct-mapped cache a
// colliding pair was encoded anew on every call.
struct MapKey {
    const void* p;
    int64_t v[8];
    bool operator==(const MapKey& o) const {
        bool same = p == o.p;
        for (int i = 0; i < 8; ++i) same = same && v[i] == o.v[i];
        return same;
    }
};
template <typename Make>
inline bool cached_map(CUtensorMap* map, const MapKey& key, Make make) {
    constexpr int kSets = 256, kWays = 4;
    struct Slot { MapKey key; CUtensorMap map; bool used; };
    struct Set { Slot way[kWays]; int next; };
    static Set sets[kSets];
    static std::mutex mu;
    uint64_t h = reinterpret_cast<uintptr_t>(key.p) * 0x9E3779B97F4A7C15ull;
    for (int i = 0; i < 8; ++i) h = (h ^ static_cast<uint64_t>(key.v[i])) * 0xC2B2AE3D27D4EB4Full;
    Set& set = sets[(h >> 40) % kSets];
    std::lock_guard<std::mutex> lock(mu);
    for (Slot& s : set.way)
        if (s.used && s.key == key) { *map = s.map; return true; }
    EncodeTiledFn fn = encode_fn();
    if (!fn || !make(fn)) return false;
    Slot& s = set.way[set.next];
    set.next = (set.next + 1) % kWays;
    s.key = key; s.map = *map; s.used = true;
    return true;
}
inline bool encode_bf16(EncodeTiledFn fn, CUtensorMap* map, const void* p, int rank, const cuuint64_t* dims, const cuuint64_t* strides,
                        const cuuint32_t* box, const cuuint32_t* estr) {
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, static_cast<cuuint32_t>(rank), const_cast<void*>(p), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 2-D bf16 tensor map over a row-major [rows, cols] matrix with row pitch ld (elements); boxes are
// 64 columns (128 bytes, the swizzle span) by box_rows rows; out-of-range elements read as zero.
inline bool cached_map_2d(CUtensorMap* map, const void* p, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
    return cached_map(map, MapKey{p, {rows, cols, ld, box_rows, -6, 0, 0, 0}}, [&](EncodeTiledFn fn) {
        const cuuint64_t dims[2] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows)};
        const cuuint64_t strides[1] = {static_cast<cuuint64_t>(ld) * 2};
        const cuuint32_t box[2] = {64u, static_cast<cuuint32_t>(box_rows)}, estr[2] = {1u, 1u};
        return encode_bf16(fn, map, p, 2, dims, strides, box, estr);
    });
}

// 3-D bf16 tensor map over `groups` row-major [rows, cols] matrices gs elements apart (boxes of 64 columns x
// box_rows rows of one group; out-of-range elements read as zero).  Cached like the 2-D maps.
inline bool cached_map_3d(CUtensorMap* map, const void* p, int64_t groups, int64_t rows, int64_t cols, int64_t ld, int64_t gs,
                   int box_rows) {
    if (groups < 1) return false;
    if (groups == 1) gs = rows * ld;                       // a single group: any valid stride
    if ((gs * 2) % 16 != 0 || gs * 2 >= (1LL << 40)) return false;
    return cached_map(map, MapKey{p, {groups, rows, cols, ld, gs, box_rows, -7, 0}}, [&](EncodeTiledFn fn) {
        const cuuint64_t dims[3] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows), static_cast<cuuint64_t>(groups)};
        const cuuint64_t strides[2] = {static_cast<cuuint64_t>(ld) * 2, static_cast<cuuint64_t>(gs) * 2};
        const cuuint32_t box[3] = {64u, static_cast<cuuint32_t>(box_rows), 1u}, estr[3] = {1u, 1u, 1u};
        return encode_bf16(fn, map, p, 3, dims, strides, box, estr);
    });
}

// 4-D bf16 tensor map over an NHWC image [N, H, W, C]: boxes are 64 channels x box_w x box_h pixels of box_n
// images (box_w * box_h * box_n rows of 128 bytes in shared memory, pixel-major), taking every stride-th
// pixel along W and H; ld: elements from one pixel to the next (0: C); coordinates may start outside the image (zero padding of the convolution),
// out-of-range pixels, channels and images read as zero.
inline bool cached_map_nhwc(CUtensorMap* map, const void* p, int64_t N, int64_t H, int64_t W, int64_t C, int box_w, int box_h,
                            int box_n, int stride, int64_t ld = 0) {
    if (ld == 0) ld = C;
    return cached_map(map, MapKey{p, {N, H, W, C, ld, box_w, box_h * 4096LL + box_n, stride}}, [&](EncodeTiledFn fn) {
        const cuuint64_t dims[4] = {static_cast<cuuint64_t>(C), static_cast<cuuint64_t>(W), static_cast<cuuint64_t>(H),
                                    static_cast<cuuint64_t>(N)};
        const cuuint64_t strides[3] = {static_cast<cuuint64_t>(ld) * 2, static_cast<cuuint64_t>(W) * ld * 2,
                                       static_cast<cuuint64_t>(H) * W * ld * 2};
        // box extents are given in traversed elements, i.e. times the stride
        const cuuint32_t box[4] = {64u, static_cast<cuuint32_t>(box_w * stride), static_cast<cuuint32_t>(box_h * stride),
                                   static_cast<cuuint32_t>(box_n)};
        const cuuint32_t estr[4] = {1u, static_cast<cuuint32_t>(stride), static_cast<cuuint32_t>(stride), 1u};
        return encode_bf16(fn, map, p, 4, dims, strides, box, estr);
    });
}

// 3-D view of a contiguous [planes][rows][cols] tensor with boxes of 64 columns x box_rows rows of one plane:
// a box that reaches past the rows of its plane reads zeros (or is clipped) instead of running into the
// next.  plane_step, in rows, is the distance between planes: `rows` for the factor of a convolution
// (planes = taps), less for overlapping windows (the output tiles of a convolution, one window per
// image row, so that a tile may start at any row and is clipped at its own end).
inline bool cached_map_planes(CUtensorMap* map, const void* p, int64_t planes, int64_t rows, int64_t cols, int64_t plane_step,
                              int box_rows, int64_t ld = 0) {
    if (ld == 0) ld = cols;
    return cached_map(map, MapKey{p, {planes, rows, cols, plane_step, box_rows, ld, -1, -1}}, [&](EncodeTiledFn fn) {
        const cuuint64_t dims[3] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows), static_cast<cuuint64_t>(planes)};
        const cuuint64_t strides[2] = {static_cast<cuuint64_t>(ld) * 2, static_cast<cuuint64_t>(plane_step) * ld * 2};
        const cuuint32_t box[3] = {64u, static_cast<cuuint32_t>(box_rows), 1u};
        const cuuint32_t estr[3] = {1u, 1u, 1u};
        return encode_bf16(fn, map, p, 3, dims, strides, box, estr);
    });
}

// Raises a kernel's dynamic shared memory limit, once per kernel and device.
template <typename... KArgs>
inline cudaError_t allow_smem(void (*kernel)(KArgs...), size_t bytes) {
    struct Done { void (*k)(KArgs...); bool dev[64]; };
    constexpr int kKernels = 16;
    static Done done[kKernels];
    static std::mutex mu;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lock(mu);
    for (Done& d : done) {
        if (d.k != nullptr && d.k != kernel) continue;
        if (d.k == kernel && dev >= 0 && dev < 64 && d.dev[dev]) return cudaSuccess;
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
        if (e == cudaSuccess && dev >= 0 && dev < 64) { d.k = kernel; d.dev[dev] = true; }
        return e;
    }
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
}

// Launch with programmatic stream serialization: the kernel's prologue (barrier set-up, TMEM
// allocation, descriptor prefetch) overlaps the tail of the previous kernel in the stream; the
// kernel itself calls griddepcontrol.wait before it touches global memory.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_overlapped(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                     Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

inline bool tma_ok(const void* p, int64_t ld) {
    return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && (ld % 8) == 0 && ld * 2 < (1LL << 40);
}
// A matrix of the caller's that TMA may store: a store fills the 16-byte piece that a row ends in with zeros, so the rows have to
// end with a piece (loads read zeros behind the last column, whatever lies there).  Rows that do not take the unfused products,
// which store single elements: 8192 x 512 -> 128 -> 2044 at a pitch of 2048: 13.1 -> 22.0 us.
inline bool tma_out(const void* p, int64_t ld, int64_t cols) { return tma_ok(p, ld) && cols % 8 == 0; }


}  // namespace tc
}  // namespace pf
#endif
