// What a call of the library launches, looked over on the host (see runtime.cpp): every tensor map that is encoded and every
// matrix and slice buffer that a launched kernel is given has to lie inside one of the buffers of the call (host_regions)
// or inside a device array of the library, and an operand that is read ahead of the launch before (kEarlyA) outside what that one writes;
// what does not is reported by host_faults.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <map>
#include <string>
#include <vector>

#include "pf_tc.h"
#define kMaxStages kChainMaxStages      // (each of the two headers has one of its own)
#include "pf_tc_chain_kernel.cuh"
#undef kMaxStages
#include "pf_tc_conv_flat.cuh"
#include "pf_tc_f32_kernel.cuh"
#include "pf_tc_gemm_kernel.cuh"
#include "pf_tc_pair_launch.h"

namespace {
struct Range {
    uint64_t base, bytes;
};
std::vector<Range> regions, written;      // `written`: what the products of the launch in hand write
// What may still be being written when that launch starts: by the launch before, and, behind one that lets its successor start
// without having waited itself, by what that one ran beside.
std::vector<Range> before;
bool before_known = false;                // (not behind the launches of another call, nor behind a kernel that is not looked over)
std::map<const void*, std::string>& kernels() { static std::map<const void*, std::string> m; return m; }
std::map<const void*, Range>& arrays() { static std::map<const void*, Range> m; return m; }      // by host symbol
std::string faults, launches;

uint64_t address(const void* p) { return reinterpret_cast<uint64_t>(p); }
// [base, base + bytes) has to lie inside one buffer.
void inside(const std::string& what, uint64_t base, uint64_t bytes) {
    auto holds = [&](const Range& r) { return base >= r.base && base + bytes <= r.base + r.bytes; };
    if (bytes == 0 || std::any_of(regions.begin(), regions.end(), holds)) return;
    for (const auto& a : arrays())
        if (holds(a.second)) return;
    uint64_t past = 0;
    for (const Range& r : regions)
        if (base >= r.base && base <= r.base + r.bytes) past = base + bytes - (r.base + r.bytes);
    faults += what + ": " + std::to_string(bytes) + " bytes, " + (past ? std::to_string(past) + " of them past the end of their buffer\n" : "in no buffer\n");
}
// ... and what the products of one launch write there may not overlap.
void writes(const std::string& what, uint64_t base, uint64_t bytes) {
    inside(what, base, bytes);
    for (const Range& w : written)
        if (base < w.base + w.bytes && w.base < base + bytes) faults += what + ": overlaps what another product of the launch writes\n";
    written.push_back(Range{base, bytes});
}
uint64_t matrix(int64_t rows, int64_t cols, int64_t ld, int64_t size) { return rows > 0 ? static_cast<uint64_t>(((rows - 1) * ld + cols) * size) : 0; }

void check(const pf::tc::GemmParams& p) {
    const int splits = p.splits < 1 ? 1 : p.splits, groups = p.groups < 1 ? 1 : p.groups;
    if (p.partial) writes("slices of a product", address(p.partial), static_cast<uint64_t>(p.tiles_x) * p.tiles_y * groups * splits * 128 * p.bn * 4);
    if (splits > 1 && !p.partial) faults += "a split product without slices\n";
    if (p.partial && splits == 1) return;
    for (int g = 0; g < groups; ++g) {
        if (p.conv_mode != 1) writes("result of a product", address(p.C) + static_cast<uint64_t>(g) * p.c_gstride * 2, matrix(p.M, p.N, p.ldc, 2));
        if (p.C2) writes("second copy of a result", address(p.C2) + static_cast<uint64_t>(g) * p.c2_gstride * 2, matrix(p.M, p.N, p.ldc2, 2));
    }
}
void check(const pf::tc::F32Params& p) {
    if (p.splits > 1) writes("slices of an fp32 product", address(p.partial), static_cast<uint64_t>(p.tiles_x) * p.tiles_y * p.splits * 128 * p.bn * 4);
    const bool whole = p.mode == 0 || p.mode == 2;      // (else the pixels of the images)
    if (whole || p.splits <= 1) writes("result of an fp32 product", address(p.C), matrix(whole ? p.M : static_cast<int64_t>(p.cv_N) * p.out_h * p.out_w, p.N, p.ldc, 4));
    if (p.C2) writes("second copy of an fp32 result", address(p.C2), matrix(p.M, p.N, p.ldc2, 4));
}
constexpr uint64_t kSlice = 128 * 64 * 4;
void check(const pf::tc::DtDvParams& p, unsigned blocks) {
    writes("dT of a convolution", address(p.dT), matrix(p.rows, p.R, p.ldt, 2));
    writes("slices of dV of a convolution", address(p.partial), p.pairs * blocks * kSlice);
}
void check(const pf::tc::DuParams& p) {
    writes("slices of dU of a convolution", address(p.partial), static_cast<uint64_t>(6 * p.split[0] + 3 * p.split[1]) * p.tb * kSlice);
    writes("dV of a convolution", address(p.sum.out), matrix(p.sum.rows, p.sum.R, p.sum.R, p.sum.f32 ? 4 : 2));
}
void check(const pf::tc::DxParams& p) {
    if (p.tiles > 0) writes("dX of a convolution", address(p.out), matrix(static_cast<int64_t>(p.f.N) * p.f.H * p.f.W, p.C, p.C, 2));
    writes("dU of a convolution", address(p.sum.out), matrix(static_cast<int64_t>(9) * p.sum.rows, p.sum.R, p.sum.R, p.sum.f32 ? 4 : 2));
}
void check(const pf::SimtGemm& g) {
    const int64_t size = g.dtype == PF_BF16 ? 2 : 4;
    if (g.splits > 1) inside("slices of an FMA product", address(g.partial), static_cast<uint64_t>(g.splits) * g.M * g.N * 4);
    inside("result of an FMA product", address(g.C), matrix(g.M, g.N, g.ldc, size));
}

// What the recorded maps hold: where the matrix lies, the bytes of its rows and of all of it.
struct MapNote {
    uint64_t base, row_bytes, bytes;
};
void early(const char* what, const CUtensorMap& map) {
    const MapNote& n = reinterpret_cast<const MapNote&>(map);
    if (!before_known) faults += std::string(what) + ": read ahead of a launch that may write it\n";
    for (const Range& w : before)
        if (n.base < w.base + w.bytes && w.base < n.base + n.bytes) faults += std::string(what) + ": read ahead of the launch that writes it\n";
}
void early(int which, const CUtensorMap& a, const CUtensorMap& b) {
    if (which & pf::tc::kEarlyA) early("first operand", a);
    if (which & pf::tc::kEarlyB) early("second operand", b);
}
int early_of(const pf::tc::GemmParams& p) { return p.independent ? pf::tc::kEarlyA | pf::tc::kEarlyB : p.early; }
// A matrix that TMA stores: it fills the last 16-byte piece of a row, so unless it lies in the workspace (the last buffer) its rows
// end with one.
void stored(const char* what, const CUtensorMap& map) {
    const MapNote& n = reinterpret_cast<const MapNote&>(map);
    const bool in_workspace = !regions.empty() && n.base >= regions.back().base && n.base < regions.back().base + regions.back().bytes;
    writes(what, n.base, n.bytes);
    if (n.row_bytes % 16 != 0 && !in_workspace && n.base < (1ull << 60)) faults += std::string(what) + ": the store fills pieces behind the ends of the rows\n";
}

template <typename T>
const T& arg(void** args, int i) { return *static_cast<const T*>(args[i]); }
void launched(const void* kernel, unsigned blocks, void** args) {
    const std::string& name = kernels()[kernel];
    auto is = [&](const char* n) { return name.find(n) != std::string::npos; };
    launches += name + "\n";
    written.clear();
    bool known = true, late = false;
    if (is("tc_gemm3_kernel")) {
        const int end0 = arg<int>(args, 9), end1 = arg<int>(args, 10);
        check(arg<pf::tc::GemmParams>(args, 6));
        if (end1 > end0) check(arg<pf::tc::GemmParams>(args, 7));
        if (static_cast<int>(blocks) > end1) check(arg<pf::tc::GemmParams>(args, 8));
        const int ends[4] = {0, end0, end1, static_cast<int>(blocks)};
        for (int i = 0; i < 3; ++i)
            if (ends[i + 1] > ends[i]) early(early_of(arg<pf::tc::GemmParams>(args, 6 + i)), arg<CUtensorMap>(args, 2 * i), arg<CUtensorMap>(args, 2 * i + 1));
    } else if (is("tc_gemm_kernel")) {
        const pf::tc::GemmParams& p = arg<pf::tc::GemmParams>(args, 2);
        check(p);
        early(early_of(p), arg<CUtensorMap>(args, 0), arg<CUtensorMap>(args, 1));
        late = p.independent;
    } else if (is("tc_gemm_pair_kernel")) {
        const pf::tc::PairLaunch& l = arg<pf::tc::PairLaunch>(args, 0);
        for (int i = 0; i < l.count; ++i) {
            const pf::tc::PairProduct& p = l.p[i];
            const int outputs = p.kb_per_group > 0 ? 1 : p.tiles_mn > 0 ? p.tiles / p.tiles_mn : 1;
            for (int g = 0; g < outputs; ++g) writes("result of a product on pairs", address(p.C) + static_cast<uint64_t>(g) * p.c_gstride * 2, matrix(p.M, p.N, p.ldc, 2));
            early(p.early, l.ta[i], l.tb[i]);
        }
    } else if (is("repack_multi_kernel")) {
        const pf::RepackBatchArgs& a = arg<pf::RepackBatchArgs>(args, 0);
        for (int j = 0; j < a.count; ++j)
            writes("copy", address(a.dst[j]), matrix((a.item_end[j] - (j > 0 ? a.item_end[j - 1] : 0u)) / a.pieces_per_row[j], a.pieces_per_row[j] * 8, a.ld_dst[j], 2));
    } else if (is("tc_chain_kernel") || is("tc_chain_pipe_kernel")) {
        const pf::tc::ChainParams& p = arg<pf::tc::ChainParams>(args, 5);
        if (p.tiles_per_split > 0) stored("output of the fused kernel", arg<CUtensorMap>(args, 3));
        if (p.store_T) stored("intermediate of the fused kernel", arg<CUtensorMap>(args, 4));
        late = is("Li3E") && p.group_flags[1];
    } else if (is("tc_f32_kernel")) {
        const pf::tc::F32Launch& l = arg<pf::tc::F32Launch>(args, 0);
        for (int i = 0; i < 3; ++i)
            if (i == 0 || l.end[i] > l.end[i - 1]) {
                check(l.p[i]);
                early(l.p[i].early, l.ta[i], l.tb[i]);
            }
    } else if (is("tc_conv_dt_dv_kernel")) {
        const pf::tc::DtDvParams& p = arg<pf::tc::DtDvParams>(args, 3);
        check(p, blocks);
        for (int i = 0; i < 3 && p.early; ++i) early("operand of dT and dV", arg<CUtensorMap>(args, i));
    } else if (is("tc_conv_du_kernel")) {
        check(arg<pf::tc::DuParams>(args, 2));
        early("x of dU", arg<CUtensorMap>(args, 0));
    } else if (is("tc_conv_dx_kernel")) {
        check(arg<pf::tc::DxParams>(args, 2));
        early("U of dX", arg<CUtensorMap>(args, 1));
    } else if (is("simt_gemm_kernel")) {
        check(arg<pf::SimtGemm>(args, 0));
        known = false;
    } else {
        known = false;
    }
    if (!late) before.clear();
    before.insert(before.end(), written.begin(), written.end());
    before_known = known && (before_known || !late);
}

CUresult encode(CUtensorMap* map, CUtensorMapDataType type, cuuint32_t rank, void* base, const cuuint64_t* dims, const cuuint64_t* strides,
                const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
    const uint64_t size = type == CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 ? 2 : 4;
    uint64_t bytes = dims[0] * size;
    for (cuuint32_t i = 1; i < rank; ++i) bytes += (dims[i] - 1) * strides[i - 1];
    inside("tensor map", address(base), bytes);
    *map = CUtensorMap();
    reinterpret_cast<MapNote&>(*map) = MapNote{address(base), dims[0] * size, bytes};
    return CUDA_SUCCESS;
}
}  // namespace

extern "C" {
// The buffers of the calls that follow.  Maps are cached by address, so a call whose maps are to be seen has to use new ones.
void host_regions(int count, const uint64_t* base, const uint64_t* bytes) {
    regions.clear();
    for (int i = 0; i < count; ++i) regions.push_back(Range{base[i], bytes[i]});
    faults.clear();
    launches.clear();
    before.clear();
    before_known = false;
}
const char* host_faults() { return faults.c_str(); }
const char* host_launches() { return launches.c_str(); }

// Kernels whose name holds `part` (null: none) get no shared memory beyond the default.
static std::string refused;
void host_refuse(const char* part) { refused = part ? part : ""; }

// For runtime.cpp:
bool host_refuses(const void* kernel) { return !refused.empty() && kernels()[kernel].find(refused) != std::string::npos; }
void host_kernel(const void* host, const char* name) { kernels()[host] = name; }
void host_array(const void* host, size_t bytes) {
    static uint64_t next = 1ull << 60;
    arrays()[host] = Range{next, bytes};
    next += (bytes + (1 << 20)) & ~static_cast<uint64_t>((1 << 20) - 1);
}
void* host_array_address(const void* host) { return arrays().count(host) ? reinterpret_cast<void*>(arrays()[host].base) : nullptr; }
void host_launch(const void* kernel, unsigned blocks, void** args) { launched(kernel, blocks, args); }
void* host_encode() { return reinterpret_cast<void*>(encode); }
}
