// Parameters of a launch on CTA pairs (pf_tc_pair.cu).
#ifndef PF_TC_PAIR_LAUNCH_H_
#define PF_TC_PAIR_LAUNCH_H_

#include <cuda.h>

namespace pf {
namespace tc {

// One product of a launch.  Grouped products: operands are 3-D maps whose outermost coordinate is the group (a
// shared operand has one), group g's output starts g * c_gstride elements after C; kb_per_group > 0 instead makes
// the groups part of the contraction (one output).
struct PairProduct {
    int M, N, nkb;
    int a_mn, b_mn;          // 1 = operand stored with the M/N index contiguous
    int a_shared, b_shared, kb_per_group;
    int tiles_m, tiles_mn, tiles;       // 256-row tile rows; tiles of one group; all tiles
    void* C;                 // bf16 [M, ldc]
    long long ldc, c_gstride;
    const void* bias;        // C = act(A B + bias), bias [N] in bf16 or null
    int act;
    int early;               // kEarlyA | kEarlyB
};
// Up to three products.  Their tiles form two lists, the long ones first: list 0 (products 0 .. first - 1) is dealt
// to the pairs in turn; list 1 (the rest) is dealt so that the pairs which got one tile of list 0 less start `delay`
// rounds earlier, i.e. all pairs finish together.
struct PairLaunch {
    CUtensorMap ta[3], tb[3];
    PairProduct p[3];
    int count, first, total0, total1, early, delay;
    unsigned int* status;
};

}  // namespace tc
}  // namespace pf
#endif
