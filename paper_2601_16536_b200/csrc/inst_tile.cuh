// Instantiations of the tcgen05 tile kernel for one 16-bit type and group size: include with W4A16_INST_BF
// (true / false), W4A16_INST_SG (1 / 2 / 4) and W4A16_INST_NAME (f16_sg1 ...) defined.
#include "kernel_tables.h"

namespace w4a16 {
namespace {
template <bool SYM, bool EPI>
TileKernel pick() {
    constexpr bool BF = W4A16_INST_BF;
    constexpr int SG = W4A16_INST_SG;
    return gemm_tile_kernel<SG, BF, SYM, EPI>;
}
}  // namespace

#define W4A16_CAT2(a, b) a##b
#define W4A16_CAT(a, b) W4A16_CAT2(a, b)

TileKernel W4A16_CAT(tile_kernel_, W4A16_INST_NAME)(bool sym, bool epi) {
    if (sym) return epi ? pick<true, true>() : pick<true, false>();
    return epi ? pick<false, true>() : pick<false, false>();
}
int W4A16_CAT(status_take_tile_, W4A16_INST_NAME)() { return status_take_this_unit(); }

}  // namespace w4a16
