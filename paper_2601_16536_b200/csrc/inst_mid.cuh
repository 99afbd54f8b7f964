// Instantiations of the two-CTAs-per-SM tcgen05 kernel for one 16-bit type: include with W4A16_INST_BF (true / false)
// and W4A16_INST_NAME (f16 / bf16) defined.
#include "kernel_tables.h"

namespace w4a16 {
namespace {
template <int SG>
MidKernel pick(bool sym) {
    constexpr bool BF = W4A16_INST_BF;
    return sym ? gemm_mid_kernel<64, SG, BF, true> : gemm_mid_kernel<64, SG, BF, false>;
}
}  // namespace

#define W4A16_CAT2(a, b) a##b
#define W4A16_CAT(a, b) W4A16_CAT2(a, b)

MidKernel W4A16_CAT(mid_kernel_, W4A16_INST_NAME)(int sg, bool sym) {
    return sg == 1 ? pick<1>(sym) : sg == 2 ? pick<2>(sym) : pick<4>(sym);
}
int W4A16_CAT(status_take_mid_, W4A16_INST_NAME)() { return status_take_this_unit(); }

}  // namespace w4a16
