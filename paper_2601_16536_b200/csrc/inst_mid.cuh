// Instantiations of the two-CTAs-per-SM tcgen05 kernel for one 16-bit type: include with W4A16_INST_BF (true / false)
// and W4A16_INST_NAME (f16 / bf16) defined.
#include "kernel_tables.h"

namespace w4a16 {
namespace {
template <int MTC>
MidKernel pick(int sg, bool sym) {
    constexpr bool BF = W4A16_INST_BF;
    if (sym) return sg == 1 ? gemm_mid_kernel<MTC, 1, BF, true> : sg == 2 ? gemm_mid_kernel<MTC, 2, BF, true> : gemm_mid_kernel<MTC, 4, BF, true>;
    return sg == 1 ? gemm_mid_kernel<MTC, 1, BF, false> : sg == 2 ? gemm_mid_kernel<MTC, 2, BF, false> : gemm_mid_kernel<MTC, 4, BF, false>;
}
}  // namespace

#define W4A16_CAT2(a, b) a##b
#define W4A16_CAT(a, b) W4A16_CAT2(a, b)

MidKernel W4A16_CAT(mid_kernel_, W4A16_INST_NAME)(int mtc, int sg, bool sym) {
    return mtc <= 64 ? pick<64>(sg, sym) : pick<128>(sg, sym);
}
int W4A16_CAT(status_take_mid_, W4A16_INST_NAME)() { return status_take_this_unit(); }

}  // namespace w4a16
