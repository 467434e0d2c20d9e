// Class counts 29 to 32 of the upsample + cross-entropy kernel for at most 32.
#include "k_fwd_ce.cuh"

namespace st {

FwdCeKernels fwd_ce_kernels_4(int n)
{
    constexpr int first = kFwdCeLast[3] + 1;
    return fwd_ce_kernels_of<first>(n, std::make_integer_sequence<int, kFwdCeLast[4] - first + 1>());
}

}  // namespace st
