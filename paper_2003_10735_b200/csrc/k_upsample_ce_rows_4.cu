// Class counts 29 to 32 of the row-walking upsample + cross-entropy kernel.
#include "k_upsample_ce_rows.cuh"

namespace st {

RowsKernels rows_kernels_4(int n)
{
    constexpr int first = kRowsLast[3] + 1;
    return rows_kernels_of<first>(n, std::make_integer_sequence<int, kRowsLast[4] - first + 1>());
}

}  // namespace st
