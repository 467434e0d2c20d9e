// Class counts 24 to 28 of the row-walking upsample + cross-entropy kernel.
#include "k_upsample_ce_rows.cuh"

namespace st {

RowsKernels rows_kernels_3(int n)
{
    constexpr int first = kRowsLast[2] + 1;
    return rows_kernels_of<first>(n, std::make_integer_sequence<int, kRowsLast[3] - first + 1>());
}

}  // namespace st
