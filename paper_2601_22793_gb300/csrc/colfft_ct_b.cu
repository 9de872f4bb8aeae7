// Bulk-copy column passes: every other supported length (colfft_ct.cuh).
#define EPR_COL_KERNELS
#include "colfft_ct.cuh"

namespace {

// 2048: also radix-8 stages, and radix 16 at five blocks per SM (48 registers)
constexpr ColKernels k2048()
{
    ColKernels k = col_entry<2048, 2>();
    k.radix8 = k_col_tma<2048, 2, 16, 8>;
    k.occ5 = k_col_tma<2048, 2, 16, 16, 5>;
    return k;
}

const ColKernels kTable[] = {
    col_entry<144, 4>(),
    col_entry<216, 4>(),
    col_entry<288, 4>(),
    col_entry<432, 4>(),
    col_entry<576, 4>(),
    col_entry<768, 4>(),
    col_entry<1024, 4>(),
    col_entry<1296, 4>(),
    col_entry<1728, 4>(),
    k2048(),
    col_entry<2592, 2>(),
    col_entry<3456, 2>(),
    col_entry<4096, 2>(),
};

}  // namespace

const eprcol::ColKernels* epr_col_table_b(int* n)
{
    *n = (int)(sizeof(kTable) / sizeof(kTable[0]));
    return kTable;
}
