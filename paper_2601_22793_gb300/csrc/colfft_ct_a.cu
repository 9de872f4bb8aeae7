// Bulk-copy column passes: every other supported length (colfft_ct.cuh).
#define EPR_COL_KERNELS
#include "colfft_ct.cuh"

namespace {

const ColKernels kTable[] = {
    col_entry<128, 4>(),
    col_entry<192, 4>(),
    col_entry<256, 4>(),
    col_entry<384, 4>(),
    col_entry<512, 4>(),
    col_entry<648, 4>(),
    col_entry<864, 4>(),
    col_entry<1152, 4>(),
    col_entry<1536, 4>(),
    col_entry<1944, 4>(),
    col_entry<2304, 2>(),
    col_entry<3072, 2>(),
    col_entry<3888, 2>(),
    col_entry<8192, 2>(),
};

}  // namespace

const eprcol::ColKernels* epr_col_table_a(int* n)
{
    *n = (int)(sizeof(kTable) / sizeof(kTable[0]));
    return kTable;
}
