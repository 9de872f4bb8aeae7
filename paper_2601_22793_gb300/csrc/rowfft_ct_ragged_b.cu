// Row passes of the lengths 2^a 3^b, b > 0 (one third of them, to build in parallel) (rowfft_ct.cuh).
#define EPR_ROW_KERNELS
#include "rowfft_ct.cuh"

namespace {

const RowKernels kTable[] = {
    row_any<144, 1>(),
    row_any<216, 4>(),
    row_any<288, 1>(),
    row_any<432, 2>(),
    row_any<576, 1>(),
    row_any<864, 1>(),
    row_full<1728, 1>(),
    row_full<2592, 1>(),
};

}  // namespace

const eprrow::RowKernels* epr_row_table_ragged_b(int* n)
{
    *n = (int)(sizeof(kTable) / sizeof(kTable[0]));
    return kTable;
}
