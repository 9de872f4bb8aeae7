// Row passes of the lengths 2^a 3^b, b > 0 (one third of them, to build in parallel) (rowfft_ct.cuh).
#define EPR_ROW_KERNELS
#include "rowfft_ct.cuh"

namespace {

const RowKernels kTable[] = {
    row_any<144, 4>(),
    row_any<192, 1>(),
    row_any<288, 2>(),
    row_any<384, 1>(),
    row_any<648, 1>(),
    row_full<1296, 1>(),
    row_full<2304, 1>(),
    row_full<3888, 1>(),
};

}  // namespace

const eprrow::RowKernels* epr_row_table_ragged_a(int* n)
{
    *n = (int)(sizeof(kTable) / sizeof(kTable[0]));
    return kTable;
}
