// Row passes of the lengths 2^a 3^b, b > 0 (one third of them, to build in parallel) (rowfft_ct.cuh).
#define EPR_ROW_KERNELS
#include "rowfft_ct.cuh"

namespace {

const RowKernels kTable[] = {
    row_any<192, 4>(),
    row_any<216, 1>(),
    row_any<384, 2>(),
    row_any<432, 1>(),
    row_full<768, 1>(),
    row_full<1152, 1>(),
    row_full<1944, 1>(),
    row_full<3456, 1>(),
};

}  // namespace

const eprrow::RowKernels* epr_row_table_ragged_c(int* n)
{
    *n = (int)(sizeof(kTable) / sizeof(kTable[0]));
    return kTable;
}
