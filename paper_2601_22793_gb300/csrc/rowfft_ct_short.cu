// Row passes of the lengths 256, 512 and 128 (rowfft_ct.cuh).
#define EPR_ROW_KERNELS
#include "rowfft_ct.cuh"

namespace {

const RowKernels kTable[] = {
    row_full<256, 4>(),
    row_any<256, 1, 4>(),
    row_full<512, 2>(),
    row_any<512, 1, 4>(),
    row_any<128, 8>(),
    row_any<128, 1, 4>(),
};

}  // namespace

const eprrow::RowKernels* epr_row_table_short(int* n)
{
    *n = (int)(sizeof(kTable) / sizeof(kTable[0]));
    return kTable;
}
