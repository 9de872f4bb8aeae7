// Row passes of the lengths 1024 and 2048 (rowfft_ct.cuh).
#define EPR_ROW_KERNELS
#include "rowfft_ct.cuh"

namespace {

// 2048: the one-line kernels also at six blocks per SM
constexpr RowKernels k2048()
{
    RowKernels k = row_full_xt<2048, 1>();
    k.fwd1_6 = k_row_fwd_ct<2048, 1, false, true, true>;
    k.inv1_6 = k_row_inv1<2048, 1, true>;
    return k;
}

const RowKernels kTable[] = {
    row_full_xt<1024, 1>(),
    k2048(),
};

}  // namespace

const eprrow::RowKernels* epr_row_table_mid(int* n)
{
    *n = (int)(sizeof(kTable) / sizeof(kTable[0]));
    return kTable;
}
