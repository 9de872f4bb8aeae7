// Row passes of the lengths 1536, 3072, 4096 and 8192 (rowfft_ct.cuh).
#define EPR_ROW_KERNELS
#include "rowfft_ct.cuh"

namespace {

// 8192 (oversampled grids): the one-line kernels with 16 elements per thread,
// which stage no thickness, at two blocks per SM
constexpr RowKernels k8192()
{
    RowKernels k = row_any<8192, 1>();
    k.fwd1 = k_row_fwd_ct<8192, 1, false, true, false, false, 16>;
    k.inv1 = k_row_inv1<8192, 1, false, false, 16>;
    k.threads16 = 8192 / 16;
    return k;
}

const RowKernels kTable[] = {
    row_full<1536, 1>(),
    row_full<3072, 1>(),
    row_full_xt<4096, 1>(),
    k8192(),
};

}  // namespace

const eprrow::RowKernels* epr_row_table_long(int* n)
{
    *n = (int)(sizeof(kTable) / sizeof(kTable[0]));
    return kTable;
}
