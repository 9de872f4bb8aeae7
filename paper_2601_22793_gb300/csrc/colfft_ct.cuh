// The column pass on the compile-time FFT engine with its tile moved by bulk
// tensor copies: kernels templated on the column length, instantiated for
// groups of lengths in colfft_ct_*.cu and launched through tables (colfft.cu,
// which also holds the plain passes and describes the pass).
#pragma once

#include <cuda.h>

#include "epr_internal.cuh"
#include "fft.cuh"
#include "tma.cuh"

namespace eprcol {

struct ColArgs {
    float2* S;            // [B][nl][ny][nx/2]
    EprProjState* st;
    const float2* tw;     // twiddle tables of length ny
    unsigned int* err;    // device error word
    const double* part_c; // [B][max_blocks] forward row pass partials
    double* rho_hist;     // [B][hist_len]
    int CW, lgCW;
    int line0, nl;
    int check_done;
    int rho_it;           // >= 0: form rho of this iteration
    int nblk, max_blocks, hist_len;
    int kind;             // symbol of the generic pass: 0 = H = 1 / (1 + a),
                          // 1, 2 = kscale a / (1 + a)^2 (the derivatives of
                          // H by mu and by L delta), a = (L delta / mu) |q|^2
    float kscale;         // 1 / mu (kind 1) or -1 / (L delta) (kind 2)
};


typedef void (*ColKernel)(const EprConsts, const ColArgs, const CUtensorMap);

// One column length: the pass with the wide tile, and with the two-column
// tile for launches whose wide tiles would leave SMs without a block.
struct ColKernels {
    int ny, cw, threads, threads2;
    ColKernel wide, narrow;      // narrow: two columns (NULL where the wide tile has two)
    ColKernel radix8, occ5;      // 2048 rows, two columns: radix-8 stages; five blocks per SM
};

}  // namespace eprcol

// Rows of one bulk-copy box of an [ny][cw] tile: the largest divisor of ny up
// to 256 whose boxes start on 128-byte boundaries in shared memory.
__host__ __device__ constexpr int epr_col_box(int ny, int cw)
{
    int d = ny < 256 ? ny : 256;
    while (ny % d != 0 || (d * cw * 8) % 128 != 0) --d;
    return d;
}

#ifdef EPR_COL_KERNELS
namespace {

using namespace eprcol;
using PC = eprfft::PadCol;  // shared layout of the column tile

constexpr int col_min_blocks(int T)
{
    const int b = T == 512 ? 2 : 1024 / ((T + 31) / 32 * 32);
    return b < 1 ? 1 : b > 16 ? 16 : b;
}

// One block of the column pass of a solve (line 0) turns the forward row
// pass's partials into rho; the grid dependency wait has made them visible.
// The bulk-copy pass launches one block more for it.
__device__ __forceinline__ void col_finalize_rho(const ColArgs& A, int b, bool lead)
{
    if (A.rho_it >= 0 && lead)
        finalize_rho(&A.st[b], A.part_c + (size_t)b * A.max_blocks, A.nblk,
                     A.rho_hist ? A.rho_hist + (size_t)b * A.hist_len : nullptr, A.hist_len, A.rho_it);
}

// The Paganin filter H = inv_n / (1 + ha kx^2 + hb ky^2) of element e of a
// [NY][CW] tile whose first column is kx0 > 0, as the output map of the last
// forward FFT stage (a fast reciprocal: 2 ulp).
template <int NY, int CW, int LGCW>
struct ColPaganin {
    float ha, hb, inv_n;
    int kx0;
    __device__ __forceinline__ float2 operator()(float2 v, int e) const
    {
        const int y = e >> LGCW, c = e & (CW - 1);
        const float ky = (float)(y <= NY / 2 ? y : y - NY), kx = (float)(kx0 + c);
        const float H = __fdividef(inv_n, fmaf(ha * kx, kx, fmaf(hb * ky, ky, 1.f)));
        return make_float2(v.x * H, v.y * H);
    }
};

// The filter of the tile holding column kx = 0, in place in buf.  That column
// packs the DC and Nyquist columns of the real transform, so its output at y
// mixes the values at y and NY - y: a thread takes both of a mirrored pair.
// The other columns of the tile are filtered pointwise.  Ends with a barrier.
template <int NY, int CW, int LGCW, int T>
__device__ __forceinline__ void col_filter0(float2* buf, const EprConsts& C, int s, int tid)
{
    const float ha = line_const(C.ha, s), hb = line_const(C.hb, s), inv_n = C.inv_n;
    const float kn = (float)C.half;
    for (int y = tid; y <= NY / 2; y += T) {
        const int yn = y == 0 ? 0 : NY - y;   // 0 and NY / 2 are their own mirror
        const float ky = (float)y;
        const float qy = hb * ky * ky;
        const float H0 = inv_n / (1.f + qy);
        const float HN = inv_n / (1.f + ha * kn * kn + qy);
        const float hp = 0.5f * (H0 + HN), hm = 0.5f * (H0 - HN);
        const float2 a = buf[eprfft::PadCol::idx(y << LGCW)];
        const float2 b = buf[eprfft::PadCol::idx(yn << LGCW)];
        buf[eprfft::PadCol::idx(y << LGCW)] = make_float2(hp * a.x + hm * b.x, hp * a.y - hm * b.y);
        if (yn != y)
            buf[eprfft::PadCol::idx(yn << LGCW)] = make_float2(hp * b.x + hm * a.x, hp * b.y - hm * a.y);
    }
    const ColPaganin<NY, CW, LGCW> f{ha, hb, inv_n, 0};
    for (int e = tid; e < NY * CW; e += T) {
        if ((e & (CW - 1)) == 0) continue;
        const int i = eprfft::PadCol::idx(e);
        buf[i] = f(buf[i], e);
    }
    __syncthreads();
}

// The same pass with the [NY][CW] tile moved by the tensor memory
// accelerator: BOXES bulk loads of [NY / BOXES][CW] into a dense tile at the
// start of the FFT buffer (no L1 traffic, one elected thread).  The first
// FFT stage reads every operand from the dense tile before its barrier and
// writes the padded layout over it; the last stage reads the padded layout
// and writes its results dense over it, which the bulk store reads.  So the
// block needs only the padded buffer.  The tile's row pitch is
// CW * 8 bytes, which keeps the strided 16-byte row segments of the column
// off the load/store unit.
constexpr unsigned int kTmaWaitPolls = 1u << 22;

// OCC > 0: that many blocks per SM (the radix-16 2048-row pass at five: 48
// registers, no spills), else the default bound.
template <int NY, int CW, int EPT, int MAXR = 16, int OCC = 0>
__global__ void __launch_bounds__(NY * CW / EPT,
                                  OCC > 0 ? OCC : col_min_blocks(NY * CW / EPT))
k_col_tma(const EprConsts C, const ColArgs A, const __grid_constant__ CUtensorMap map)
{
    constexpr int T = NY * CW / EPT;
    static_assert(NY * CW % EPT == 0, "every element has a thread");
    constexpr int LGCW = CW == 2 ? 1 : CW == 4 ? 2 : 3;
    constexpr int BOXY = epr_col_box(NY, CW);
    constexpr int BOXES = NY / BOXY;
    constexpr unsigned int BYTES = NY * CW * sizeof(float2);
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ alignas(8) uint64_t bar;
    // the 128-byte aligned FFT buffer; the dense tile occupies its start
    const size_t base = ((size_t)__cvta_generic_to_shared(smem_raw) + 127) & ~size_t(127);
    float2* buf = reinterpret_cast<float2*>(smem_raw + (base - (size_t)__cvta_generic_to_shared(smem_raw)));
    const int b = blockIdx.z, sl = blockIdx.y, tid = threadIdx.x;
    const int kx0 = ((int)blockIdx.x - (A.rho_it >= 0 ? 1 : 0)) * CW;
    if (A.rho_it >= 0 && blockIdx.x == 0) {   // the block that forms rho, in the first wave
        epr_grid_wait();
        if (!(A.check_done && A.st[b].done)) col_finalize_rho(A, b, sl == 0);
        return;
    }
    if (tid == 0) {
        epr_tma::mbar_init(&bar, 1);
        epr_tma::fence_async_shared();
    }
    __syncthreads();
    epr_grid_wait();
    if (A.check_done && A.st[b].done) return;
    const int row0 = (b * A.nl + sl) * NY;
    if (tid == 0) {
        epr_tma::fence_async_global();
        epr_tma::mbar_arrive_expect_tx(&bar, BYTES);
#pragma unroll
        for (int i = 0; i < BOXES; ++i)
            epr_tma::load_2d(buf + i * BOXY * CW, &map, 2 * kx0, row0 + i * BOXY, &bar);
    }
    if (!epr_tma::mbar_wait(&bar, 0, kTmaWaitPolls)) {
        // the copy did not arrive: report, and wait once more (bounded) so
        // that no copy lands after the block has left
        if (tid == 0) atomicOr(A.err, EPR_DEVERR_TIMEOUT);
        epr_tma::mbar_wait(&bar, 0, kTmaWaitPolls);
        return;
    }
    const int s = A.line0 + sl;
    constexpr int NST = eprfft::ct_n_stages(NY, MAXR);
    // the inverse runs the reversed stage plan, whose first stage takes the
    // last forward stage's results as they are
    if (kx0 != 0) {   // last forward stage, filter, first inverse stage in registers
        const ColPaganin<NY, CW, LGCW> f{line_const(C.ha, s), line_const(C.hb, s), C.inv_n, kx0};
        eprfft::fft_ct_from_stages<PC, -1, NY, EPT, LGCW, CW, 1, NST - 1, MAXR>(buf, buf, A.tw, tid);
        eprfft::stage_turn<PC, -1, +1, EPT, NY, LGCW, CW, 1, MAXR>(buf, A.tw, tid, f);
        eprfft::fft_ct_rev_stages<PC, +1, NY, EPT, LGCW, CW, 1, 1, NST - 1, MAXR>(buf, A.tw, tid);
    } else {   // the packed DC / Nyquist column filters mirrored pairs in place
        eprfft::fft_ct_from<PC, -1, NY, EPT, LGCW, CW, 1, MAXR>(buf, buf, A.tw, tid);
        col_filter0<NY, CW, LGCW, T>(buf, C, s, tid);
        eprfft::fft_ct_rev_stages<PC, +1, NY, EPT, LGCW, CW, 1, 0, NST - 1, MAXR>(buf, A.tw, tid);
    }
    epr_grid_release();
    // the last stage writes the dense tile the bulk store reads, in place:
    // every operand is read before the stage's barrier
    eprfft::fft_ct_rev_last<eprfft::Dense, true, false, PC, +1, NY, EPT, LGCW, CW, 1, MAXR>(buf, A.tw, tid);
    epr_tma::fence_async_shared();
    __syncthreads();
    if (tid == 0) {
#pragma unroll
        for (int i = 0; i < BOXES; ++i)
            epr_tma::store_2d(&map, 2 * kx0, row0 + i * BOXY, buf + i * BOXY * CW);
        epr_tma::bulk_commit();
        epr_tma::bulk_wait_read_all();   // the tile must outlive the copy's reads
    }
}

// 16 elements per thread and radix-16 stages: 2048 = 16 16 8 and 1024 = 16 16 4
// in three round trips through shared memory instead of four with radix 8.
// The narrow tile serves launches that leave the chip idle, where the chain
// of one thread's instructions is the time: 8 elements per thread.
template <int NY, int CW>
constexpr ColKernels col_entry()
{
    ColKernels k = {};
    k.ny = NY;
    k.cw = CW;
    k.threads = NY * CW / 16;
    k.wide = k_col_tma<NY, CW, 16>;
    if constexpr (CW > 2) {
        k.threads2 = NY * 2 / 8;
        k.narrow = k_col_tma<NY, 2, 8, 8>;
    }
    return k;
}

}  // namespace
#endif  // EPR_COL_KERNELS
