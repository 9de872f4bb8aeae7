// Column pass of the 2-D preconditioner: forward FFT along y, the
// FFT-diagonal Paganin-type filter H_s(q) = mu_s / (mu_s + L delta_s |q|^2)
// (arXiv 2601.22793, "Linear term and relation to Paganin"; the approximate
// inverse P_{1,s}^{-1} applied in "Iteration structure"), inverse FFT along y.
// The 1 / (nx ny) normalisation of the two inverse transforms is folded into
// the filter.
//
// One block transforms CW adjacent columns of the packed half spectrum of
// one (projection, line); the tile [ny][CW] lives in shared memory.  Column 0
// holds two real-input columns packed as one complex column (X[0] in the
// real part, the Nyquist X[nx/2] in the imaginary part); after the forward
// transform the two are separated with C[ky] and conj C[-ky], filtered with
// their own symbols and packed again:
//   C'[ky] = (H0 + HN)/2 C[ky] + (H0 - HN)/2 conj C[-ky].
#include <cudaTypedefs.h>

#define EPR_COL_KERNELS   // the shared helpers; no table is instantiated here
#include "colfft_ct.cuh"

// column lengths with the bulk-copy pass (colfft_ct_*.cu)
const eprcol::ColKernels* epr_col_table_a(int* n);
const eprcol::ColKernels* epr_col_table_b(int* n);

int epr_row_blocks(const EprConsts& C, int batch);

namespace {

// Symbol of the generic column pass at a = (L delta / mu) |q|^2, times the
// 1 / (nx ny) of the two inverse transforms.  With H = mu / (mu + L delta
// |q|^2) = 1 / (1 + a): dH/dmu = (a / mu) / (1 + a)^2 and dH/d(L delta) =
// -(a / (L delta)) / (1 + a)^2.
__device__ __forceinline__ float col_symbol(const ColArgs& A, float inv_n, float a)
{
    if (A.kind == 0) return inv_n / (1.f + a);
    const float d = 1.f + a;
    return A.kscale * inv_n * a / (d * d);
}

template <int EPT>
__global__ void __launch_bounds__(512, 2) k_col(const EprConsts C, const ColArgs A)
{
    extern __shared__ __align__(16) float2 buf[];
    const int b = blockIdx.z, sl = blockIdx.y;
    epr_grid_wait();
    if (A.check_done && A.st[b].done) return;
    epr_grid_release();
    col_finalize_rho(A, b, blockIdx.x == 0 && sl == 0);
    const int s = A.line0 + sl;
    const int ny = C.ny, half = C.half, CW = A.CW, lgCW = A.lgCW;
    const int T = blockDim.x, tid = threadIdx.x;
    const int kx0 = blockIdx.x * CW;
    float2* Sb = A.S + ((size_t)b * A.nl + sl) * (size_t)ny * half;

    for (int e = tid; e < ny * CW; e += T) {
        const int y = e >> lgCW, c = e & (CW - 1);
        buf[PC::idx(e)] = Sb[(size_t)y * half + kx0 + c];
    }
    __syncthreads();
    eprfft::fft<PC, -1, EPT>(buf, ny, lgCW, CW, 1, A.tw, T, tid);

    // filter (two phases: column 0 reads the mirrored frequency)
    const float ha = C.ha[s], hb = C.hb[s], inv_n = C.inv_n;
    float2 nv[EPT];
#pragma unroll
    for (int k = 0; k < EPT; ++k) {
        const int e = tid + k * T;
        const int y = e >> lgCW, c = e & (CW - 1);
        const int kx = kx0 + c;
        const float ky = (float)(y <= ny / 2 ? y : y - ny);
        const float qy = hb * ky * ky;
        const float2 v = buf[PC::idx(e)];
        if (kx != 0) {
            const float H = col_symbol(A, inv_n, ha * (float)kx * (float)kx + qy);
            nv[k] = cscale(v, H);
        } else {
            const float kn = (float)half;
            const float H0 = col_symbol(A, inv_n, qy);
            const float HN = col_symbol(A, inv_n, ha * kn * kn + qy);
            const int yneg = (y == 0) ? 0 : ny - y;
            const float2 w = cconj(buf[PC::idx((yneg << lgCW) + c)]);
            const float hp = 0.5f * (H0 + HN), hm = 0.5f * (H0 - HN);
            nv[k] = make_float2(hp * v.x + hm * w.x, hp * v.y + hm * w.y);
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < EPT; ++k) buf[PC::idx(tid + k * T)] = nv[k];
    __syncthreads();
    eprfft::fft<PC, +1, EPT>(buf, ny, lgCW, CW, 1, A.tw, T, tid);
    for (int e = tid; e < ny * CW; e += T) {
        const int y = e >> lgCW, c = e & (CW - 1);
        Sb[(size_t)y * half + kx0 + c] = buf[PC::idx(e)];
    }
}

// Compile-time column length NY and width CW, on the compile-time FFT engine.
template <int NY, int CW, int EPT>
__global__ void __launch_bounds__(NY * CW / EPT, (65536 / 64) / (NY * CW / EPT))
k_col_ct(const EprConsts C, const ColArgs A)
{
    constexpr int T = NY * CW / EPT;
    constexpr int LGCW = CW == 1 ? 0 : CW == 2 ? 1 : CW == 4 ? 2 : CW == 8 ? 3 : 4;
    static_assert(!eprfft::tw_exact(NY), "table 0 alone is there");
    extern __shared__ __align__(16) float2 buf[];
    const int b = blockIdx.z, sl = blockIdx.y;
    epr_grid_wait();
    if (A.check_done && A.st[b].done) return;
    col_finalize_rho(A, b, blockIdx.x == 0 && sl == 0);
    const int s = A.line0 + sl;
    const int half = C.half, tid = threadIdx.x;
    const int kx0 = blockIdx.x * CW;
    float2* Sb = A.S + ((size_t)b * A.nl + sl) * (size_t)NY * half;
#pragma unroll
    for (int k = 0; k < EPT; ++k) {
        const int e = tid + k * T;
        const int y = e >> LGCW, c = e & (CW - 1);
        buf[PC::idx(e)] = Sb[(size_t)y * half + kx0 + c];
    }
    __syncthreads();
    if (kx0 != 0) {   // the filter as the output map of the forward transform
        const ColPaganin<NY, CW, LGCW> f{line_const(C.ha, s), line_const(C.hb, s), C.inv_n, kx0};
        eprfft::fft_ct<PC, -1, NY, EPT, LGCW, CW, 1, 0>(buf, A.tw, tid, f);
    } else {
        eprfft::fft_ct<PC, -1, NY, EPT, LGCW, CW, 1>(buf, A.tw, tid);
        col_filter0<NY, CW, LGCW, T>(buf, C, s, tid);
    }
    eprfft::fft_ct<PC, +1, NY, EPT, LGCW, CW, 1>(buf, A.tw, tid);
    epr_grid_release();
#pragma unroll
    for (int k = 0; k < EPT; ++k) {
        const int e = tid + k * T;
        const int y = e >> LGCW, c = e & (CW - 1);
        Sb[(size_t)y * half + kx0 + c] = buf[PC::idx(e)];
    }
}

}  // namespace

struct EprColLaunch {
    int CW, lgCW, EPT, threads;
    size_t smem;
};

EprColLaunch epr_col_config(const EprConsts& C, int cw_hint)
{
    EprColLaunch L;
    int cw = cw_hint > 0 ? cw_hint : 4;
    while (cw > 1 && C.half % cw != 0) cw >>= 1;
    // keep the block at 512 threads or fewer, 8 elements per thread if possible
    int ept = 8;
    // 8192-point columns (oversampled internal grids): one column, 1024 threads
    const int tmax = C.ny >= 8192 ? 1024 : 512;
    while (C.ny * cw / ept > tmax && cw > 1) cw >>= 1;
    while (C.ny * cw / ept > tmax && ept < 16) ept *= 2;
    L.CW = cw;
    L.lgCW = 0;
    while ((1 << L.lgCW) < cw) ++L.lgCW;
    L.EPT = ept;
    L.threads = C.ny * cw / ept;
    L.smem = (size_t)PC::len(C.ny * cw) * sizeof(float2);
    return L;
}

namespace {

const ColKernels* col_kernels(int ny)
{
    int n = 0;
    for (auto table : {epr_col_table_a, epr_col_table_b}) {
        const ColKernels* k = table(&n);
        for (int i = 0; i < n; ++i)
            if (k[i].ny == ny) return &k[i];
    }
    return nullptr;
}

size_t col_tma_smem(int ny, int cw) { return 128 + (size_t)PC::len(ny * cw) * sizeof(float2); }

// Launches with fewer wide tiles than this take the two-column tile: twice the
// blocks, half the work in each, but a row of it is 16 bytes, half a sector.
// Solve iterations, us, with wide and two-column tiles (wide tiles in
// parentheses): 1024 rows 512 x 1024 (64) 22.7, 21.3; 1024^2 (128) 28.2, 28.9;
// two of 1152 x 1728 (288) 70.7, 75.7; eight of 1024^2 (1024) 116, 121.  512
// rows (512) 42.5, 40.8, (1024) 68.3, 67.3, (4096) 222, 226; 864 rows (256)
// 41.3, 39.2; 256 rows (64) 16.7, 15.8, (1024) 46.2, 46.2, (8192) 253, 265.
constexpr int col_wide_blocks(int ny) { return ny >= 1024 ? 128 : 1024; }

}  // namespace

// Tensor maps of S seen as `rows` rows of nx floats, with boxes of the wide
// and of the two-column tile, for the bulk-copy column pass (out[2]).  Returns
// false (and leaves the plain pass in use) when the size has no such pass or
// the CUDA driver API entry point cuTensorMapEncodeTiled is not available.
bool epr_col_make_map(const EprConsts& C, const float2* S, long long rows, CUtensorMap* out)
{
    const ColKernels* k = col_kernels(C.ny);
    if (!k || C.half % k->cw != 0 || !S || rows <= 0 || rows > (1ll << 31)) return false;
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    if (!encode) {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault,
                                             &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess || !fn)
            return false;
        encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    }
    for (int i = 0; i < 2; ++i) {
        const int cw = i == 0 ? k->cw : 2;
        const cuuint64_t dims[2] = {(cuuint64_t)C.nx, (cuuint64_t)rows};
        const cuuint64_t strides[1] = {(cuuint64_t)C.nx * sizeof(float)};
        const cuuint32_t box[2] = {(cuuint32_t)(2 * cw), (cuuint32_t)epr_col_box(C.ny, cw)};
        const cuuint32_t estr[2] = {1, 1};
        const CUresult r = encode(&out[i], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float2*>(S), dims,
                                  strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                  CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return false;
    }
    return true;
}

// rho_it >= 0 (a solve): a further block (block 0 of the passes without bulk
// copies) forms rho of iteration rho_it from the
// forward row pass's partials.
cudaError_t epr_launch_col(const EprConsts& C, const EprWork& W, int line0, int nl, int batch,
                           int check_done, int cw_hint, int rho_it, cudaStream_t stream)
{
    const EprColLaunch L = epr_col_config(C, cw_hint);
    ColArgs A;
    A.S = W.S;
    A.st = W.st;
    A.tw = W.tw_y;
    A.err = W.err;
    A.part_c = W.part_c;
    A.rho_hist = W.rho_hist;
    A.rho_it = rho_it;
    A.nblk = rho_it >= 0 ? epr_row_blocks(C, batch) : 0;
    A.max_blocks = W.max_blocks;
    A.hist_len = W.hist_len;
    A.CW = L.CW;
    A.lgCW = L.lgCW;
    A.line0 = line0;
    A.nl = nl;
    A.check_done = check_done;
    A.kind = 0;
    A.kscale = 0.f;
    const dim3 grid(C.half / L.CW, nl, batch);
    const bool pdl = C.pdl != 0;
    cudaError_t e = cudaSuccess;
    bool done = false;
    if (W.col_map && cw_hint == 0) {   // a map exists only for lengths in the tables
        const ColKernels& k = *col_kernels(C.ny);
        const CUtensorMap* maps = static_cast<const CUtensorMap*>(W.col_map);
        const bool r8 = k.radix8 && !W.col_radix16, o5 = k.occ5 && W.col_occ5;
        const long long tiles = (long long)(C.half / k.cw) * (C.det ? 1 : nl) * epr_rule_batch(C, batch);
        const bool narrow = k.narrow && tiles < col_wide_blocks(C.ny);
        const int cw = narrow ? 2 : k.cw;
        A.CW = cw;
        A.lgCW = cw == 2 ? 1 : 2;
        const ColKernel q = r8 ? k.radix8 : o5 ? k.occ5 : narrow ? k.narrow : k.wide;
        e = epr_launch_kernel(pdl, q, dim3(C.half / cw + (rho_it >= 0 ? 1 : 0), nl, batch), dim3(narrow ? k.threads2 : k.threads),
                              col_tma_smem(C.ny, cw), stream, C, A, maps[narrow ? 1 : 0]);
        done = true;
    }
#define EPR_COL_CASE(NYV, CWV, EPTV)                                                           \
    if (!done && C.ny == NYV && L.CW == CWV && L.EPT == EPTV) {                               \
        e = epr_launch_kernel(pdl, k_col_ct<NYV, CWV, EPTV>, grid, dim3(NYV * CWV / EPTV),    \
                              L.smem, stream, C, A);                                          \
        done = true;                                                                          \
    }
    EPR_COL_CASE(256, 4, 8)
    EPR_COL_CASE(512, 4, 8)
    EPR_COL_CASE(1024, 4, 8)
    EPR_COL_CASE(1536, 2, 8)
    EPR_COL_CASE(2048, 2, 8)
    EPR_COL_CASE(2048, 1, 8)
    EPR_COL_CASE(3072, 1, 8)
    EPR_COL_CASE(4096, 1, 8)
    EPR_COL_CASE(8192, 1, 8)
#undef EPR_COL_CASE
    if (!done) {
        if (L.EPT == 8)
            e = epr_launch_kernel(pdl, k_col<8>, grid, dim3(L.threads), L.smem, stream, C, A);
        else
            e = epr_launch_kernel(pdl, k_col<16>, grid, dim3(L.threads), L.smem, stream, C, A);
    }
    epr_count_launch(1);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// The generic column pass with symbol `kind` (col_symbol) for one line of a
// batch of spectra (line slot 0 of S, the constants of line `line`): the
// filter derivatives of the reverse pass through the solve.
cudaError_t epr_launch_col_kind(const EprConsts& C, const EprWork& W, int line, int batch,
                                int kind, float kscale, cudaStream_t stream)
{
    const EprColLaunch L = epr_col_config(C, 0);
    ColArgs A = {};
    A.S = W.S;
    A.st = W.st;
    A.tw = W.tw_y;
    A.err = W.err;
    A.rho_it = -1;
    A.CW = L.CW;
    A.lgCW = L.lgCW;
    A.line0 = line;
    A.nl = 1;
    A.check_done = 0;
    A.kind = kind;
    A.kscale = kscale;
    const dim3 grid(C.half / L.CW, 1, batch);
    cudaError_t e;
    if (L.EPT == 8)
        e = epr_launch_kernel(false, k_col<8>, grid, dim3(L.threads), L.smem, stream, C, A);
    else
        e = epr_launch_kernel(false, k_col<16>, grid, dim3(L.threads), L.smem, stream, C, A);
    epr_count_launch(1);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t epr_col_init()
{
    cudaError_t e = cudaSuccess;
    auto allow = [&](auto kernel) { if (e == cudaSuccess) e = epr_allow_max_smem(kernel); };
    allow(k_col<8>);
    allow(k_col<16>);
    allow(k_col_ct<256, 4, 8>);
    allow(k_col_ct<512, 4, 8>);
    allow(k_col_ct<1024, 4, 8>);
    allow(k_col_ct<1536, 2, 8>);
    allow(k_col_ct<2048, 2, 8>);
    allow(k_col_ct<2048, 1, 8>);
    allow(k_col_ct<3072, 1, 8>);
    allow(k_col_ct<4096, 1, 8>);
    allow(k_col_ct<8192, 1, 8>);
    return e;
}

// The bulk-copy passes of length ny (none: nothing to do).
cudaError_t epr_col_init_tma(int ny)
{
    const ColKernels* k = col_kernels(ny);
    if (!k) return cudaSuccess;
    for (ColKernel q : {k->wide, k->narrow, k->radix8, k->occ5})
        if (q) {
            const cudaError_t e = epr_allow_max_smem(q);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}
