// Row passes of the 2-D preconditioner FFT, fused with the steps around it.
//
// Forward row pass (R2C), one block per RP pairs of rows of one projection:
//   prologue  back-transport of the split residual (arXiv 2601.22793, Eq. 4
//             and "Iteration structure"): for every object pixel and line,
//             g_s = sum of the four bilinear weights times the residual
//             r_s = (D - P) P_s / P at the shifted corners (mono: D - P,
//             read directly when the splat stored it); or the identity
//             back-transport of the local solver; or a plain load of a real
//             map (standalone filter).  The thickness rows needed for the
//             gradient are staged in shared memory first.
//   transform two real rows packed as one complex row, z = g(y0) + i g(y1),
//             shared-memory Stockham FFT of length nx;
//   epilogue  unpack X0[k] = (Z[k] + conj Z[-k]) / 2, X1[k] = (Z[k] -
//             conj Z[-k]) / 2i and store k < nx/2 with the real Nyquist
//             value packed into the imaginary part of k = 0.
// The block also stores its share of |D - P|^2; a block of its own of the
// column pass that follows adds the shares in a fixed order (deterministic)
// into rho.
//
// Inverse row pass (C2R), the mirror image, fused with the update
// ("Iterative inversion"): per line, I'_s = max(I_s + omega h_s, eps f_s),
// then the single-thickness projection of Eq. 7,
//   T' = - sum_s f_s mu_s ln(I'_s / f_s) / sum_s f_s mu_s^2,
// evaluated as T' = T - sum_s w_s ln(1 + omega h_s / I_s) (w_s = f_s mu_s /
// sum f mu^2), the same quantity without forming exp then log of values
// near one.  Each block stores its shares of |T' - T|^2 and |T'|^2; a block of
// its own of the next forward row pass (or a one-block kernel after the last
// iteration) adds them in a fixed order into kappa and retires the
// projection when kappa <= tol.
#include <mutex>

#define EPR_ROW_KERNELS   // the shared helpers; no table is instantiated here
#include "rowfft_ct.cuh"

// row lengths with compile-time kernels (rowfft_ct_*.cu)
const eprrow::RowKernels* epr_row_table_short(int* n);
const eprrow::RowKernels* epr_row_table_mid(int* n);
const eprrow::RowKernels* epr_row_table_long(int* n);
const eprrow::RowKernels* epr_row_table_ragged_a(int* n);
const eprrow::RowKernels* epr_row_table_ragged_b(int* n);
const eprrow::RowKernels* epr_row_table_ragged_c(int* n);

namespace {

enum { FWD_SOLVE_NL = 0, FWD_SOLVE_LOCAL = 1, FWD_LOAD = 2 };
enum { INV_UPDATE = 0, INV_STORE = 1 };

__device__ __forceinline__ int fdiv(int i, float inv_d) { return (int)(((float)i + 0.5f) * inv_d); }

// split residual of line s at detector pixel q of projection b (pb = b * npix)
__device__ __forceinline__ float resid(const EprConsts& C, const RowArgs& A, size_t pb, size_t q, int s)
{
    if (C.ns == 1) return __ldg(&A.P[pb + q]);
    return __ldg(&A.Ps[pb * C.ns + (size_t)s * C.nx * C.ny + q]);
}

// bilinear gather of line s's residual at (y + uy, x + ux); corners outside
// the grid read 0 (Eq. 4)
__device__ __forceinline__ float gather_px(const EprConsts& C, const RowArgs& A, size_t pb, int y,
                                           int x, float uy, float ux, int s)
{
    const float lim = 2.f * (float)(C.nx > C.ny ? C.nx : C.ny);
    ux = fminf(fmaxf(ux, -lim), lim);
    uy = fminf(fmaxf(uy, -lim), lim);
    const float fx = floorf(ux), fy = floorf(uy);
    const float dx = ux - fx, dy = uy - fy;
    const int cx = x + (int)fx, cy = y + (int)fy;
    const int nx = C.nx, ny = C.ny;
    const bool x0 = (unsigned)cx < (unsigned)nx, x1 = (unsigned)(cx + 1) < (unsigned)nx;
    float r00 = 0.f, r10 = 0.f, r01 = 0.f, r11 = 0.f;
    if ((unsigned)cy < (unsigned)ny) {
        const size_t row = (size_t)cy * nx;
        if (x0) r00 = resid(C, A, pb, row + cx, s);
        if (x1) r10 = resid(C, A, pb, row + cx + 1, s);
    }
    if ((unsigned)(cy + 1) < (unsigned)ny) {
        const size_t row = (size_t)(cy + 1) * nx;
        if (x0) r01 = resid(C, A, pb, row + cx, s);
        if (x1) r11 = resid(C, A, pb, row + cx + 1, s);
    }
    const float top = r00 + dx * (r10 - r00);
    const float bot = r01 + dx * (r11 - r01);
    return (1.f - dy) * top + dy * bot;
}

// XT: an x-dependent spectrum, the shift constant read per object column.
template <int MODE, int NS, bool XT = false>
__global__ void __launch_bounds__(512, 2) k_row_fwd(const EprConsts C, const RowArgs A)
{
    extern __shared__ __align__(16) float2 zs[];
    __shared__ float red[64];
    const int b = row_batch_index();
    const int nx = C.nx, ny = C.ny, half = C.half;
    const int T = blockDim.x, tid = threadIdx.x;
    const int RP = A.RP, sm = nx + kPad;
    const size_t npix = (size_t)nx * ny;
    const size_t pb = (size_t)b * npix;
    const int yb = blockIdx.x * RP * 2;   // first row of the block
    const int nl = NS ? NS : A.nl;
    // thickness rows yb-1 .. yb+2RP (clamped), after the FFT buffer
    float* Ts = reinterpret_cast<float*>(zs + ((PR::len(RP * sm) + 1) & ~1));
    const int nrows = 2 * RP + 2;

    if constexpr (MODE == FWD_SOLVE_NL) {   // T is not written by the predecessor
        const float* Tb = A.T + pb;
        const int q4 = nx >> 2;
        const float inv_q4 = 1.f / (float)q4;
        for (int i = tid; i < nrows * q4; i += T) {
            const int r = fdiv(i, inv_q4), c4 = i - r * q4;
            const int gy = min(max(yb - 1 + r, 0), ny - 1);
            cp_async16(reinterpret_cast<float4*>(Ts) + i,
                       reinterpret_cast<const float4*>(Tb + (size_t)gy * nx) + c4);
        }
        cp_async_commit();
    }
    epr_grid_wait();
    if constexpr (MODE != FWD_LOAD) fwd_finalize_kappa(A, b, blockIdx.x == 0, (int)gridDim.x);
    if (A.check_done && A.st[b].done) {
        cp_async_wait_all();   // no copy may land after the block has left
        return;
    }
    epr_grid_release();
    if constexpr (MODE == FWD_SOLVE_NL) {
        cp_async_wait_all();
        __syncthreads();
    }

    float ra = 0.f;   // |D - P|^2 share
    const float inv_nx = 1.f / (float)nx;
    for (int sl = 0; sl < nl; ++sl) {
        const int s = A.line0 + sl;
        // prologue: packed complex input rows in shared memory
#pragma unroll 2
        for (int k = 0; k < kEPT; ++k) {
            const int e = tid + k * T;
            const int m = RP == 1 ? 0 : fdiv(e, inv_nx);
            const int x = e - m * nx;
            const int y0 = yb + 2 * m;
            float v[2];
#pragma unroll
            for (int r0 = 0; r0 < 2; ++r0) {
                const int y = y0 + r0;
                if constexpr (MODE == FWD_SOLVE_NL) {
                    const float* tr = Ts + (2 * m + r0 + 1) * nx;   // row y
                    const float t = tr[x];
                    float gx, gy;
                    if (x == 0) gx = tr[1] - t;
                    else if (x == nx - 1) gx = t - tr[x - 1];
                    else gx = 0.5f * (tr[x + 1] - tr[x - 1]);
                    if (y == 0) gy = tr[nx + x] - t;
                    else if (y == ny - 1) gy = t - tr[x - nx];
                    else gy = 0.5f * (tr[nx + x] - tr[x - nx]);
                    const float cs = XT ? xt_get(C, EPR_XT_C, s, x) : line_const(C.c, s);
                    v[r0] = gather_px(C, A, pb, y, x, cs * gy, cs * gx, s);
                } else if constexpr (MODE == FWD_SOLVE_LOCAL) {
                    v[r0] = resid(C, A, pb, (size_t)y * nx + x, s);
                } else {
                    v[r0] = __ldg(&A.G[pb + (size_t)y * nx + x]);
                }
                if constexpr (MODE != FWD_LOAD) {
                    if (sl == 0) {
                        const size_t q = (size_t)y * nx + x;
                        float r;
                        r = __ldg(&A.P[pb + q]);
                        ra += r * r;
                    }
                }
            }
            zs[PR::idx(m * sm + x)] = make_float2(v[0], v[1]);
        }
        __syncthreads();
        eprfft::fft<PR, -1, kEPT>(zs, nx, A.lgRP, 1, sm, A.tw, T, tid);
        // epilogue: unpack the two real spectra and store k < nx/2
        float2* Sb = A.S + ((size_t)b * A.nl + sl) * (size_t)ny * half;
        const float inv_half = 1.f / (float)half;
        for (int e = tid; e < RP * half; e += T) {
            const int m = RP == 1 ? 0 : fdiv(e, inv_half);
            const int k = e - m * half;
            const int y0 = yb + 2 * m;
            const int zb = m * sm;
            float2 X0, X1;
            if (k == 0) {
                const float2 z0 = zs[PR::idx(zb)], zn = zs[PR::idx(zb + half)];
                X0 = make_float2(z0.x, zn.x);
                X1 = make_float2(z0.y, zn.y);
            } else {
                const float2 a = zs[PR::idx(zb + k)], bb = cconj(zs[PR::idx(zb + nx - k)]);
                const float2 sp = cadd(a, bb), df = csub(a, bb);
                X0 = make_float2(0.5f * sp.x, 0.5f * sp.y);
                X1 = make_float2(0.5f * df.y, -0.5f * df.x);
            }
            Sb[(size_t)y0 * half + k] = X0;
            Sb[(size_t)(y0 + 1) * half + k] = X1;
        }
        __syncthreads();
    }

    if constexpr (MODE != FWD_LOAD) {   // |D - P|^2 partials; rho is formed by the column pass
        float rb = 0.f;
        block_sum2(ra, rb, red);
        store_partials(A.part_c + (size_t)b * A.max_blocks, nullptr, ra, rb);
    }
}

// XT: an x-dependent spectrum, the update's constants read per column.
template <int MODE, int NS, bool XT = false>
__global__ void __launch_bounds__(512, 2) k_row_inv(const EprConsts C, const RowArgs A)
{
    extern __shared__ __align__(16) float2 zs[];
    __shared__ float red[64];
    const int b = row_batch_index();
    epr_grid_wait();
    if (A.check_done && A.st[b].done) return;
    epr_grid_release();
    const int nx = C.nx, ny = C.ny, half = C.half;
    const int T = blockDim.x, tid = threadIdx.x;
    const int RP = A.RP, sm = nx + kPad;
    const size_t npix = (size_t)nx * ny;
    const size_t pb = (size_t)b * npix;
    const int yb = blockIdx.x * RP * 2;
    const int nl = NS ? NS : A.nl;
    float* acc = reinterpret_cast<float*>(zs + ((PR::len(RP * sm) + 1) & ~1));  // [2 RP][nx]
    const float inv_nx = 1.f / (float)nx, inv_half = 1.f / (float)half;
    float da = 0.f, db = 0.f;

    for (int sl = 0; sl < nl; ++sl) {
        const int s = A.line0 + sl;
        const float2* Sb = A.S + ((size_t)b * A.nl + sl) * (size_t)ny * half;
        // unpack Z[k] = X0[k] + i X1[k] over the full row
        for (int e = tid; e < RP * half; e += T) {
            const int m = RP == 1 ? 0 : fdiv(e, inv_half);
            const int k = e - m * half;
            const int y0 = yb + 2 * m;
            const float2 s0 = Sb[(size_t)y0 * half + k];
            const float2 s1 = Sb[(size_t)(y0 + 1) * half + k];
            const int zb = m * sm;
            if (k == 0) {
                zs[PR::idx(zb)] = make_float2(s0.x, s1.x);
                zs[PR::idx(zb + half)] = make_float2(s0.y, s1.y);
            } else {
                zs[PR::idx(zb + k)] = make_float2(s0.x - s1.y, s0.y + s1.x);
                zs[PR::idx(zb + nx - k)] = make_float2(s0.x + s1.y, s1.x - s0.y);
            }
        }
        __syncthreads();
        eprfft::fft<PR, +1, kEPT>(zs, nx, A.lgRP, 1, sm, A.tw, T, tid);
#pragma unroll 2
        for (int k = 0; k < kEPT; ++k) {
            const int e = tid + k * T;
            const int m = RP == 1 ? 0 : fdiv(e, inv_nx);
            const int x = e - m * nx;
            const float2 h = zs[PR::idx(m * sm + x)];
            const size_t q0 = pb + (size_t)(yb + 2 * m) * nx + x;
            if constexpr (MODE == INV_UPDATE) {
                const float fs = XT ? xt_get(C, EPR_XT_F, s, x) : line_const(C.f, s);
                const float mus = XT ? xt_get(C, EPR_XT_MU, s, x) : line_const(C.mu, s);
                const float w = XT ? xt_get(C, EPR_XT_WPROJ, s, x) : line_const(C.wproj, s);
                const float om_f = A.omega / fs;
                const float t0 = A.Out[q0], t1 = A.Out[q0 + nx];
                const float l0 = w * log_ratio(t0, h.x, om_f, mus, A.eps);
                const float l1 = w * log_ratio(t1, h.y, om_f, mus, A.eps);
                if (nl == 1) {
                    const float n0 = t0 - l0, n1 = t1 - l1;
                    A.Out[q0] = n0;
                    A.Out[q0 + nx] = n1;
                    da += l0 * l0 + l1 * l1;
                    db += n0 * n0 + n1 * n1;
                } else {
                    float* a0 = acc + (2 * m) * nx + x;
                    if (sl == 0) {
                        a0[0] = l0;
                        a0[nx] = l1;
                    } else {
                        a0[0] += l0;
                        a0[nx] += l1;
                    }
                }
            } else {
                A.Out[q0] = h.x;
                A.Out[q0 + nx] = h.y;
            }
        }
        __syncthreads();
    }

    if constexpr (MODE == INV_UPDATE) {
        if (nl > 1) {
            for (int k = 0; k < kEPT; ++k) {
                const int e = tid + k * T;
                const int m = RP == 1 ? 0 : fdiv(e, inv_nx);
                const int x = e - m * nx;
                const size_t q0 = pb + (size_t)(yb + 2 * m) * nx + x;
                const float l0 = acc[(2 * m) * nx + x], l1 = acc[(2 * m + 1) * nx + x];
                const float n0 = A.Out[q0] - l0, n1 = A.Out[q0 + nx] - l1;
                A.Out[q0] = n0;
                A.Out[q0 + nx] = n1;
                da += l0 * l0 + l1 * l1;
                db += n0 * n0 + n1 * n1;
            }
        }
        block_sum2(da, db, red);   // kappa partials, finalised by the next forward pass
        store_partials(A.part_a + (size_t)b * A.max_blocks, A.part_b + (size_t)b * A.max_blocks, da,
                       db);
    }
}

// Start of a solve: the state of the projection and the error word cleared,
// T := 0 (T may be NULL), and the block partials of |D|^2 (deterministic: a
// fixed-order sum follows).  One launch instead of three fills and a
// reduction.
__global__ void __launch_bounds__(256) k_solve_begin(const float* __restrict__ D, size_t npd, float* T,
                                                     size_t npix, double* part, int max_blocks,
                                                     EprProjState* st, unsigned int* err)
{
    __shared__ float red[64];
    const int b = blockIdx.y;
    const size_t first = blockIdx.x * (size_t)blockDim.x + threadIdx.x, step = (size_t)gridDim.x * blockDim.x;
    if (blockIdx.x == 0) {
        int* w = reinterpret_cast<int*>(&st[b]);
        for (int i = threadIdx.x; i < (int)(sizeof(EprProjState) / sizeof(int)); i += blockDim.x) w[i] = 0;
        if (b == 0 && threadIdx.x == 0) *err = 0u;
    }
    if (T) {
        float4* Tb = reinterpret_cast<float4*>(T + (size_t)b * npix);
        for (size_t i = first; i < npix / 4; i += step) Tb[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const float4* Db = reinterpret_cast<const float4*>(D + (size_t)b * npd);
    float a = 0.f, z = 0.f;
    for (size_t i = first; i < npd / 4; i += step) {
        const float4 v = __ldg(&Db[i]);
        a += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
    }
    block_sum2(a, z, red);
    if (threadIdx.x == 0) part[(size_t)b * max_blocks + blockIdx.x] = (double)a;
}

// A NaN or an infinity anywhere in D makes the sum non-finite (finite float
// squares cannot overflow a double sum): flagged in the device error word.
__global__ void __launch_bounds__(256) k_sumsq_final(const double* part, int nparts, int max_blocks,
                                                     double scale, EprProjState* st, unsigned int* err)
{
    const int b = blockIdx.x;
    double s, none;
    sum_partials(part + (size_t)b * max_blocks, nullptr, nparts, s, none);
    if (threadIdx.x != 0) return;
    st[b].dnorm2 = s * scale;
    if (!isfinite(s)) atomicOr(err, EPR_DEVERR_NONFINITE);
}

template <class F>
void each_table(F f)
{
    const RowKernels* (*const tables[])(int*) = {epr_row_table_short,    epr_row_table_mid,
                                                 epr_row_table_long,     epr_row_table_ragged_a,
                                                 epr_row_table_ragged_b, epr_row_table_ragged_c};
    for (auto t : tables) {
        int n = 0;
        const RowKernels* k = t(&n);
        for (int i = 0; i < n; ++i) f(k[i]);
    }
}

// Lengths up to 512 have blocks of several row pairs (96 to 128 threads) and of
// one.  Fewer blocks of several than this (four per SM) leave SMs idle or with
// too few warps: one pair per block is then the faster.  Solve iterations, us,
// with several pairs and with one: 256^2 18.4, 15.1; 16 of 256^2 (512 blocks)
// 29.8, 27.8; 32 (1024) 42.6, 44.1; four of 512^2 (512) 27.5, 26.6; 64 (8192)
// 217, 243; eight of 384^2 (768) 34.3, 35.9.  Longer rows are one pair per
// block at every count: two pairs (256 threads) took 115 for eight of 1024^2
// where one takes 110, and 796 where it takes 697 for 16 of four lines.
constexpr int kRowMinBlocks = 4 * EPR_SMS;

}  // namespace

struct EprRowLaunch {
    int RP, lgRP, threads;
    size_t smem;            // of the runtime-sized kernels
    const RowKernels* k;    // compile-time kernels of this length and RP, or NULL
};

// solve: the passes of an iteration (of a plan with an x-dependent spectrum,
// which not every length has compile-time kernels for).
EprRowLaunch epr_row_config(const EprConsts& C, int batch, bool solve)
{
    EprRowLaunch L = {};
    const RowKernels *many = nullptr, *one = nullptr;
    each_table([&](const RowKernels& k) {
        if (k.nx != C.nx) return;
        if (k.rp > 1 && (C.ny / 2) % k.rp == 0) many = &k;
        if (k.rp == 1) one = &k;
    });
    int rp = 1;   // of the runtime-sized kernels
    while (rp * 2 * C.nx <= 2048 && (C.ny / 2) % (rp * 2) == 0) rp *= 2;
    if (many && (long long)(C.ny / (2 * many->rp)) * epr_rule_batch(C, batch) >= kRowMinBlocks) L.k = many;
    else if (one) L.k = one;
    if (solve && C.xt && L.k && !L.k->xfwd1) L.k = nullptr;
    L.RP = L.k ? L.k->rp : rp;
    L.lgRP = 0;
    while ((1 << L.lgRP) < L.RP) ++L.lgRP;
    L.threads = C.nx * L.RP / kEPT;
    // FFT rows, then the staged thickness rows (forward) or line accumulators
    // (inverse); the larger of the two
    const size_t extra = (size_t)(2 * L.RP + 2) * C.nx * sizeof(float);
    L.smem = row_fft_smem(C.nx, L.RP) + extra;
    return L;
}

// mode: 0 = non-local solve, 1 = local solve, 2 = load real map G.
// FWD_SOLVE_NL reads the residual D - P from P and the split residuals from P_s.
// In a solve (it > 0) a further block finalises kappa of iteration it - 1
// against tol.
cudaError_t epr_launch_row_fwd(const EprConsts& C, const EprWork& W, int mode, const float* T,
                               const float* D, const float* G, int line0, int nl, int it,
                               float tol, int batch, int check_done, cudaStream_t stream)
{
    const EprRowLaunch L = epr_row_config(C, batch, mode != FWD_LOAD);
    RowArgs A = {};
    A.T = T; A.D = D; A.G = mode == FWD_LOAD ? G : nullptr;
    A.P = W.P; A.Ps = W.Ps;
    A.S = W.S; A.st = W.st; A.part_a = W.part_a; A.part_b = W.part_b; A.part_c = W.part_c;
    A.hist = W.kappa_hist; A.hist_len = W.hist_len; A.max_blocks = W.max_blocks;
    A.tw = W.tw_x; A.RP = L.RP; A.lgRP = L.lgRP; A.line0 = line0; A.nl = nl; A.it = it;
    A.check_done = check_done;
    A.fin = mode != FWD_LOAD && it > 0;
    A.tol = tol;
    const dim3 grid(C.ny / (2 * L.RP), batch);
    const bool one = nl == 1, pdl = C.pdl != 0;
    // compile-time kernels: a line per grid z.  The residual D - P is in P
    // and, with several lines, the split residuals in P_s (written by the
    // splat flush, the long-shift passes or the stencil kernel); the local closure back-transports with
    // the identity.
    RowKernel k = nullptr;
    size_t smem = 0;
    int threads = L.k ? L.k->threads : 0;
    if (L.k && mode == FWD_SOLVE_NL) {
        smem = L.k->smem_fwd;
        if (C.xt) k = one ? L.k->xfwd1 : L.k->xfwdn;
        else if (one && W.row_occ6 && L.k->fwd1_6) k = L.k->fwd1_6;
        else k = one && L.k->fwd1 ? L.k->fwd1 : L.k->fwdn;
        if (k == L.k->fwd1 && L.k->threads16) {
            threads = L.k->threads16;
            smem = L.k->smem_plain;
        }
    } else if (L.k) {
        smem = L.k->smem_plain;
        threads = L.k->threads_plain;
        k = L.k->plain;
    }
    cudaError_t e = cudaSuccess;
    auto go = [&](auto kernel) {
        e = epr_launch_kernel(pdl, kernel, grid, dim3(L.threads), L.smem, stream, C, A);
    };
    if (k) {
        e = epr_launch_kernel(pdl, k, dim3(grid.x + (A.fin ? 1 : 0), grid.y, nl), dim3(threads), smem, stream, C,
                              A);
    } else if (mode == FWD_SOLVE_NL && C.xt) {   // per-column shift constants
        go(k_row_fwd<FWD_SOLVE_NL, 0, true>);
    } else if (mode == FWD_SOLVE_NL) {
        if (one) go(k_row_fwd<FWD_SOLVE_NL, 1>);
        else go(k_row_fwd<FWD_SOLVE_NL, 0>);
    } else if (mode == FWD_SOLVE_LOCAL) {
        go(k_row_fwd<FWD_SOLVE_LOCAL, 0>);
    } else {
        go(k_row_fwd<FWD_LOAD, 1>);
    }
    epr_count_launch(1);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t epr_launch_row_inv(const EprConsts& C, const EprWork& W, int mode, float* Out,
                               int line0, int nl, int it, float omega, float eps, float tol,
                               int batch, int check_done, cudaStream_t stream)
{
    const EprRowLaunch L = epr_row_config(C, batch, mode == INV_UPDATE);
    RowArgs A = {};
    A.Out = Out; A.S = W.S; A.st = W.st; A.part_a = W.part_a; A.part_b = W.part_b;
    A.hist_len = W.hist_len; A.max_blocks = W.max_blocks;
    A.tw = W.tw_x; A.RP = L.RP; A.lgRP = L.lgRP; A.line0 = line0; A.nl = nl; A.it = it;
    A.omega = omega; A.eps = eps; A.tol = tol; A.check_done = check_done;
    const dim3 grid(C.ny / (2 * L.RP), batch);
    const bool one = nl == 1, pdl = C.pdl != 0;
    RowKernel k = nullptr;
    size_t smem = 0;
    int threads = L.k ? L.k->threads : 0;
    if (L.k && mode == INV_UPDATE) {
        if (C.xt) k = one ? L.k->xinv1 : L.k->xinvn;
        else if (one && W.row_occ6 && L.k->inv1_6) k = L.k->inv1_6;
        else k = one && L.k->inv1 ? L.k->inv1 : L.k->invn;
        smem = !one ? L.k->smem_invn : k == L.k->invn ? L.k->smem_invn1 : L.k->smem_inv1;
        if (k == L.k->inv1 && L.k->threads16) {
            threads = L.k->threads16;
            smem = L.k->smem_plain;
        }
    } else if (L.k) {
        k = L.k->store;
        threads = L.k->threads_plain;
        smem = L.k->smem_plain;
    }
    cudaError_t e = cudaSuccess;
    auto go = [&](auto kernel) {
        e = epr_launch_kernel(pdl, kernel, grid, dim3(L.threads), L.smem, stream, C, A);
    };
    if (k) {
        e = epr_launch_kernel(pdl, k, grid, dim3(threads), smem, stream, C, A);
    } else if (mode == INV_UPDATE && C.xt) {   // per-column update constants
        go(k_row_inv<INV_UPDATE, 0, true>);
    } else if (mode == INV_UPDATE) {
        if (nl == 1) go(k_row_inv<INV_UPDATE, 1>);
        else go(k_row_inv<INV_UPDATE, 0>);
    } else {
        go(k_row_inv<INV_STORE, 1>);
    }
    epr_count_launch(1);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// Start of a solve (two small launches): see k_solve_begin; |D|^2 of each
// projection (D of npd pixels) times scale goes into the solver state.
cudaError_t epr_launch_solve_begin(const EprConsts& C, const EprWork& W, const float* D, float* T,
                                   int batch, size_t npd, size_t npix, double scale,
                                   cudaStream_t stream)
{
    size_t parts = (npix / 4 + 255) / 256;   // a float4 per thread, up to 4 blocks per SM
    if (parts > 4 * EPR_SMS) parts = 4 * EPR_SMS;
    if (parts > (size_t)W.max_blocks) parts = W.max_blocks;
    k_solve_begin<<<dim3((unsigned)parts, batch), 256, 0, stream>>>(D, npd, T, npix, W.part_a, W.max_blocks,
                                                                    W.st, W.err);
    k_sumsq_final<<<batch, 256, 0, stream>>>(W.part_a, (int)parts, W.max_blocks, scale, W.st, W.err);
    epr_count_launch(2);
    return cudaGetLastError();
}

// Blocks of a row pass (the number of partials a reduction adds up).
int epr_row_blocks(const EprConsts& C, int batch) { return C.ny / (2 * epr_row_config(C, batch, true).RP); }

// Largest radix of the plain row transforms of a launch (which stage table they
// read); 0: the runtime-sized ones.
int epr_row_plain_radix(const EprConsts& C, int batch)
{
    const EprRowLaunch L = epr_row_config(C, batch, false);
    return L.k ? row_maxr(C.nx * L.RP / L.k->threads_plain) : 0;
}

namespace {

// kappa of the last iteration of a solve (the forward pass of a following
// iteration finalises the others): one block per projection.
__global__ void __launch_bounds__(256) k_finalize_kappa(EprProjState* st, const double* part_a,
                                                        const double* part_b, int max_blocks,
                                                        int nblk, double* hist, int hist_len,
                                                        int it, float tol)
{
    const int b = blockIdx.x;
    epr_grid_wait();
    if (st[b].done) return;   // converged earlier: the partials are stale
    finalize_kappa(&st[b], part_a + (size_t)b * max_blocks, part_b + (size_t)b * max_blocks, nblk,
                   hist ? hist + (size_t)b * hist_len : nullptr, hist_len, it, tol);
}

}  // namespace

cudaError_t epr_launch_finalize_kappa(const EprConsts& C, const EprWork& W, int it, float tol,
                                      int batch, cudaStream_t stream)
{
    const cudaError_t e =
        epr_launch_kernel(C.pdl != 0, k_finalize_kappa, dim3(batch), dim3(256), 0, stream, W.st,
                          (const double*)W.part_a, (const double*)W.part_b, W.max_blocks,
                          epr_row_blocks(C, batch), W.kappa_hist, W.hist_len, it, tol);
    epr_count_launch(1);
    return e != cudaSuccess ? e : cudaGetLastError();
}

namespace {

std::mutex g_row_mu;
constexpr int kMaxDevices = 64, kMaxEntries = 128;
bool g_row_ready[kMaxDevices][kMaxEntries + 1];   // the last: the runtime-sized kernels
bool g_row_plain_ready[kMaxDevices];

cudaError_t allow_runtime_sized()
{
    cudaError_t e = cudaSuccess;
    auto allow = [&](auto kernel) { if (e == cudaSuccess) e = epr_allow_max_smem(kernel); };
    allow(k_row_fwd<FWD_SOLVE_NL, 1>);
    allow(k_row_fwd<FWD_SOLVE_NL, 0>);
    allow(k_row_fwd<FWD_SOLVE_LOCAL, 0>);
    allow(k_row_fwd<FWD_LOAD, 1>);
    allow(k_row_inv<INV_UPDATE, 1>);
    allow(k_row_inv<INV_UPDATE, 0>);
    allow(k_row_inv<INV_STORE, 1>);
    allow(k_row_fwd<FWD_SOLVE_NL, 0, true>);
    allow(k_row_inv<INV_UPDATE, 0, true>);
    return e;
}

}  // namespace

// Lets the row kernels of length nx (nx = 0: the plain transforms of every
// length) use the device's opt-in shared memory; once per device and length,
// not while a stream is being captured.
cudaError_t epr_row_init(int nx)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(g_row_mu);
    if (!g_row_ready[dev][kMaxEntries]) {
        e = allow_runtime_sized();
        if (e != cudaSuccess) return e;
        g_row_ready[dev][kMaxEntries] = true;
    }
    if (nx == 0 && g_row_plain_ready[dev]) return cudaSuccess;
    int i = 0;
    each_table([&](const RowKernels& k) {
        const int at = i++;
        if (e != cudaSuccess || at >= kMaxEntries) return;
        if (nx == 0) {
            e = epr_allow_max_smem(k.plain);
            if (e == cudaSuccess) e = epr_allow_max_smem(k.store);
            return;
        }
        if (k.nx != nx || g_row_ready[dev][at]) return;
        const RowKernel all[] = {k.fwd1, k.fwdn, k.plain, k.inv1, k.invn, k.store,
                                 k.fwd1_6, k.inv1_6, k.xfwd1, k.xfwdn, k.xinv1, k.xinvn};
        for (RowKernel q : all)
            if (q && e == cudaSuccess) e = epr_allow_max_smem(q);
        g_row_ready[dev][at] = e == cudaSuccess;
    });
    if (nx == 0 && e == cudaSuccess) g_row_plain_ready[dev] = true;
    return e;
}
