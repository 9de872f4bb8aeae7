// The row passes on the compile-time FFT engine: kernels templated on the row
// length, instantiated for groups of lengths in rowfft_ct_*.cu and launched
// through tables of kernel pointers (rowfft.cu, which also holds the
// runtime-sized passes of the remaining lengths and describes the passes).
#pragma once

#include <type_traits>

#include "epr_internal.cuh"
#include "fft.cuh"

namespace eprrow {

constexpr int kEPT = 8;   // complex elements per thread in the row FFT
constexpr int kPad = 4;   // float2 padding between packed rows in shared memory

struct RowArgs {
    const float* T;          // [B][ny][nx]
    const float* D;          // [B][ny][nx]
    const float* P;          // [B][ny][nx]   residual D - P
    const float* Ps;         // [B][ns][ny][nx]   split residuals r_s (ns > 1)
    const float* G;          // [B][ny][nx] real input of a plain transform, else NULL
    float* Out;              // [B][ny][nx] real output (INV_STORE) or T (INV_UPDATE)
    float2* S;               // [B][nl][ny][nx/2]
    EprProjState* st;
    double* part_a;          // [B][max_blocks] inverse pass partials (kappa)
    double* part_b;
    double* part_c;          // [B][max_blocks] forward pass partials (rho)
    double* hist;            // kappa history (finalised by the forward pass)
    const float2* tw;        // twiddle tables of length nx
    int RP, lgRP;            // row pairs per block
    int line0, nl;           // first physical line, number of lines handled
    int it, hist_len, max_blocks;
    int check_done;
    int fin;                 // forward: a further block finalises kappa of iteration it - 1
    float omega, eps, tol;
};


typedef void (*RowKernel)(const EprConsts, const RowArgs);

// The kernels of one row length and block shape; a null pointer: none (the
// several-line kernel serves one line too where fwd1 or inv1 is null).
struct RowKernels {
    int nx, rp, threads;   // row length, row pairs per block, threads (forward and inverse)
    RowKernel fwd1, fwdn;  // gather, one line or a line per grid z
    RowKernel plain;       // the split residuals at the pixel itself, or a real map
    RowKernel inv1, invn;  // inverse and update, one line or looping over them
    RowKernel store;       // inverse to a real map
    RowKernel fwd1_6, inv1_6;        // six blocks per SM
    RowKernel xfwd1, xfwdn, xinv1, xinvn;   // x-dependent spectrum
    size_t smem_fwd, smem_plain, smem_inv1, smem_invn1, smem_invn;   // invn1: one line on invn
    int threads16;         // one-line kernels with 16 elements per thread: their block, or 0
    int threads_plain;     // block of plain and store
};

}  // namespace eprrow

#ifdef EPR_ROW_KERNELS
namespace {

using namespace eprrow;
using PR = eprfft::PadRow;    // shared layout of the packed rows
using PP = eprfft::PadPlain;  // the same, of the plain transforms

// Projection of a row-pass block.  The row passes walk the batch from the
// last projection to the first (grid y), the splat and the column pass from
// the first to the last: each kernel starts on the projections its
// predecessor touched last, whose data are still in L2.
__device__ __forceinline__ int row_batch_index() { return (int)(gridDim.y - 1 - blockIdx.y); }
// One block of a forward solve pass (line 0) turns the inverse pass's nblk
// partials of the previous iteration into kappa, the iteration count and
// the convergence flag, unless the projection had already converged; the
// grid dependency wait has made every partial visible.  The other blocks of
// this pass may not see the flag: a projection that converges here runs this
// pass and the splat before it once more, which changes nothing it keeps.
// The compile-time passes launch one block more for it (double-precision sums
// of up to 2048 partials are a serial chain: 2.6 us of a 9.8 us pass over
// 256^2 when a block did both).
__device__ __forceinline__ void fwd_finalize_kappa(const RowArgs& A, int b, bool lead, int nblk)
{
    if (A.fin && lead && !A.st[b].done)
        finalize_kappa(&A.st[b], A.part_a + (size_t)b * A.max_blocks,
                       A.part_b + (size_t)b * A.max_blocks, nblk,
                       A.hist ? A.hist + (size_t)b * A.hist_len : nullptr, A.hist_len, A.it - 1,
                       A.tol);
}

// ln(1 + q) for |q| < 1/4 from ln(1 + q) = 2 atanh(z), z = q / (2 + q), and
// the Taylor series of atanh: 2 z (1 + z^2/3 + z^4/5 + ... + z^10/11).  Here
// |z| < 1/7, so the first omitted term, 2 |z|^13 / 13, is below 1.2e-11 |z|:
// the error is the rounding of the few operations.
__device__ __forceinline__ float log1p_atanh(float q)
{
    const float z = __fdividef(q, 2.f + q);
    const float w = z * z;
    float p = fmaf(w, 1.f / 11.f, 1.f / 9.f);
    p = fmaf(w, p, 1.f / 7.f);
    p = fmaf(w, p, 1.f / 5.f);
    p = fmaf(w, p, 1.f / 3.f);
    p = fmaf(w, p, 1.f);
    return 2.f * z * p;
}

// ln(I'_s / I_s) for the update of one pixel and line, I_s = f_s exp(-mu_s t),
// I'_s = max(I_s + omega h_s, eps f_s).  With q = (omega / f_s) h_s exp(mu_s t)
// = omega h_s / I_s, the ratio is 1 + q above the floor, and
// eps f_s / I_s = eps exp(mu_s t) at it.  om_f = omega / f_s.
__device__ __forceinline__ float log_ratio(float t, float h, float om_f, float mus, float eps)
{
    const float Einv = __expf(mus * t);        // f_s / I_s
    const float q = om_f * h * Einv;
    if (1.f + q >= eps * Einv) return (fabsf(q) < 0.25f) ? log1p_atanh(q) : logf(1.f + q);
    return logf(eps) + mus * t;
}

// largest radix of a row transform with EPT elements per thread
__host__ __device__ constexpr int row_maxr(int EPT) { return EPT >= 16 ? 16 : EPT >= 8 ? 8 : 4; }

__device__ __forceinline__ float ex2_approx(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// log_ratio of two pixels of one column (packed): both above the floor with
// |q| < 1/4 by the series of log1p_atanh, else one by one.  The update is
// bound by instruction issue (70 % active in a batch); the packed form takes
// 21 arithmetic instructions for two pixels.
__device__ __forceinline__ float2 log_ratio2(float2 t, float2 h, float om_f, float mus, float eps)
{
    const float mk = mus * 1.4426950408889634f;   // e^(mu t) = 2^(mk t)
    const float2 a = mul2(both(mk), t);
    const float2 E = make_float2(ex2_approx(a.x), ex2_approx(a.y));   // f_s / I_s
    const float2 q = mul2(mul2(both(om_f), h), E);
    const float2 r = add2(both(1.f), q), fl = mul2(both(eps), E);
    if (!(fmaxf(fabsf(q.x), fabsf(q.y)) < 0.25f && r.x >= fl.x && r.y >= fl.y))
        return make_float2(log_ratio(t.x, h.x, om_f, mus, eps), log_ratio(t.y, h.y, om_f, mus, eps));
    const float2 d = add2(both(2.f), q);
    const float2 z = mul2(q, make_float2(rcp_approx(d.x), rcp_approx(d.y)));
    const float2 w = mul2(z, z);
    float2 p = fma2(w, both(1.f / 11.f), both(1.f / 9.f));
    p = fma2(w, p, both(1.f / 7.f));
    p = fma2(w, p, both(1.f / 5.f));
    p = fma2(w, p, both(1.f / 3.f));
    p = fma2(w, p, both(1.f));
    return mul2(add2(z, z), p);
}

// blocks per SM that a block of T threads is bounded to: 64 registers, or 80
// where `threads` is 768 (the several-line update of ragged lengths with
// several row pairs, whose per-element row and column would spill)
// (a block of 352 or 384 threads fits three times into 1152)
constexpr int row_min_blocks(int T, int threads = 1024)
{
    const int t32 = (T + 31) / 32 * 32;
    const int b = (threads == 1024 && t32 >= 352 && t32 <= 384 ? 1152 : threads) / t32;
    return b < 1 ? 1 : b > 16 ? 16 : b;
}

template <int NX>
__host__ __device__ constexpr int ct_lg(int v) { return v <= 1 ? 0 : 1 + ct_lg<NX>(v / 2); }

// packed row pair m and column x of element tid + k T (0 <= that < NX RP)
template <int NX, int RP, int T>
__device__ __forceinline__ void row_of(int tid, int k, int& m, int& x)
{
    if constexpr (NX % T == 0) {   // the thread's elements of one k are one column's
        m = k * T / NX;
        x = tid + k * T % NX;
    } else {
        m = RP == 1 ? 0 : (int)((unsigned)(tid + k * T) / NX);
        x = tid + k * T - m * NX;
    }
}

// The gather of one pixel with any mapped point: corners outside the grid
// read 0 (Eq. 4); a shift that is not finite or beyond the grid reads only 0.
__device__ __noinline__ float gather_guarded(const float* R, int y, int x, float uy, float ux, int ny,
                                             int nx)
{
    const float lim = 2.f * (float)(nx > ny ? nx : ny);
    ux = fminf(fmaxf(ux, -lim), lim);
    uy = fminf(fmaxf(uy, -lim), lim);
    const float fx = floorf(ux), fy = floorf(uy);
    const float dx = ux - fx, dy = uy - fy;
    const int cx = x + (int)fx, cy = y + (int)fy;
    const bool x0 = (unsigned)cx < (unsigned)nx, x1 = (unsigned)(cx + 1) < (unsigned)nx;
    float r00 = 0.f, r10 = 0.f, r01 = 0.f, r11 = 0.f;
    if ((unsigned)cy < (unsigned)ny) {
        const float* r = R + (size_t)cy * nx + cx;
        if (x0) r00 = __ldg(r);
        if (x1) r10 = __ldg(r + 1);
    }
    if ((unsigned)(cy + 1) < (unsigned)ny) {
        const float* r = R + (size_t)(cy + 1) * nx + cx;
        if (x0) r01 = __ldg(r);
        if (x1) r11 = __ldg(r + 1);
    }
    const float top = r00 + dx * (r10 - r00);
    const float bot = r01 + dx * (r11 - r01);
    return (1.f - dy) * top + dy * bot;
}

// Shared memory: the thickness rows yb - 1 .. yb + 2 RP, staged for the
// gradient, alias the FFT rows, which are written only after the last
// thickness read (row_fwd_smem).  256-thread one-line blocks run five per SM
// (48 registers).  With 16 elements per thread only the block's own 2 RP rows
// are staged (the rows above and below are read once per pixel, coalesced),
// so the FFT rows set the shared memory.
//
// OCC6: six 256-thread blocks per SM (40 registers) instead of five: better
// in a batch of projections, worse for one (the autotuner decides).
// XT: an x-dependent spectrum, the shift constant of each object column from
// the plan's table.
template <int NX, int RP, bool POLY, bool GATHER, bool OCC6 = false, bool XT = false, int EPT = kEPT>
__global__ void __launch_bounds__(NX * RP / EPT, OCC6 ? 6 : (NX * RP / EPT == 256 && !POLY) ? 5
                                                 : row_min_blocks(NX * RP / EPT))
k_row_fwd_ct(const EprConsts C, const RowArgs A)
{
    constexpr int T = NX * RP / EPT;
    static_assert(NX * RP % EPT == 0 && RP * (NX / 2) % T == 0, "every element has a thread");
    constexpr int MAXR = row_maxr(EPT);   // radix-16 stages with 16 elements per thread
    constexpr int kRim = EPT <= kEPT ? 1 : 0;   // rows staged above and below the block's own
    constexpr int SM = NX + kPad;
    constexpr int HALF = NX / 2;
    constexpr int LGRP = ct_lg<NX>(RP);
    using PF = std::conditional_t<GATHER, PR, PP>;
    constexpr int kRowLines = (NX + 31) / 32;   // 128-byte lines of a row
    extern __shared__ __align__(16) float2 zs[];
    __shared__ float red[64];
    const int b = row_batch_index();
    const int sl = POLY ? (int)blockIdx.z : 0;   // line of this block (polychromatic)
    const int ny = C.ny, tid = threadIdx.x;
    const size_t npix = (size_t)NX * ny;
    const size_t pb = (size_t)b * npix;
    const int bx = (int)blockIdx.x - (A.fin ? 1 : 0);   // row block
    const int yb = bx * RP * 2;
    if (A.fin && blockIdx.x == 0) {   // the block that finishes the last iteration, in the first wave
        epr_grid_wait();
        if (sl == 0) fwd_finalize_kappa(A, b, true, (int)gridDim.x - 1);
        return;
    }
    float* Ts = reinterpret_cast<float*>(zs);   // aliases the FFT rows (see above)
    if constexpr (GATHER) {   // T is not written by the predecessor: fetch it before the wait
        const float* Tb = A.T + pb;
        constexpr int Q4 = NX / 4;
        constexpr int NROWS = 2 * RP + 2 * kRim;
#pragma unroll
        for (int i0 = 0; i0 < NROWS * Q4; i0 += T) {
            const int i = i0 + tid;
            if (NROWS * Q4 % T == 0 || i < NROWS * Q4) {
                const int r = i / Q4, c4 = i % Q4;
                const int gy = min(max(yb - kRim + r, 0), ny - 1);
                cp_async16(reinterpret_cast<float4*>(Ts) + i,
                           reinterpret_cast<const float4*>(Tb + (size_t)gy * NX) + c4);
            }
        }
        cp_async_commit();
        if constexpr (kRim == 0) {
            for (int i = tid; i < 2 * kRowLines; i += T) {
                const int y = i < kRowLines ? yb - 1 : yb + 2 * RP;
                if (y >= 0 && y < ny) prefetch_l1(Tb + (size_t)y * NX + 32 * (i % kRowLines));
            }
        }
    }
    epr_grid_wait();
    if (A.check_done && A.st[b].done) {
        cp_async_wait_all();   // no copy may land after the block has left
        return;
    }
    const float cs = POLY ? line_const(C.c, A.line0 + sl) : C.c[0];
    // residual D - P (one line) or the line's split residual, or a real map
    const float* Rb = !GATHER && A.G ? A.G + pb
                      : POLY && C.ns > 1 ? A.Ps + (pb * C.ns + (size_t)(A.line0 + sl) * npix)
                                         : A.P + pb;
    const float* Rt = A.P + pb;   // D - P, for |D - P|^2
    // |D - P|^2 of the block's rows, while the thickness rows arrive; for one
    // line this also brings into L1 the rows that most corners lie in (and
    // the two next to them are asked for), so the gather below finds them
    float ra = 0.f;
    const bool norm = (GATHER || !A.G) && (!POLY || sl == 0);   // this block's share is wanted
    if (norm) {
        float2 own[EPT];
#pragma unroll
        for (int k = 0; k < EPT; ++k) {
            int m, x;
            row_of<NX, RP, T>(tid, k, m, x);
            const float* q = Rt + (size_t)(yb + 2 * m) * NX + x;
            own[k] = make_float2(__ldg(q), __ldg(q + NX));
        }
        if (GATHER && !POLY) {
            for (int i = tid; i < 2 * kRowLines; i += T) {
                const int y = i < kRowLines ? yb - 1 : yb + 2 * RP;
                if (y >= 0 && y < ny) prefetch_l1(Rb + (size_t)y * NX + 32 * (i % kRowLines));
            }
        }
        float2 r2 = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < EPT; ++k) r2 = fma2(own[k], own[k], r2);
        ra = r2.x + r2.y;
    }
    if (GATHER && POLY) {   // a line's own rows and the two next to them
        for (int i = tid; i < (2 * RP + 2) * kRowLines; i += T) {
            const int y = yb - 1 + i / kRowLines;
            if (y >= 0 && y < ny) prefetch_l1(Rb + (size_t)y * NX + 32 * (i % kRowLines));
        }
    }
    cp_async_wait_all();
    __syncthreads();
    float2 vk[EPT];   // the packed row pair values, stored once the thickness is dead
    // The gather of a row pair's two pixels (y0, x) and (y0 + 1, x), packed:
    // 126 -> 95 thread instructions per pixel of this kernel, 148 -> 135 us for
    // eight 2048^2 projections (with the loads ahead of the gather above).
    // Pixels whose four corners all lie on the grid load them unconditionally
    // on the spot; the others (the rim of the field) are flagged and redone
    // with guarded loads after the loop, so the loop has no branch between
    // one element's loads and the next's.
    unsigned int rim = 0u;   // bits 2 k + r0
    auto shift2 = [&](int k, int& x, int& y0, float2& ux, float2& uy) {
        int m;
        row_of<NX, RP, T>(tid, k, m, x);
        y0 = yb + 2 * m;
        const float* tr = Ts + (2 * m + kRim) * NX + x;
        const float* tg = A.T + pb + (size_t)y0 * NX + x;   // the same pixel in memory
        auto ld = [&](int o) { return tr[o]; };
        auto ld_rim = [&](int o) { return kRim || (RP > 1 && (o < 0 ? m > 0 : m < RP - 1)) ? tr[o] : __ldg(tg + o); };
        // edges (one-sided differences): with one row pair per block only the
        // first and last element of a thread can be an edge column, and only
        // the first (last) row of the pair the top (bottom) row
        const bool xlo = (RP > 1 || k == 0) && x == 0;
        const bool xhi = (RP > 1 || k == EPT - 1) && x == NX - 1;
        const bool ylo = y0 == 0, yhi = y0 + 1 == ny - 1;
        const float2 t = make_float2(ld(0), ld(NX));
        const float2 l = xlo ? t : make_float2(ld(-1), ld(NX - 1));
        const float2 r = xhi ? t : make_float2(ld(1), ld(NX + 1));
        const float2 up = make_float2(ylo ? t.x : ld_rim(-NX), t.x);
        const float2 dn = make_float2(t.y, yhi ? t.y : ld_rim(2 * NX));
        // half the shift constant multiplies the doubled central difference
        // (0.5 scales exactly), the whole one a one-sided difference
        const float csx = XT ? xt_get(C, EPR_XT_C, A.line0 + sl, x) : cs;
        const float ch = 0.5f * csx;
        ux = mul2(both(xlo || xhi ? csx : ch), sub2(r, l));
        uy = mul2(make_float2(ylo ? csx : ch, yhi ? csx : ch), sub2(dn, up));
    };
#pragma unroll
    for (int k = 0; k < EPT; ++k) {
        if constexpr (!GATHER) {   // identity back-transport of the local closure
            int m, x;
            row_of<NX, RP, T>(tid, k, m, x);
            const size_t q = (size_t)(yb + 2 * m) * NX + x;
            vk[k] = make_float2(__ldg(Rb + q), __ldg(Rb + q + NX));
        } else {
            int x, y0;
            float2 ux, uy;
            shift2(k, x, y0, ux, uy);
            int ix0, ix1, iy0, iy1;
            const float2 dx = floor_frac2(ux, ix0, ix1), dy = floor_frac2(uy, iy0, iy1);
            const int cx0 = x + ix0, cx1 = x + ix1, cy0 = y0 + iy0, cy1 = y0 + 1 + iy1;
            const bool in0 = (unsigned)cx0 < (unsigned)(NX - 1) && (unsigned)cy0 < (unsigned)(ny - 1);
            const bool in1 = (unsigned)cx1 < (unsigned)(NX - 1) && (unsigned)cy1 < (unsigned)(ny - 1);
            if (!in0) rim |= 1u << (2 * k);
            if (!in1) rim |= 2u << (2 * k);
            const float* p0 = Rb + (in0 ? cy0 * NX + cx0 : 0);
            const float* p1 = Rb + (in1 ? cy1 * NX + cx1 : 0);
            const float2 r00 = make_float2(__ldg(p0), __ldg(p1));
            const float2 r10 = make_float2(__ldg(p0 + 1), __ldg(p1 + 1));
            const float2 r01 = make_float2(__ldg(p0 + NX), __ldg(p1 + NX));
            const float2 r11 = make_float2(__ldg(p0 + NX + 1), __ldg(p1 + NX + 1));
            const float2 top = fma2(dx, sub2(r10, r00), r00);
            const float2 bot = fma2(dx, sub2(r11, r01), r01);
            vk[k] = fma2(dy, bot, mul2(sub2(both(1.f), dy), top));
        }
    }
    if (GATHER && rim) {
#pragma unroll
        for (int k = 0; k < EPT; ++k) {
            if (!((rim >> (2 * k)) & 3u)) continue;
            int x, y0;
            float2 ux, uy;
            shift2(k, x, y0, ux, uy);
            if ((rim >> (2 * k)) & 1u) vk[k].x = gather_guarded(Rb, y0, x, uy.x, ux.x, ny, NX);
            if ((rim >> (2 * k)) & 2u) vk[k].y = gather_guarded(Rb, y0 + 1, x, uy.y, ux.y, ny, NX);
        }
    }
    if constexpr (GATHER) __syncthreads();   // every thickness read is done
    if constexpr (RP == 1 && eprfft::ct_radix(NX, 0, MAXR) == EPT) {
        // vk[r] = element tid + r T, the first stage's operands
        eprfft::stage0_regs<PF, -1, NX, EPT, MAXR>(vk, zs, tid);
        eprfft::fft_ct<PF, -1, NX, EPT, LGRP, 1, SM, 1, MAXR>(zs, A.tw, tid);
    } else {
#pragma unroll
        for (int k = 0; k < EPT; ++k) {
            int m, x;
            row_of<NX, RP, T>(tid, k, m, x);
            zs[PR::idx(m * SM + x)] = vk[k];
        }
        __syncthreads();
        eprfft::fft_ct<PF, -1, NX, EPT, LGRP, 1, SM, 0, MAXR>(zs, A.tw, tid);
    }
    epr_grid_release();
    float2* Sb = A.S + ((size_t)b * A.nl + sl) * (size_t)ny * HALF;
#pragma unroll 2
    for (int i0 = 0; i0 < RP * HALF; i0 += T) {
        const int e = i0 + tid;
        const int m = e / HALF, k = e % HALF;
        const int y0 = yb + 2 * m;
        const int zb = m * SM;
        float2 X0, X1;
        if (k == 0) {
            const float2 z0 = zs[PR::idx(zb)], zn = zs[PR::idx(zb + HALF)];
            X0 = make_float2(z0.x, zn.x);
            X1 = make_float2(z0.y, zn.y);
        } else {
            const float2 a = zs[PR::idx(zb + k)], bb = cconj(zs[PR::idx(zb + NX - k)]);
            const float2 sp = cadd(a, bb), df = csub(a, bb);
            X0 = make_float2(0.5f * sp.x, 0.5f * sp.y);
            X1 = make_float2(0.5f * df.y, -0.5f * df.x);
        }
        Sb[(size_t)y0 * HALF + k] = X0;
        Sb[(size_t)(y0 + 1) * HALF + k] = X1;
    }
    if (!norm) return;
    float rb = 0.f;
    block_sum2(ra, rb, red);   // |D - P|^2 partials; rho is formed by the column pass
    if (tid == 0) A.part_c[(size_t)b * A.max_blocks + bx] = (double)ra;
}

// Z[k] = X0[k] + i X1[k] of the block's row pairs over the full rows, into
// zs; ends with a barrier.
template <int NX, int RP, int EPT>
__device__ __forceinline__ void inv_unpack(const float2* __restrict__ Sb, float2* zs, int yb, int tid)
{
    constexpr int T = NX * RP / EPT, HALF = NX / 2, SM = NX + kPad;
    static_assert(NX * RP % EPT == 0 && RP * HALF % T == 0, "every element has a thread");
#pragma unroll 2
    for (int i0 = 0; i0 < RP * HALF; i0 += T) {
        const int e = i0 + tid;
        const int m = e / HALF, k = e % HALF;
        const int y0 = yb + 2 * m;
        const float2 s0 = Sb[(size_t)y0 * HALF + k];
        const float2 s1 = Sb[(size_t)(y0 + 1) * HALF + k];
        const int zb = m * SM;
        if (k == 0) {
            zs[PR::idx(zb)] = make_float2(s0.x, s1.x);
            zs[PR::idx(zb + HALF)] = make_float2(s0.y, s1.y);
        } else {
            zs[PR::idx(zb + k)] = make_float2(s0.x - s1.y, s0.y + s1.x);
            zs[PR::idx(zb + NX - k)] = make_float2(s0.x + s1.y, s1.x - s0.y);
        }
    }
    __syncthreads();
}

// The stages of a row inverse but the last, and the last.  Lengths with a
// factor 3 run the reversed stage plan, whose last stage is the radix-8 one:
// each thread then ends with one butterfly of 8 results instead of up to
// three of 3, which the update would spill.
template <class PF, int NX, int RP, int EPT, int MAXR>
__device__ __forceinline__ void inv_stages(float2* zs, const float2* tw, int tid)
{
    constexpr int LGRP = ct_lg<NX>(RP), SM = NX + kPad, NST = eprfft::ct_n_stages(NX, MAXR);
    if constexpr (NX % 3 == 0)
        eprfft::fft_ct_rev_stages<PF, +1, NX, EPT, LGRP, 1, SM, 0, NST - 1, MAXR>(zs, tw, tid);
    else
        eprfft::fft_ct_stages<PF, +1, NX, EPT, LGRP, 1, SM, 0, NST - 1, MAXR>(zs, tw, tid);
}
template <class PF, int NX, int RP, int EPT, int MAXR, class POST>
__device__ __forceinline__ void inv_last(float2* zs, const float2* tw, int tid, const POST& post)
{
    constexpr int LGRP = ct_lg<NX>(RP), SM = NX + kPad;
    if constexpr (NX % 3 == 0)
        eprfft::fft_ct_rev_last<PF, false, false, PF, +1, NX, EPT, LGRP, 1, SM, MAXR>(zs, tw, tid, post);
    else
        eprfft::fft_ct_last<PF, false, false, PF, +1, NX, EPT, LGRP, 1, SM, MAXR>(zs, tw, tid, post);
}

// The update of one result of the last inverse stage of a one-line block:
// element e = m SM + x holds rows 2m and 2m + 1 of the block at column x;
// T' = T - w ln(I'/I) from the staged thickness rows, stored, with the kappa
// partial sums kept in the functor (its call sites are inlined, so they stay
// in registers).
template <int NX, int SM, int RP, bool XT, bool STAGED = true>
struct InvUpdate1 {
    const EprConsts& C;
    const float* Tsh;      // [2 RP][NX] thickness rows of the block (STAGED), else unused
    float* out;            // T at the block's first row (read there when not STAGED)
    float mus, w, om_f, omega, eps;
    mutable float2 da, db;
    __device__ __forceinline__ float2 operator()(float2 h, int e) const
    {
        const int m = RP == 1 ? 0 : e / SM;
        const int x = e - m * SM;
        float* o = out + (size_t)(2 * m) * NX + x;
        const float2 t = STAGED ? make_float2(Tsh[(2 * m) * NX + x], Tsh[(2 * m + 1) * NX + x])
                                : make_float2(o[0], o[NX]);
        float wx = w, omx = om_f, mux = mus;
        if constexpr (XT) {
            wx = xt_get(C, EPR_XT_WPROJ, 0, x);
            mux = xt_get(C, EPR_XT_MU, 0, x);
            omx = omega / xt_get(C, EPR_XT_F, 0, x);
        }
        const float2 l = mul2(both(wx), log_ratio2(t, h, omx, mux, eps));
        const float2 n = sub2(t, l);
        o[0] = n.x;
        o[NX] = n.y;
        da = fma2(l, l, da);
        db = fma2(n, n, db);
        return h;
    }
};

// five 256-thread blocks per SM (48 registers): its shared memory is the FFT
// rows and 2 RP thickness rows only (row_inv_mono_smem).  EPT = 16 (8192-point
// rows): radix-16 stages, and the update reads T through L1 instead of staging
// it, so two 512-thread blocks fit on an SM.
template <int NX, int RP, bool OCC6 = false, bool XT = false, int EPT = kEPT>
__global__ void __launch_bounds__(NX * RP / EPT, OCC6 ? 6 : NX * RP / EPT == 256 ? 5
                                                 : row_min_blocks(NX * RP / EPT))
k_row_inv1(const EprConsts C, const RowArgs A)
{
    constexpr int T = NX * RP / EPT;
    constexpr int MAXR = row_maxr(EPT);
    constexpr bool kStageT = EPT <= kEPT;
    constexpr int SM = NX + kPad;
    constexpr int HALF = NX / 2;
    constexpr int LGRP = ct_lg<NX>(RP);
    extern __shared__ __align__(16) float2 zs[];
    __shared__ float red[64];
    const int b = row_batch_index();
    const int ny = C.ny, tid = threadIdx.x;
    const size_t pb = (size_t)b * NX * ny;
    const int yb = blockIdx.x * RP * 2;
    // rows yb .. yb + 2RP - 1 of T, copied while the spectrum is transformed
    float* Tsh = reinterpret_cast<float*>(zs + ((PR::len(RP * SM) + 1) & ~1));
    if constexpr (kStageT) {
        constexpr int Q4 = 2 * RP * NX / 4;
        const float4* src = reinterpret_cast<const float4*>(A.Out + pb + (size_t)yb * NX);
#pragma unroll
        for (int i0 = 0; i0 < Q4; i0 += T) {
            const int i = i0 + tid;
            if (Q4 % T == 0 || i < Q4) cp_async16(reinterpret_cast<float4*>(Tsh) + i, src + i);
        }
        cp_async_commit();
    }
    if constexpr (!kStageT) {   // read once per pixel after the transform
        constexpr int kRowLines = (NX + 31) / 32;
        for (int i = tid; i < 2 * RP * kRowLines; i += T)
            prefetch_l2(A.Out + pb + (size_t)(yb + i / kRowLines) * NX + 32 * (i % kRowLines));
    }
    epr_grid_wait();
    if (A.check_done && A.st[b].done) {
        cp_async_wait_all();
        return;
    }
    inv_unpack<NX, RP, EPT>(A.S + (size_t)b * (size_t)ny * HALF, zs, yb, tid);
    inv_stages<PR, NX, RP, EPT, MAXR>(zs, A.tw, tid);
    epr_grid_release();
    cp_async_wait_all();   // the thickness rows: visible to all after the last stage's barrier
    // the last stage hands each result to the update (no store, no barrier)
    const InvUpdate1<NX, SM, RP, XT, kStageT> up{C, Tsh, A.Out + pb + (size_t)yb * NX, C.mu[0],
                                                 C.wproj[0], A.omega / C.f[0], A.omega, A.eps,
                                                 {0.f, 0.f}, {0.f, 0.f}};
    inv_last<PR, NX, RP, EPT, MAXR>(zs, A.tw, tid, up);
    float da = up.da.x + up.da.y, db = up.db.x + up.db.y;
    block_sum2(da, db, red);   // kappa partials, finalised by the next forward pass
    store_partials(A.part_a + (size_t)b * A.max_blocks, A.part_b + (size_t)b * A.max_blocks, da, db);
}

// The per-line step of the polychromatic update, applied to each result of
// a line's last inverse stage (element e = m SM + x: rows 2m, 2m + 1 at
// column x): w_s ln(I'_s / I_s) added to the pixel's sum in shared memory
// (the element-to-thread map of the last stage is the same for every line,
// so each thread reads and writes its own pixels only); on the last line
// T' = T - sum is stored instead, with the kappa partial sums.
template <int NX, int SM, int RP, bool XT>
struct InvUpdatePoly {
    const EprConsts& C;
    const float* Tsh;      // [2 RP][NX] thickness rows of the block
    float* acc;            // [2 RP][NX] sums over the lines so far
    float* out;            // T at the block's first row
    int s;                 // line of this pass
    bool first, last;
    float mus, w, om_f, omega, eps;
    mutable float2 da, db;
    __device__ __forceinline__ float2 operator()(float2 h, int e) const
    {
        const int m = RP == 1 ? 0 : e / SM;
        const int x = e - m * SM;
        const int i0 = (2 * m) * NX + x;
        float wx = w, omx = om_f, mux = mus;
        if constexpr (XT) {
            wx = xt_get(C, EPR_XT_WPROJ, s, x);
            mux = xt_get(C, EPR_XT_MU, s, x);
            omx = omega / xt_get(C, EPR_XT_F, s, x);
        }
        const float2 t = make_float2(Tsh[i0], Tsh[i0 + NX]);
        float2 l = mul2(both(wx), log_ratio2(t, h, omx, mux, eps));
        if (!first) l = add2(make_float2(acc[i0], acc[i0 + NX]), l);
        if (last) {
            const float2 n = sub2(t, l);
            float* o = out + (size_t)(2 * m) * NX + x;
            o[0] = n.x;
            o[NX] = n.y;
            da = fma2(l, l, da);
            db = fma2(n, n, db);
        } else {
            acc[i0] = l.x;
            acc[i0 + NX] = l.y;
        }
        return h;
    }
};

// Polychromatic update on the compile-time engine: for each line, the C2R
// rows of its filtered spectrum and w_s ln(I'_s / I_s), accumulated per
// pixel in shared memory (each thread owns its pixels); then T' = T - sum
// and the kappa partial sums.
template <int NX, int RP, bool XT = false, int EPT = kEPT>
__global__ void __launch_bounds__(NX * RP / EPT, row_min_blocks(NX * RP / EPT, NX % 3 == 0 && RP > 1 ? 768 : 1024))
k_row_invn(const EprConsts C, const RowArgs A)
{
    constexpr int T = NX * RP / EPT;
    constexpr int SM = NX + kPad;
    constexpr int HALF = NX / 2;
    constexpr int LGRP = ct_lg<NX>(RP);
    extern __shared__ __align__(16) float2 zs[];
    __shared__ float red[64];
    const int b = row_batch_index();
    const int ny = C.ny, tid = threadIdx.x;
    const size_t pb = (size_t)b * NX * ny;
    const int yb = blockIdx.x * RP * 2;
    float* Tsh = reinterpret_cast<float*>(zs + ((PR::len(RP * SM) + 1) & ~1));   // [2 RP][NX]
    float* acc = Tsh + 2 * RP * NX;                                              // [2 RP][NX]
    {
        constexpr int Q4 = 2 * RP * NX / 4;
        const float4* src = reinterpret_cast<const float4*>(A.Out + pb + (size_t)yb * NX);
#pragma unroll
        for (int i0 = 0; i0 < Q4; i0 += T) {
            const int i = i0 + tid;
            if (Q4 % T == 0 || i < Q4) cp_async16(reinterpret_cast<float4*>(Tsh) + i, src + i);
        }
        cp_async_commit();
    }
    epr_grid_wait();
    if (A.check_done && A.st[b].done) {
        cp_async_wait_all();
        return;
    }
    InvUpdatePoly<NX, SM, RP, XT> up{C, Tsh, acc, A.Out + pb + (size_t)yb * NX, 0, true, false,
                                     0.f, 0.f, 0.f, A.omega, A.eps, {0.f, 0.f}, {0.f, 0.f}};
    for (int sl = 0; sl < A.nl; ++sl) {
        const int s = A.line0 + sl;
        inv_unpack<NX, RP, EPT>(A.S + ((size_t)b * A.nl + sl) * (size_t)ny * HALF, zs, yb, tid);
        inv_stages<PR, NX, RP, EPT, row_maxr(EPT)>(zs, A.tw, tid);
        if (sl == 0) {
            epr_grid_release();
            cp_async_wait_all();   // the thickness rows: visible after the last stage's barrier
        }
        // the last stage adds the line's term to each thread's own pixels;
        // after its barrier nothing reads zs, so the next unpack may follow
        up.s = s;
        up.first = sl == 0;
        up.last = sl == A.nl - 1;
        up.mus = line_const(C.mu, s);
        up.w = line_const(C.wproj, s);
        up.om_f = A.omega / line_const(C.f, s);
        inv_last<PR, NX, RP, EPT, row_maxr(EPT)>(zs, A.tw, tid, up);
    }
    float da = up.da.x + up.da.y, db = up.db.x + up.db.y;
    block_sum2(da, db, red);   // kappa partials, finalised by the next forward pass
    store_partials(A.part_a + (size_t)b * A.max_blocks, A.part_b + (size_t)b * A.max_blocks, da, db);
}

// The last inverse stage of a plain inverse transform: element e = m SM + x
// holds rows 2m and 2m + 1 of the block at column x.
template <int NX, int SM, int RP>
struct InvStore {
    float* out;            // the map at the block's first row
    __device__ __forceinline__ float2 operator()(float2 h, int e) const
    {
        const int m = RP == 1 ? 0 : e / SM;
        float* o = out + (size_t)(2 * m) * NX + (e - m * SM);
        o[0] = h.x;
        o[NX] = h.y;
        return h;
    }
};

// C2R rows to a real map.
template <int NX, int RP, int EPT = kEPT>
__global__ void __launch_bounds__(NX * RP / EPT, row_min_blocks(NX * RP / EPT))
k_row_store(const EprConsts C, const RowArgs A)
{
    constexpr int SM = NX + kPad;
    extern __shared__ __align__(16) float2 zs[];
    const int b = row_batch_index();
    const int ny = C.ny, tid = threadIdx.x;
    const int yb = blockIdx.x * RP * 2;
    epr_grid_wait();
    inv_unpack<NX, RP, EPT>(A.S + (size_t)b * (size_t)ny * (NX / 2), zs, yb, tid);
    inv_stages<PP, NX, RP, EPT, row_maxr(EPT)>(zs, A.tw, tid);
    epr_grid_release();
    const InvStore<NX, SM, RP> st{A.Out + (size_t)b * NX * ny + (size_t)yb * NX};
    inv_last<PP, NX, RP, EPT, row_maxr(EPT)>(zs, A.tw, tid, st);
}

// dynamic shared memory: the FFT rows; the forward gather aliases them with
// the 2 RP + 2 staged thickness rows, the updates add the block's thickness
// rows and, for several lines, the accumulators
constexpr size_t row_fft_smem(int nx, int rp)
{
    return (size_t)((((rp * (nx + kPad) + 15) & ~15) + 1) & ~1) * sizeof(float2);
}
constexpr size_t row_fwd_smem(int nx, int rp)
{
    const size_t fft = row_fft_smem(nx, rp), ts = (size_t)(2 * rp + 2) * nx * sizeof(float);
    return fft > ts ? fft : ts;
}
constexpr size_t row_inv_smem(int nx, int rp, int maps)
{
    return row_fft_smem(nx, rp) + (size_t)maps * (2 * rp * nx) * sizeof(float);
}

// Table entries.  ANY: the several-line kernels serve one line as well (row
// lengths with a factor 9, small blocks); FULL: the one-line kernels too.
template <int NX, int RP, int EPT = kEPT>
constexpr RowKernels row_any()
{
    RowKernels k = {};
    k.nx = NX;
    k.rp = RP;
    k.threads = NX * RP / EPT;
    k.fwdn = k_row_fwd_ct<NX, RP, true, true, false, false, EPT>;
    k.invn = k_row_invn<NX, RP, false, EPT>;
    // the plain transforms hold nothing but the row: 16 elements per thread
    // and radix-16 stages (2304 = 16 16 9 instead of 8 8 4 9) where that
    // leaves a block of at least three warps
    constexpr int EPTP = EPT == kEPT && RP == 1 && NX >= 1536 && NX % 16 == 0 ? 16 : EPT;
    k.threads_plain = NX * RP / EPTP;
    k.plain = k_row_fwd_ct<NX, RP, true, false, false, false, EPTP>;
    k.store = k_row_store<NX, RP, EPTP>;
    k.smem_fwd = row_fwd_smem(NX, RP);
    k.smem_plain = row_fft_smem(NX, RP);
    k.smem_inv1 = k.smem_invn1 = row_inv_smem(NX, RP, 1);
    k.smem_invn = row_inv_smem(NX, RP, 2);
    return k;
}
template <int NX, int RP>
constexpr RowKernels row_full()
{
    RowKernels k = row_any<NX, RP>();
    k.fwd1 = k_row_fwd_ct<NX, RP, false, true>;
    k.inv1 = k_row_inv1<NX, RP>;
    return k;
}
template <int NX, int RP>
constexpr RowKernels row_full_xt()
{
    RowKernels k = row_full<NX, RP>();
    k.xfwd1 = k_row_fwd_ct<NX, RP, false, true, false, true>;
    k.xfwdn = k_row_fwd_ct<NX, RP, true, true, false, true>;
    k.xinv1 = k_row_inv1<NX, RP, false, true>;
    k.xinvn = k_row_invn<NX, RP, true>;
    return k;
}

}  // namespace
#endif  // EPR_ROW_KERNELS
