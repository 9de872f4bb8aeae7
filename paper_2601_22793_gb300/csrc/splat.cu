// Forward non-local transport around the tile kernel (splat_tile.cuh, which
// describes it): the long-shift sources, the residual split, the oversampled
// forms, and the host launchers.
#include "splat_tile.cuh"

namespace {

using namespace eprsplat;

// What the long-shift pass adds a contribution to.
//   FAR_MODEL  P and P_s (a forward), float
//   FAR_RESID  the residual D - P of one line (negative), float
//   FAR_SPLIT  the split residuals r_s of several lines, float (see far_scale)
//   FAR_FX     the fixed-point sums
enum { FAR_MODEL = 0, FAR_RESID = 1, FAR_SPLIT = 2, FAR_FX = 3 };

// Every corner pixel o on the grid, line s and contribution v of a list entry.
template <bool XT, class F>
__device__ __forceinline__ void far_corners(const EprConsts& C, int pix, unsigned int mask, float4 tg, F f)
{
    const int nx = C.nx, ny = C.ny;
    const int sy = pix / nx, sx = pix - sy * nx;
    const float t = tg.x;
    for (int s = 0; s < C.ns; ++s) {
        if (!((mask >> s) & 1u)) continue;
        const float ch = 0.5f * (XT ? xt_get(C, EPR_XT_C, s, sx) : C.c[s]);
        const float ux = ch * tg.y, uy = ch * tg.z;
        const float fx = floorf(ux), fy = floorf(uy);
        const float dx = ux - fx, dy = uy - fy;
        const float fs = XT ? xt_get(C, EPR_XT_F, s, sx) : C.f[s];
        const float mus = XT ? xt_get(C, EPR_XT_MU, s, sx) : C.mu[s];
        const float m = fs * __expf(-mus * t);
        const float w[4] = {(1.f - dx) * (1.f - dy), dx * (1.f - dy), (1.f - dx) * dy, dx * dy};
        // corner coordinates in float first: a huge shift must not wrap an int
        const float cxf = (float)sx + fx, cyf = (float)sy + fy;
        for (int k = 0; k < 4; ++k) {
            const float xf = cxf + (float)(k & 1), yf = cyf + (float)(k >> 1);
            if (!(xf >= 0.f && xf < (float)nx && yf >= 0.f && yf < (float)ny)) continue;
            f((size_t)(int)yf * nx + (int)xf, s, m * w[k]);
        }
    }
}

// The scale in which a pixel's split residuals hold its line predictions.
// The splat flush of a several-line float solve stores P (of the near sources),
// r = D - P and r_s = k P_s with k = r / P (never 0), and a long-shift
// contribution to P_s is added k times as large.  Where no near source reaches
// the pixel (P = 0) r_s is r f_s; a contribution is then added 2^64 |r| times,
// beside which r f_s is rounding error.  P is a map of its own because D - r
// has lost its digits where D is much larger than P: the relative error of r_s
// was 3e-4 at D = 1e4 P and of order 1 at D = 2e7 P.
constexpr float kDarkScale = 18446744073709551616.f;
__device__ __forceinline__ float far_scale(float r, float p)
{
    if (p > 1e-30f) return split_ratio(r, p);
    return r != 0.f ? kDarkScale * fabsf(r) : 1.f;
}

// The long-shift sources of the overflow list, added with global atomics.
// FAR_SPLIT marks every pixel it touches in `claim` for k_overflow_fix.
template <int TO, bool XT = false>
__global__ void __launch_bounds__(128) k_splat_overflow(const __grid_constant__ EprConsts C, const SplatArgs A)
{
    const int b = blockIdx.y;
    epr_grid_wait();
    if (A.check_done && A.st[b].done) return;
    epr_grid_release();
    const int ns = C.ns;
    const size_t npix = (size_t)C.nx * C.ny, pb = (size_t)b * npix;
    const int cnt_raw = A.st[b].ovf_count[A.parity];
    const int cnt = cnt_raw < C.ovf_cap ? cnt_raw : C.ovf_cap;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        A.st[b].ovf_count[A.parity ^ 1] = 0;   // the next splat's slot
        if (cnt > 0) A.st[b].ovf_total += cnt;
    }
    // entries come with T and twice the gradient; the first round's entry is
    // loaded together with the count (every slot below the capacity exists)
    const int stride = gridDim.x * blockDim.x;
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    int pix = 0;
    unsigned int mask = 0u;
    float4 tg = make_float4(0.f, 0.f, 0.f, 0.f);
    if (e < C.ovf_cap) {
        pix = A.ovf_idx[(size_t)b * C.ovf_cap + e];
        mask = A.ovf_mask[(size_t)b * C.ovf_cap + e];
        tg = A.ovf_tg[(size_t)b * C.ovf_cap + e];
    }
    for (; e < cnt; e += stride) {
        if (e >= stride) {   // later rounds
            pix = A.ovf_idx[(size_t)b * C.ovf_cap + e];
            mask = A.ovf_mask[(size_t)b * C.ovf_cap + e];
            tg = A.ovf_tg[(size_t)b * C.ovf_cap + e];
        }
        far_corners<XT>(C, pix, mask, tg, [&](size_t o, int s, float v) {
            const size_t po = pb + o, ps = pb * ns + (size_t)s * npix + o;
            if constexpr (TO == FAR_FX) {
                const unsigned long long q = (unsigned long long)__float2ll_rn(v * EPR_FX_SCALE);
                atomicAdd(&A.Pq[po], q);
                if (ns > 1) atomicAdd(&A.Psq[ps], q);
            } else if constexpr (TO == FAR_RESID) {
                atomicAdd(&A.P[po], -v);
            } else if constexpr (TO == FAR_SPLIT) {
                const float p = __ldg(&A.Pnear[po]);
                atomicAdd(&A.Ps[ps], v * far_scale(__ldg(&A.D[po]) - p, p));
                atomicAdd(&A.P[po], -v);
                atomicOr(&A.claim[po >> 5], 1u << (po & 31));
            } else {
                atomicAdd(&A.P[po], v);
                if (ns > 1 && A.Ps) atomicAdd(&A.Ps[ps], v);
            }
        });
    }
}

// The split at the pixels that long-shift sources reached, once they are all
// in: r_s = r P_s / P (r f_s where P vanishes).  Fixed point forms it and r
// anew from the sums (every visitor of a pixel writes the same values).  Float
// has r, and the lines' predictions in a common scale (far_scale): their shares
// are the ratios to their sum.  The one visitor that takes the pixel's claim
// bit writes them.  A few thousand pixels instead of a pass over every map: the
// separate split of eight lines of a 2048^2 map took 46 us.
template <bool DET, bool XT = false>
__global__ void __launch_bounds__(128) k_overflow_fix(const __grid_constant__ EprConsts C, const SplatArgs A)
{
    const int b = blockIdx.y;
    const int ns = C.ns, nx = C.nx;
    const size_t npix = (size_t)nx * C.ny, pb = (size_t)b * npix;
    // the list is the splat's, complete before the long-shift pass began
    const int cnt_raw = A.st[b].ovf_count[A.parity];
    const int cnt = cnt_raw < C.ovf_cap ? cnt_raw : C.ovf_cap;
    epr_grid_wait();
    if (A.check_done && A.st[b].done) return;
    epr_grid_release();
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < cnt; e += gridDim.x * blockDim.x) {
        const size_t at = (size_t)b * C.ovf_cap + e;
        far_corners<XT>(C, A.ovf_idx[at], A.ovf_mask[at], A.ovf_tg[at], [&](size_t o, int, float) {
            const size_t po = pb + o, ps = pb * ns + o;
            const int x = XT ? (int)(o % (size_t)nx) : 0;
            auto weight = [&](int l) { return XT ? xt_get(C, EPR_XT_F, l, x) : C.f[l]; };
            const float d = __ldg(&A.D[po]);
            if constexpr (DET) {
                const float p = (float)A.Pq[po] * EPR_FX_INV;
                const float r = d - p, k = p > 1e-30f ? split_ratio(r, p) : r;
                for (int l = 0; ns > 1 && l < ns; ++l)
                    A.Ps[ps + l * npix] = k * (p > 1e-30f ? (float)A.Psq[ps + l * npix] * EPR_FX_INV : weight(l));
                A.P[po] = r;
            } else {
                const unsigned int bit = 1u << (po & 31);
                if (!(atomicAnd(&A.claim[po >> 5], ~bit) & bit)) return;   // another visitor's
                const float pn = __ldg(&A.Pnear[po]), r = A.P[po];
                const bool lit = pn > 1e-30f;
                auto line = [&](int l) {   // the scaled P_s with the long-shift contributions
                    const float v = A.Ps[ps + l * npix];
                    return lit ? v : fmaxf(__fsub_rn(v, __fmul_rn(d, weight(l))), 0.f);
                };
                double sum = 0.0;
                for (int l = 0; l < ns; ++l) sum += (double)line(l);
                const float all = (float)sum;
                const bool any = lit || all > 1e-30f * far_scale(d, 0.f);
                for (int l = 0; l < ns; ++l) A.Ps[ps + l * npix] = r * (any ? line(l) / all : weight(l));
            }
        });
    }
}

// Oversampled grid (os > 1): the detector image of the model is the mean of
// each os x os block of the fine P; the residual D - mean is formed per
// detector pixel and replicated to the fine pixels of its block, where it is
// split over the lines with the fine weights P_s / P.  One thread per
// detector pixel; P <- replicated residual, P_s <- split residuals.
//
// OS is the factor at compile time for 2, 3 and 4 (0: any): the block's
// values are then loaded together, as pairs or quads where they are aligned,
// kept for the split, and written once.
template <int OS>
__device__ __forceinline__ void os_load(const float* p, float (&v)[OS])
{
    if constexpr (OS == 2) {
        const float2 a = *reinterpret_cast<const float2*>(p);
        v[0] = a.x;
        v[1] = a.y;
    } else if constexpr (OS == 4) {
        const float4 a = *reinterpret_cast<const float4*>(p);
        v[0] = a.x;
        v[1] = a.y;
        v[2] = a.z;
        v[3] = a.w;
    } else {
#pragma unroll
        for (int i = 0; i < OS; ++i) v[i] = p[i];
    }
}
template <int OS>
__device__ __forceinline__ void os_store(float* p, const float (&v)[OS])
{
    if constexpr (OS == 2) {
        *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
    } else if constexpr (OS == 4) {
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
        for (int i = 0; i < OS; ++i) p[i] = v[i];
    }
}

template <bool DET, int OS>
__global__ void __launch_bounds__(256) k_split_os(const EprConsts C, const SplatArgs A)
{
    const int b = blockIdx.y;
    epr_grid_wait();
    if (A.check_done && A.st[b].done) return;
    epr_grid_release();
    const int ns = C.ns, os = OS ? OS : C.os, nx = C.nx;
    const int nxd = C.nx / os, nyd = C.ny / os;
    const size_t npix = (size_t)C.nx * C.ny, pb = (size_t)b * npix;
    const size_t npd = (size_t)nxd * nyd;
    const float inv_o2 = 1.f / (float)(os * os);
    for (size_t qd = (size_t)blockIdx.x * blockDim.x + threadIdx.x; qd < npd;
         qd += (size_t)gridDim.x * blockDim.x) {
        const int yd = (int)(qd / nxd), xd = (int)(qd - (size_t)yd * nxd);
        const size_t f0 = pb + (size_t)yd * os * nx + (size_t)xd * os;   // block corner
        const float d = __ldg(&A.D[(size_t)b * npd + qd]);
        if constexpr (OS > 0 && !DET) {
            float p[OS][OS];
#pragma unroll
            for (int a = 0; a < OS; ++a) os_load<OS>(A.P + f0 + (size_t)a * nx, p[a]);
            float sum = 0.f;
#pragma unroll
            for (int a = 0; a < OS; ++a)
#pragma unroll
                for (int c = 0; c < OS; ++c) sum += p[a][c];
            const float r = d - sum * inv_o2;
            for (int s = 0; ns > 1 && s < ns; ++s) {
                const float fs = line_const(C.f, s);
                float* ps = A.Ps + pb * ns + (size_t)s * npix + (f0 - pb);
                float v[OS][OS];
#pragma unroll
                for (int a = 0; a < OS; ++a) os_load<OS>(ps + (size_t)a * nx, v[a]);
#pragma unroll
                for (int a = 0; a < OS; ++a) {
#pragma unroll
                    for (int c = 0; c < OS; ++c)
                        v[a][c] = p[a][c] > 1e-30f ? r * (v[a][c] / p[a][c]) : r * fs;
                    os_store<OS>(ps + (size_t)a * nx, v[a]);
                }
            }
            float o[OS];
#pragma unroll
            for (int c = 0; c < OS; ++c) o[c] = r;
#pragma unroll
            for (int a = 0; a < OS; ++a) os_store<OS>(A.P + f0 + (size_t)a * nx, o);
            continue;
        }
        float mean;
        if constexpr (DET) {
            unsigned long long q = 0ull;
            for (int a = 0; a < os; ++a)
                for (int c = 0; c < os; ++c) q += A.Pq[f0 + (size_t)a * nx + c];
            mean = (float)q * EPR_FX_INV * inv_o2;
        } else {
            float sum = 0.f;
            for (int a = 0; a < os; ++a)
                for (int c = 0; c < os; ++c) sum += A.P[f0 + (size_t)a * nx + c];
            mean = sum * inv_o2;
        }
        const float r = d - mean;
        for (int a = 0; a < os; ++a)
            for (int c = 0; c < os; ++c) {
                const size_t i = f0 + (size_t)a * nx + c;
                if (ns > 1) {
                    const float p = DET ? (float)A.Pq[i] * EPR_FX_INV : A.P[i];
                    for (int s = 0; s < ns; ++s) {
                        const size_t o = pb * ns + (size_t)s * npix + (i - pb);
                        const float pl = DET ? (float)A.Psq[o] * EPR_FX_INV : A.Ps[o];
                        A.Ps[o] = (p > 1e-30f) ? r * (pl / p) : r * line_const(C.f, s);
                    }
                }
                A.P[i] = r;
            }
    }
}

// Detector image of the forward model on an oversampled grid: the mean of
// each os x os block of P (out) and of each P_s (outs, may be NULL).
template <bool DET>
__global__ void __launch_bounds__(256) k_bin_os(const EprConsts C, const SplatArgs A, float* out,
                                                float* outs)
{
    const int b = blockIdx.y;
    const int ns = C.ns, os = C.os, nx = C.nx;
    const int nxd = C.nx / os, nyd = C.ny / os;
    const size_t npix = (size_t)C.nx * C.ny, pb = (size_t)b * npix;
    const size_t npd = (size_t)nxd * nyd;
    const float inv_o2 = 1.f / (float)(os * os);
    for (size_t qd = (size_t)blockIdx.x * blockDim.x + threadIdx.x; qd < npd;
         qd += (size_t)gridDim.x * blockDim.x) {
        const int yd = (int)(qd / nxd), xd = (int)(qd - (size_t)yd * nxd);
        const size_t f0 = (size_t)yd * os * nx + (size_t)xd * os;
        for (int s = -1; s < (outs ? ns : 0); ++s) {   // s = -1: P
            const bool tot = s < 0;
            const size_t base = tot ? pb : (pb * ns + (size_t)s * npix);
            if (!tot && ns == 1) {   // one line: P_s is P
                outs[(size_t)b * npd + qd] = out[(size_t)b * npd + qd];
                continue;
            }
            float m;
            if constexpr (DET) {
                const unsigned long long* q = tot ? A.Pq : A.Psq;
                unsigned long long sum = 0ull;
                for (int a = 0; a < os; ++a)
                    for (int c = 0; c < os; ++c) sum += q[base + f0 + (size_t)a * nx + c];
                m = (float)sum * EPR_FX_INV * inv_o2;
            } else {
                const float* q = tot ? A.P : A.Ps;
                float sum = 0.f;
                for (int a = 0; a < os; ++a)
                    for (int c = 0; c < os; ++c) sum += q[base + f0 + (size_t)a * nx + c];
                m = sum * inv_o2;
            }
            if (tot) out[(size_t)b * npd + qd] = m;
            else outs[((size_t)b * ns + s) * npd + qd] = m;
        }
    }
}

}  // namespace

// Whether the six-blocks-per-SM residual splat exists for this tile and reach.
bool epr_splat_has_occ6(int TH, int TW, int reach) { return TH * TW < 64 * 64 && (reach == 3 || reach == 4); }

size_t epr_splat_smem(const EprConsts& C, int TH, int TW)
{
    const int R = C.smax;
    const int HX = (R + 1 + 3) & ~3;
    const int SH = (TH + 2 * R + kQuad - 1) / kQuad * kQuad + 2;
    const size_t acc_bytes = (size_t)C.ns * (TH + 2) * (TW + 2 * kAccX) * (C.det ? 8 : 4);
    return ((acc_bytes + 15) & ~size_t(15)) + (size_t)SH * (TW + 2 * HX) * sizeof(float);
}

// Host launcher: the tile kernel, then the long-shift pass.  With D (a solve
// on the detector grid) P receives D - P, P_s the split residuals, and where
// the split needs the whole prediction of a pixel (several lines, fixed
// point) a third launch redoes the pixels that long shifts reached.  `parity`
// alternates the overflow counter slot between consecutive splats of a solve.
cudaError_t epr_launch_splat(const EprConsts& C, const EprWork& W, const float* T, const float* D,
                             int parity, int batch, int TH, int TW, int check_done, cudaStream_t stream)
{
    SplatArgs A;
    A.T = T;
    A.D = D;
    A.P = W.P;
    A.Ps = W.Ps;
    A.Pq = W.Pq;
    A.Psq = W.Psq;
    A.ovf_idx = W.ovf_idx;
    A.ovf_mask = W.ovf_mask;
    A.ovf_tg = W.ovf_tg;
    A.st = W.st;
    A.err = W.err;
    A.Pnear = W.Pnear;
    A.claim = W.claim;
    A.parity = parity & 1;
    A.check_done = check_done;
    {   // 2^(32 - S) >= 2 (2 reach + 3)^2: the largest pixel sum fits in uint32
        const int win = 2 * (2 * C.smax + 3) * (2 * C.smax + 3);
        int bits = 0;
        while ((1 << bits) < win) ++bits;
        A.fxs = ldexpf(1.f, 32 - bits);
        A.fxs_inv = ldexpf(1.f, bits - 32);
        // fixed point: W 2^L and W 2^(41 - L) < 2^32 with W < 2^(bits - 1)
        A.fx_lo = bits - 1 <= 11 ? 32 - (bits - 1) : 0;
        A.fx_lo_s = ldexpf(1.f, A.fx_lo);
        A.fx_lo_inv = ldexpf(1.f, -A.fx_lo);
        A.ch_max = 0.f;
        A.tneg_max = C.tneg[0];
        for (int i = 0; i < C.ns; ++i) {
            A.ch_max = fmaxf(A.ch_max, 0.5f * fabsf(C.c[i]));
            A.tneg_max = fmaxf(A.tneg_max, C.tneg[i]);
        }
    }
    const size_t smem = epr_splat_smem(C, TH, TW);
    dim3 grid((C.nx + TW - 1) / TW, (C.ny + TH - 1) / TH, batch);
    const bool occ6 = W.splat_occ6 != 0;
    // one float line: P receives D - P and there is nothing to split, whichever
    // kernel the tile ran (an x-dependent spectrum has the several-line one)
    const bool mono = D && C.ns == 1 && !C.det;
    const int resid = mono && !C.xt;   // its own kernels
    if (D && !mono && !C.det && (!W.Ps || !W.Pnear || !W.claim)) return cudaErrorInvalidValue;
    cudaError_t e;
    if (TH == 64 && TW == 64) e = epr_splat_launch_64x64(C, A, resid, occ6, grid, smem, stream);
    else if (TH == 32 && TW == 64) e = epr_splat_launch_32x64(C, A, resid, occ6, grid, smem, stream);
    else if (TH == 64 && TW == 32) e = epr_splat_launch_64x32(C, A, resid, occ6, grid, smem, stream);
    else if (TH == 32 && TW == 32) e = epr_splat_launch_32x32(C, A, resid, occ6, grid, smem, stream);
    else return cudaErrorInvalidValue;
    if (e != cudaSuccess) return e;
    auto go = [&](auto kernel) {
        if (e != cudaSuccess) return;
        e = epr_launch_kernel(C.pdl != 0, kernel, dim3(128, batch), dim3(128), 0, stream, C, A);
        epr_count_launch(1);
    };
    epr_count_launch(1);
    if (C.det) {
        if (C.xt) go(k_splat_overflow<FAR_FX, true>);
        else go(k_splat_overflow<FAR_FX>);
        if (D && C.xt) go(k_overflow_fix<true, true>);
        else if (D) go(k_overflow_fix<true>);
    } else if (mono) {
        if (C.xt) go(k_splat_overflow<FAR_RESID, true>);
        else go(k_splat_overflow<FAR_RESID>);
    } else if (D) {
        if (C.xt) {
            go(k_splat_overflow<FAR_SPLIT, true>);
            go(k_overflow_fix<false, true>);
        } else {
            go(k_splat_overflow<FAR_SPLIT>);
            go(k_overflow_fix<false>);
        }
    } else if (C.xt) {
        go(k_splat_overflow<FAR_MODEL, true>);
    } else {
        go(k_splat_overflow<FAR_MODEL>);
    }
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t epr_splat_init()
{
    cudaError_t e = epr_splat_init_64x64();
    if (e == cudaSuccess) e = epr_splat_init_32x64();
    if (e == cudaSuccess) e = epr_splat_init_64x32();
    if (e == cudaSuccess) e = epr_splat_init_32x32();
    return e;
}

// Oversampled solve: the split at detector resolution (k_split_os).
cudaError_t epr_launch_split_os(const EprConsts& C, const EprWork& W, const float* D, int batch,
                                int fixed_point, int check_done, cudaStream_t stream)
{
    SplatArgs A = {};
    A.D = D;
    A.P = W.P;
    A.Ps = W.Ps;
    A.Pq = W.Pq;
    A.Psq = W.Psq;
    A.st = W.st;
    A.check_done = check_done;
    const size_t npd = (size_t)(C.nx / C.os) * (C.ny / C.os);
    size_t blocks = (npd + 255) / 256;
    if (blocks > 1216) blocks = 1216;
    const dim3 grid((unsigned)blocks, batch), blk(256);
    const bool pdl = C.pdl != 0;
    cudaError_t e;
    if (fixed_point) e = epr_launch_kernel(pdl, k_split_os<true, 0>, grid, blk, 0, stream, C, A);
    else if (C.os == 2) e = epr_launch_kernel(pdl, k_split_os<false, 2>, grid, blk, 0, stream, C, A);
    else if (C.os == 3) e = epr_launch_kernel(pdl, k_split_os<false, 3>, grid, blk, 0, stream, C, A);
    else if (C.os == 4) e = epr_launch_kernel(pdl, k_split_os<false, 4>, grid, blk, 0, stream, C, A);
    else e = epr_launch_kernel(pdl, k_split_os<false, 0>, grid, blk, 0, stream, C, A);
    epr_count_launch(1);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// Oversampled forward: detector images of P and of each P_s (outs may be NULL).
cudaError_t epr_launch_bin_os(const EprConsts& C, const EprWork& W, int fixed_point, float* out,
                              float* outs, int batch, cudaStream_t stream)
{
    SplatArgs A = {};
    A.P = W.P;
    A.Ps = W.Ps;
    A.Pq = W.Pq;
    A.Psq = W.Psq;
    const size_t npd = (size_t)(C.nx / C.os) * (C.ny / C.os);
    size_t blocks = (npd + 255) / 256;
    if (blocks > 1216) blocks = 1216;
    const dim3 grid((unsigned)blocks, batch), blk(256);
    if (fixed_point) k_bin_os<true><<<grid, blk, 0, stream>>>(C, A, out, outs);
    else k_bin_os<false><<<grid, blk, 0, stream>>>(C, A, out, outs);
    epr_count_launch(1);
    return cudaGetLastError();
}
