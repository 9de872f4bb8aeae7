// Forward non-local transport: the conservative bilinear redistribution of
// the object intensity of every spectral line onto the detector grid
// (arXiv 2601.22793, Eq. 3 and "Discrete implementation: conservative
// bilinear redistribution"), with the polychromatic sum of Eq. 5.
//
// Design (destination-tile binning):
//  * A block owns one TH x TW destination tile of one projection and holds
//    its accumulators (one per line) in shared memory.
//  * It scans every source pixel whose shifted corners can land in the tile:
//    the tile grown by the reach on each side (a shift of exactly +reach
//    gives its far corner weight 0, so no further pixel contributes).  The
//    thickness of that region plus a one-pixel ring (for the gradient) is
//    staged in shared memory with asynchronous copies; beyond the grid the
//    edge value is replicated, which makes the central difference half the
//    one-sided one.  Blocks whose staged region lies inside the grid take a
//    path without edge tests.
//  * Per source and line it forms the shift u = c_s G[T] (central
//    differences, one-sided at the grid edges), splits u into floor and
//    fraction, and adds f_s exp(-mu_s T) times the four bilinear weights to
//    the corners inside the tile with shared-memory atomics.  exp is
//    evaluated only when the source reaches the tile.  A thread takes four
//    vertically adjacent sources as two packed pairs; only a quad that holds
//    a long shift tests every source and line.
//  * The shared accumulators are integers, because integer shared-memory
//    atomics are single instructions while float ones are not.  The float
//    mode adds round(v * 2^S) in uint32 with S chosen from the reach so that
//    no pixel can overflow: at most (2 reach + 3)^2 sources reach a pixel,
//    each with a contribution <= f_s <= 1, so 2^(32-S) >= (2 reach + 3)^2.
//    With a factor 2 of headroom, 2^(32-S) >= 2 (2 reach + 3)^2 holds for
//    contributions up to 2 f_s, and a source whose intensity exceeds that
//    (T < -ln 2 / mu_s, a negative thickness far outside any physical
//    iterate) takes the overflow path with the long shifts.  For reach 4,
//    S = 24: a rounding error of at most 3e-8 per contribution, half an fp32
//    ulp of a unit intensity.
//  * Every destination pixel is written exactly once, with plain coalesced
//    stores: no zero fill and no global atomics on the fast path.  In a solve
//    on the detector grid the flush stores the residual D - P instead of P
//    and, for several lines, its split r_s = r P_s / P instead of P_s (the
//    adjoint gather then reads one value per corner), so no pass over the maps
//    is left between the splat and the gather; the pixels that long-shift
//    sources reach afterwards are redone one by one (splat.cu).
//  * A source-line with |u| > reach in either axis (or T below the bound
//    above) is never splatted by the scan; the block that owns the source
//    pixel appends it (with a bit mask of its long lines, its thickness and
//    twice its gradient) to a per-projection overflow list, and a second
//    kernel adds those contributions with global atomics.  No mass is lost,
//    whatever the shift.  The list fill counter alternates between two slots
//    by iteration parity, so the overflow kernel can clear the next slot.
//  * Fixed-point mode accumulates round(v * 2^40) (contributions are
//    non-negative), as uint64 in global memory: integer addition is
//    associative, so the result is bit-identical across runs.  In shared
//    memory the sums are kept as two uint32 planes, q = hi 2^L + lo, because
//    64-bit shared-memory atomics are compare-and-swap loops: with at most
//    W = (2 reach + 3)^2 sources per pixel of at most 2^41 each, W 2^L and
//    W 2^(41 - L) both fit in 32 bits for L = 32 - ceil(log2 W) and
//    W <= 2^11 (reach <= 21); a longer reach keeps the uint64 sums.
#pragma once

#include <type_traits>

#include "epr_internal.cuh"

namespace eprsplat {

struct SplatArgs {
    const float* T;          // [B][ny][nx]
    const float* D;          // [B][ny][nx] (residual output)
    float* P;                // [B][ny][nx]   P, or D - P (residual output)
    float* Ps;               // [B][ns][ny][nx] P_s, or r_s (residual output), or NULL:
                             //    not wanted (float mode, ns > 1)
    unsigned long long* Pq;  // fixed-point mode
    unsigned long long* Psq;
    int* ovf_idx;
    unsigned int* ovf_mask;
    float4* ovf_tg;          // (T, twice the gradient x, y, 0) of each entry
    EprProjState* st;
    unsigned int* err;
    float* Pnear;            // [B][ny][nx] P without the long shifts (residual output of
                             //    several float lines)
    unsigned int* claim;     // [B ny nx / 32] bits, all 0 between solves (float mode, ns > 1)
    int parity;
    int check_done;
    float fxs, fxs_inv;      // float mode: scale 2^S of the uint32 accumulators
    int fx_lo;               // fixed-point mode: bits L of the low plane, 0 = uint64 sums
    float fx_lo_s, fx_lo_inv;   // 2^L, 2^-L
    float ch_max, tneg_max;  // largest |c_s| / 2 and largest tneg of the lines
};

constexpr int kFarList = 256;
constexpr int kQuad = 4;   // sources per scan work item
constexpr int kAccX = 4;   // accumulator column of tile column 0 (16-byte aligned rows)

// r / P of the residual split, never 0, so that the shares P_s / P can still be
// had from r_s = P_s r / P (r = 0 counts as 1e-20 P)
__device__ __forceinline__ float split_ratio(float r, float p)
{
    const float k = r / p;
    return fabsf(k) < 1e-20f ? 1e-20f : k;
}

}  // namespace eprsplat

// The tile kernel for one tile shape (splat_*.cu): launch, and the shared
// memory attributes of its variants.
#define EPR_SPLAT_DECLARE(TH, TW)                                                                \
    cudaError_t epr_splat_launch_##TH##x##TW(const EprConsts& C, const eprsplat::SplatArgs& A,      \
                                             int resid, bool occ6, dim3 grid, size_t smem,       \
                                             cudaStream_t stream);                              \
    cudaError_t epr_splat_init_##TH##x##TW();
EPR_SPLAT_DECLARE(64, 64)
EPR_SPLAT_DECLARE(32, 64)
EPR_SPLAT_DECLARE(64, 32)
EPR_SPLAT_DECLARE(32, 32)
#undef EPR_SPLAT_DECLARE

#ifdef EPR_SPLAT_KERNELS
namespace {

using namespace eprsplat;

// Threads of a splat block: 256 for one line; 512 for several lines (a
// runtime count, or 4 or 8 at compile time), whose per-line accumulators
// limit a 32 x 64 tile to two blocks per SM: the wider block doubles the
// warps that hide the latency of the shared-memory atomics.  With the line
// count known at compile time the line loop unrolls, so the compiler can
// interleave the lines' dependency chains.
__host__ __device__ constexpr int splat_threads(int NS) { return NS == 1 ? 256 : 512; }

// i / d for 0 <= i < 2^20 and d < 2^12 without an integer division
__device__ __forceinline__ int fdiv(int i, float inv_d) { return (int)(((float)i + 0.5f) * inv_d); }

__device__ __forceinline__ float exp2_approx(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// largest magnitude of three, and the smaller of two; NaN if one is NaN
__device__ __forceinline__ float max_abs3(float a, float b, float c)
{
    float r;
    asm("max.ftz.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float min_nan(float a, float b)
{
    float r;
    asm("min.ftz.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

// Accumulator modes: float (uint32 of value * 2^S), fixed point as two uint32
// planes, fixed point as uint64.
enum { ACC_F32 = 0, ACC_FX2 = 1, ACC_FX64 = 2 };

// v is already scaled by the accumulator's 2^S (2^40 in fixed point); the
// second plane of ACC_FX2 follows the first at `plane` words.
template <int MODE>
__device__ __forceinline__ void acc_add(void* acc, int idx, int plane, float v, const SplatArgs& A)
{
    if constexpr (MODE == ACC_F32) {
        atomicAdd(reinterpret_cast<unsigned int*>(acc) + idx, __float2uint_rn(v));
    } else if constexpr (MODE == ACC_FX2) {
        // hi = floor(v / 2^L); v - hi 2^L is exact (v has 24 bits), and its
        // rounding is that of v to an integer
        const unsigned int hi = __float2uint_rz(v * A.fx_lo_inv);
        const unsigned int lo = __float2uint_rn(fmaf(-(float)hi, A.fx_lo_s, v));
        unsigned int* a = reinterpret_cast<unsigned int*>(acc) + idx;
        atomicAdd(a, lo);
        atomicAdd(a + plane, hi);
    } else {
        atomicAdd(reinterpret_cast<unsigned long long*>(acc) + idx,
                  (unsigned long long)__float2ll_rn(v));
    }
}

template <int MODE>
__device__ __forceinline__ unsigned long long acc_fx(const void* acc, int idx, int plane, int L)
{
    if constexpr (MODE == ACC_FX2) {
        const unsigned int* a = reinterpret_cast<const unsigned int*>(acc) + idx;
        return (unsigned long long)a[0] + ((unsigned long long)a[plane] << L);
    } else {
        return reinterpret_cast<const unsigned long long*>(acc)[idx];
    }
}

// NS = 1: single line known at compile time; NS = 0: C.ns lines.
// Shared layout: accumulators [ns][TH + 2][TW + 8], the tile with a one-pixel
// apron (its rows start at a 16-byte boundary, so the flush reads four pixels
// at once); the staged thickness window [SH][SWa] whose first column
// ax0 = tx0 - HX is 16-byte aligned (HX = reach + 1 rounded up to 4); a list
// of far sources.
//
// The tile shape is a compile-time parameter (64 x 64, 32 x 64, 64 x 32 or
// 32 x 32, chosen on the host), and so is the reach RC for the reaches the
// tuner tries (RC = 0 takes C.smax), so every tile- and reach-derived index,
// stride and offset folds into immediates.  Five blocks per SM (48 registers;
// a 64 x 64 tile at reach 4 takes 43 KB of shared memory).
// XT: an x-dependent spectrum, the line constants read per source column
// from the plan's table (runtime line count and reach only).
// OCC > 0: that many blocks per SM (six for the one-line residual kernels of
// the tiles smaller than 64 x 64 at reach 3 and 4: 40 registers).
template <int NS, int MODE, bool RESID, int TH, int TW, int RC = 0, bool XT = false, int OCC = 0>
__global__ void __launch_bounds__(splat_threads(NS),
                                  OCC > 0 ? OCC : NS != 1 ? 2 : ((RESID && RC == 0) ? 4 : 5))
k_splat(const __grid_constant__ EprConsts C, const SplatArgs A)
{
    constexpr int kSplatThreads = splat_threads(NS);
    constexpr bool DET = MODE != ACC_F32;
    static_assert((TW & (TW - 1)) == 0 && TH * TW <= 4 * 4 * kSplatThreads, "tile shape");
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_far_idx[kFarList];
    __shared__ unsigned int s_far_mask[kFarList];
    __shared__ int s_far_n, s_far_base;
    const int b = blockIdx.z;
    const int nx = C.nx, ny = C.ny;
    const int ns = NS ? NS : C.ns;
    const int ty0 = blockIdx.y * TH, tx0 = blockIdx.x * TW;
    const int R = RC > 0 ? RC : C.smax;
    const int RH = TH + 2 * R, RW = TW + 2 * R;     // source region
    const int RHq = (RH + kQuad - 1) / kQuad;         // its rows in quads
    const int HX = (R + 1 + 3) & ~3;
    const int SH = RHq * kQuad + 2, SWa = TW + 2 * HX;   // staged thickness
    const int coff = HX - R - 1;                     // staged column of source column tx0 - R - 1
    constexpr int tile = TH * TW;
    constexpr int AP = TW + 2 * kAccX, ACC = (TH + 2) * AP;
    const int plane = ns * ACC;                       // words of one plane (ACC_FX2)
    const size_t npix = (size_t)nx * ny;
    const int tid = threadIdx.x;

    void* acc = smem;
    const size_t acc_bytes = (size_t)ns * ACC * (DET ? 8 : 4);
    float* Ts = reinterpret_cast<float*>(smem + ((acc_bytes + 15) & ~size_t(15)));
    const float* Tb = A.T + (size_t)b * npix;
    if (tid == 0) s_far_n = 0;

    // the detector data of the tile (residual output): its lines are asked for
    // here and loaded after the scan, whose registers they would take
    constexpr int kDq = 4;   // float4 per thread: tiles up to 64 x 64
    constexpr int nq = tile >> 2;
    constexpr int tw4 = TW >> 2;
    const bool split = !RESID && A.D != nullptr;   // a solve with several lines or in fixed point
    if (RESID || split) {
        constexpr int kLine = TW / 32;   // 128-byte lines of a row
        if (tid < TH * kLine) {
            const int gy = ty0 + tid / kLine, gx = tx0 + 32 * (tid % kLine);
            if (gy < ny && gx < nx) prefetch_l2(A.D + (size_t)b * npix + (size_t)gy * nx + gx);
        }
    }

    {   // ACC = 2 (TH + 2)(TW / 2 + 4), a multiple of 4
        uint4* a = reinterpret_cast<uint4*>(acc);
        for (int i = tid; i < ns * ACC / (DET ? 2 : 4); i += kSplatThreads) a[i] = make_uint4(0u, 0u, 0u, 0u);
    }
    // T, the done flags and the overflow counters come from earlier kernels
    epr_grid_wait();
    if (A.check_done && A.st[b].done) return;

    const int sy0 = ty0 - R - 1, sx0 = tx0 - R - 1, ax0 = tx0 - HX;
    const bool interior = sy0 >= 0 && sx0 >= 0 && sy0 + SH <= ny && sx0 + RW + 2 <= nx;
    {
        const int q = SWa >> 2;
        const float inv_q = 1.f / (float)q;
        for (int i = tid; i < SH * q; i += kSplatThreads) {
            const int ly = fdiv(i, inv_q), c4 = i - ly * q;
            const int gy = min(max(sy0 + ly, 0), ny - 1), gx = ax0 + 4 * c4;
            const float* src = Tb + (size_t)gy * nx;
            if (gx >= 0 && gx < nx) {   // nx % 4 == 0: all four or none
                cp_async16(reinterpret_cast<float4*>(Ts) + i, src + gx);
            } else {                     // the edge value (only the nearest column is read)
                const float v = __ldg(src + (gx < 0 ? 0 : nx - 1));
                reinterpret_cast<float4*>(Ts)[i] = make_float4(v, v, v, v);
            }
        }
        cp_async_commit();
        cp_async_wait_all();
    }
    __syncthreads();

    const float fsmax = (float)R;
    // the accumulator scale 2^S is folded into the line weight: a power of two
    // scales exactly, so each contribution rounds to the same integer
    const float fxs = DET ? EPR_FX_SCALE : A.fxs;
    constexpr float kLog2e = 1.4426950408889634f;
    // A source with lines too far for the scan (bits of `far`), at region-local
    // (ly, lx): its owner appends it.  Gradients are kept doubled (hi - lo),
    // and half the shift constant multiplies them: 0.5 scales exactly.
    auto append_far = [&](int ly, int lx, unsigned int far, float t, float gx2, float gy2) {
        if (!((unsigned)(ly - R) < (unsigned)TH && (unsigned)(lx - R) < (unsigned)TW)) return;
        const int sy = ty0 - R + ly, sx = tx0 - R + lx;
        const int pos = atomicAdd(&s_far_n, 1);
        if (pos < kFarList) {
            s_far_idx[pos] = sy * nx + sx;
            s_far_mask[pos] = far;
        } else {   // list full: append to the global list directly
            const int gpos = atomicAdd(&A.st[b].ovf_count[A.parity], 1);
            if (gpos < C.ovf_cap) {
                A.ovf_idx[(size_t)b * C.ovf_cap + gpos] = sy * nx + sx;
                A.ovf_mask[(size_t)b * C.ovf_cap + gpos] = far;
                A.ovf_tg[(size_t)b * C.ovf_cap + gpos] = make_float4(t, gx2, gy2, 0.f);
            } else {
                atomicOr(A.err, EPR_DEVERR_OVERFLOW);
            }
        }
    };
    // The scan: a thread takes kQuad vertically adjacent sources of one
    // column (rows ly0 .. ly0 + kQuad - 1 of the region, padded to a multiple
    // of kQuad; padding rows cannot reach the tile and are not owned by it),
    // reusing the column's thickness values.  Sources 0, 1 and 2, 3 of the
    // quad are the two lanes of packed arithmetic: the column's six values
    // form the pairs (c0, c1), (c2, c3), (c4, c5), whose differences are the
    // row gradients of both pairs.  The scan was bound by instruction issue
    // (75 % active in a batch): the packed forms, the floor by rounding mode
    // (FRND and F2I run at an eighth of the FMA rate) and one long-shift test
    // per quad took the kernel from 123 to 94 thread instructions per pixel and
    // from 142 to 103 us for eight 2048^2 projections.  Instruction issue is
    // still what bounds it (81 % active; the L1 data path, for the staged
    // window and the accumulator atomics, 66 %).
    // Work item (qy, lx) is advanced by kSplatThreads = dly quad rows +
    // dlx columns.
    const int nitem = RHq * RW;
    const int dly = kSplatThreads / RW, dlx = kSplatThreads - dly * RW;
    auto scan = [&](auto interior_tag) {
        constexpr bool IN = decltype(interior_tag)::value;
        int qy = tid / RW, lx = tid - (tid / RW) * RW;
        for (int i = tid; i < nitem; i += kSplatThreads, lx += dlx,
                 qy += dly + (lx >= RW ? 1 : 0), lx -= (lx >= RW ? RW : 0)) {
            const int ly0 = qy * kQuad;
            const float* tp = Ts + (ly0 + 1) * SWa + (lx + 1 + coff);   // source (ly0, lx)
            float2 c[kQuad / 2 + 1], g_x[kQuad / 2], g_y[kQuad / 2];   // column pairs, twice the gradients
#pragma unroll
            for (int j = 0; j < kQuad / 2 + 1; ++j)
                c[j] = make_float2(tp[(2 * j - 1) * SWa], tp[2 * j * SWa]);
            const int sx = tx0 - R + lx;
            if (!IN && (sx < 0 || sx >= nx)) continue;
#pragma unroll
            for (int j = 0; j < kQuad / 2; ++j) {
                g_x[j] = sub2(make_float2(tp[2 * j * SWa + 1], tp[(2 * j + 1) * SWa + 1]),
                              make_float2(tp[2 * j * SWa - 1], tp[(2 * j + 1) * SWa - 1]));
                g_y[j] = sub2(c[j + 1], c[j]);
                if constexpr (!IN) {   // one-sided differences are not halved
                    if (sx == 0 || sx == nx - 1) g_x[j] = add2(g_x[j], g_x[j]);
                    const int sy = ty0 - R + ly0 + 2 * j;
                    if (sy == 0 || sy == ny - 1) g_y[j].x += g_y[j].x;
                    if (sy + 1 == 0 || sy + 1 == ny - 1) g_y[j].y += g_y[j].y;
                }
            }
            bool ok[kQuad];   // sources on the grid
#pragma unroll
            for (int j = 0; j < kQuad; ++j) ok[j] = IN || (unsigned)(ty0 - R + ly0 + j) < (unsigned)ny;
            const float t[kQuad] = {c[0].y, c[1].x, c[1].y, c[2].x};
            // The lines' contributions; CHECK tests every source and line for a
            // long shift, which goes to the list instead.
            auto lines = [&](auto check_tag) {
                constexpr bool CHECK = decltype(check_tag)::value;
                unsigned int far[kQuad] = {0u, 0u, 0u, 0u};
#pragma unroll(NS ? NS : 1)
                for (int s = 0; s < ns; ++s) {
                    const float ch = 0.5f * (XT ? xt_get(C, EPR_XT_C, s, sx) : C.c[s]);
#pragma unroll
                    for (int j = 0; j < kQuad / 2; ++j) {
                        const float2 ux = mul2(both(ch), g_x[j]), uy = mul2(both(ch), g_y[j]);
                        bool near0 = ok[2 * j], near1 = ok[2 * j + 1];
                        if constexpr (CHECK) {   // false for a NaN
                            const float tneg = XT ? xt_get(C, EPR_XT_TNEG, s, sx) : C.tneg[s];
                            const bool n0 = fabsf(ux.x) <= fsmax && fabsf(uy.x) <= fsmax && t[2 * j] >= tneg;
                            const bool n1 = fabsf(ux.y) <= fsmax && fabsf(uy.y) <= fsmax && t[2 * j + 1] >= tneg;
                            if (near0 && !n0) far[2 * j] |= 1u << s;
                            if (near1 && !n1) far[2 * j + 1] |= 1u << s;
                            near0 = near0 && n0;
                            near1 = near1 && n1;
                        }
                        int ix0, ix1, iy0, iy1;
                        const float2 dx = floor_frac2(ux, ix0, ix1), dy = floor_frac2(uy, iy0, iy1);
                        // corner 00, counted from the apron: all four corners have
                        // a slot when one is in the tile
                        const int cx0 = lx - R + 1 + ix0, cx1 = lx - R + 1 + ix1;
                        const int cy0 = ly0 + 2 * j - R + 1 + iy0, cy1 = ly0 + 2 * j - R + 2 + iy1;
                        const bool in0 = near0 && (unsigned)cx0 <= (unsigned)TW && (unsigned)cy0 <= (unsigned)TH;
                        const bool in1 = near1 && (unsigned)cx1 <= (unsigned)TW && (unsigned)cy1 <= (unsigned)TH;
                        if (in0 || in1) {
                            const float fs = XT ? xt_get(C, EPR_XT_F, s, sx) : C.f[s];
                            const float mk = -(XT ? xt_get(C, EPR_XT_MU, s, sx) : C.mu[s]) * kLog2e;
                            // 2^S f e^(-mu t)
                            const float2 m = mul2(both(fs * fxs),
                                                  make_float2(exp2_approx(mk * t[2 * j]), exp2_approx(mk * t[2 * j + 1])));
                            const float2 mx1 = mul2(m, dx), mx0 = sub2(m, mx1);
                            const float2 w = sub2(both(1.f), dy);
                            const float2 v00 = mul2(mx0, w), v10 = mul2(mx1, w);
                            const float2 v01 = mul2(mx0, dy), v11 = mul2(mx1, dy);
                            if (in0) {
                                const int idx = s * ACC + cy0 * AP + cx0 + kAccX - 1;
                                acc_add<MODE>(acc, idx, plane, v00.x, A);
                                acc_add<MODE>(acc, idx + 1, plane, v10.x, A);
                                acc_add<MODE>(acc, idx + AP, plane, v01.x, A);
                                acc_add<MODE>(acc, idx + AP + 1, plane, v11.x, A);
                            }
                            if (in1) {
                                const int idx = s * ACC + cy1 * AP + cx1 + kAccX - 1;
                                acc_add<MODE>(acc, idx, plane, v00.y, A);
                                acc_add<MODE>(acc, idx + 1, plane, v10.y, A);
                                acc_add<MODE>(acc, idx + AP, plane, v01.y, A);
                                acc_add<MODE>(acc, idx + AP + 1, plane, v11.y, A);
                            }
                        }
                    }
                }
                if constexpr (CHECK) {
#pragma unroll
                    for (int j = 0; j < kQuad; ++j)
                        if (far[j])
                            append_far(ly0 + j, lx, far[j], t[j], j & 1 ? g_x[j / 2].y : g_x[j / 2].x,
                                       j & 1 ? g_y[j / 2].y : g_y[j / 2].x);
                }
            };
            if constexpr (!IN || XT) {
                lines(std::true_type{});
            } else {
                // no line's shift is long when that of the largest |c_s| is not;
                // a NaN fails the test
                const float um = max_abs3(max_abs3(max_abs3(g_x[0].x, g_x[0].y, g_x[1].x), g_x[1].y, g_y[0].x),
                                          g_y[0].y, max_abs3(g_y[1].x, g_y[1].y, 0.f));
                if (A.ch_max * um <= fsmax &&
                    min_nan(min_nan(t[0], t[1]), min_nan(t[2], t[3])) >= A.tneg_max)
                    lines(std::false_type{});
                else
                    lines(std::true_type{});
            }
        }
    };
    if (interior) scan(std::true_type{});
    else scan(std::false_type{});
    float4 dreg[kDq];
    if (RESID || (split && !DET)) {   // under way while the block meets at the barrier
#pragma unroll
        for (int k = 0; k < kDq; ++k) {
            const int i4 = tid + k * kSplatThreads;
            dreg[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (i4 < nq) {
                const int ly = i4 / tw4, lx = (i4 - ly * tw4) << 2;
                const int gy = ty0 + ly, gx = tx0 + lx;
                if (gy < ny && gx < nx)
                    dreg[k] = __ldg(reinterpret_cast<const float4*>(A.D + (size_t)b * npix + (size_t)gy * nx + gx));
            }
        }
    }
    __syncthreads();
    epr_grid_release();

    // far sources of this block: one reservation in the global list.  Each
    // entry carries T and twice the gradient, formed from the staged window
    // as in the scan (the same bits), so the overflow kernel reads no T.
    const int nfar = s_far_n < kFarList ? s_far_n : kFarList;
    if (nfar > 0) {
        if (tid == 0) s_far_base = atomicAdd(&A.st[b].ovf_count[A.parity], nfar);
        __syncthreads();
        for (int e = tid; e < nfar; e += kSplatThreads) {
            const int gpos = s_far_base + e;
            if (gpos < C.ovf_cap) {
                const int pix = s_far_idx[e];
                const int sy = pix / nx, sx = pix - sy * nx;
                const int ly = sy - ty0 + R, lx = sx - tx0 + R;   // in the source region
                const float* tp = Ts + (ly + 1) * SWa + (lx + 1 + coff);
                const float t = tp[0];
                float gx2 = tp[1] - tp[-1], gy2 = tp[SWa] - tp[-SWa];
                if (sx == 0 || sx == nx - 1) gx2 += gx2;
                if (sy == 0 || sy == ny - 1) gy2 += gy2;
                A.ovf_idx[(size_t)b * C.ovf_cap + gpos] = pix;
                A.ovf_mask[(size_t)b * C.ovf_cap + gpos] = s_far_mask[e];
                A.ovf_tg[(size_t)b * C.ovf_cap + gpos] = make_float4(t, gx2, gy2, 0.f);
            } else {
                atomicOr(A.err, EPR_DEVERR_OVERFLOW);
            }
        }
    }

    // flush: every pixel of the tile inside the grid, once, coalesced, four
    // at a time
    if constexpr (!DET) {
        const uint4* a = reinterpret_cast<const uint4*>(acc);
        const float inv = A.fxs_inv;
#pragma unroll
        for (int kk = 0; kk < kDq; ++kk) {
            const int i4 = tid + kk * kSplatThreads;
            if (i4 >= nq) continue;
            const int ly = i4 / tw4, lx = (i4 - ly * tw4) << 2;
            const int gy = ty0 + ly, gx = tx0 + lx;
            if (gy >= ny || gx >= nx) continue;
            const size_t o = (size_t)b * npix + (size_t)gy * nx + gx;
            const int i0 = ((ly + 1) * AP + lx + kAccX) >> 2;
            if constexpr (RESID) {
                const uint4 v = a[i0];
                const float4 d = dreg[kk];
                *reinterpret_cast<float4*>(A.P + o) =
                    make_float4(d.x - (float)v.x * inv, d.y - (float)v.y * inv,
                                d.z - (float)v.z * inv, d.w - (float)v.w * inv);
            } else {
                // sum <= 2 (2 reach + 3)^2 sum_s f_s: no overflow either
                uint4 sum = make_uint4(0u, 0u, 0u, 0u);
                for (int s = 0; s < ns; ++s) {
                    const uint4 v = a[s * (ACC / 4) + i0];
                    sum = make_uint4(sum.x + v.x, sum.y + v.y, sum.z + v.z, sum.w + v.w);
                }
                float4 p = make_float4((float)sum.x * inv, (float)sum.y * inv, (float)sum.z * inv,
                                       (float)sum.w * inv);
                // what the lines' values are multiplied by: 1, or r / P
                float4 k = make_float4(1.f, 1.f, 1.f, 1.f);
                const bool bx = p.x > 1e-30f, by = p.y > 1e-30f, bz = p.z > 1e-30f, bw = p.w > 1e-30f;
                if (split) {
                    const float4 d = dreg[kk];
                    const float4 r = make_float4(d.x - p.x, d.y - p.y, d.z - p.z, d.w - p.w);
                    if (ns > 1) *reinterpret_cast<float4*>(A.Pnear + o) = p;
                    k = make_float4(bx ? split_ratio(r.x, p.x) : r.x, by ? split_ratio(r.y, p.y) : r.y,
                                    bz ? split_ratio(r.z, p.z) : r.z, bw ? split_ratio(r.w, p.w) : r.w);
                    p = r;
                }
                *reinterpret_cast<float4*>(A.P + o) = p;
                for (int s = 0; ns > 1 && A.Ps && s < ns; ++s) {
                    const uint4 q = a[s * (ACC / 4) + i0];
                    float4 v = make_float4((float)q.x * inv, (float)q.y * inv, (float)q.z * inv, (float)q.w * inv);
                    if (split) {   // f_s where P vanishes
                        auto f = [&](int i) { return XT ? xt_get(C, EPR_XT_F, s, gx + i) : C.f[s]; };
                        if (!(bx && by && bz && bw))
                            v = make_float4(bx ? v.x : f(0), by ? v.y : f(1), bz ? v.z : f(2), bw ? v.w : f(3));
                        v = make_float4(k.x * v.x, k.y * v.y, k.z * v.z, k.w * v.w);
                    }
                    *reinterpret_cast<float4*>(A.Ps + (size_t)s * npix + o + (size_t)b * (ns - 1) * npix) = v;
                }
            }
        }
    } else {
        for (int i = tid; i < tile; i += kSplatThreads) {
            const int ly = i / TW, lx = i & (TW - 1);
            const int gy = ty0 + ly, gx = tx0 + lx;
            if (gy >= ny || gx >= nx) continue;
            const size_t o = (size_t)b * npix + (size_t)gy * nx + gx;
            unsigned long long sum = 0ull;
            for (int s = 0; s < ns; ++s) {
                const unsigned long long q =
                    acc_fx<MODE>(acc, s * ACC + (ly + 1) * AP + lx + kAccX, plane, A.fx_lo);
                sum += q;
                if (ns > 1) A.Psq[(size_t)s * npix + o + (size_t)b * (ns - 1) * npix] = q;
            }
            A.Pq[o] = sum;
            if (split) {
                const float p = (float)sum * EPR_FX_INV, r = __ldg(&A.D[o]) - p;
                const bool lit = p > 1e-30f;
                const float k = lit ? split_ratio(r, p) : r;
                A.P[o] = r;
                for (int s = 0; ns > 1 && s < ns; ++s) {
                    const unsigned long long q =
                        acc_fx<MODE>(acc, s * ACC + (ly + 1) * AP + lx + kAccX, plane, A.fx_lo);
                    const float f = XT ? xt_get(C, EPR_XT_F, s, gx) : C.f[s];
                    A.Ps[(size_t)s * npix + o + (size_t)b * (ns - 1) * npix] =
                        k * (lit ? (float)q * EPR_FX_INV : f);
                }
            }
        }
    }
}

template <int NS, int MODE, bool RESID, int TH, int TW, int RC = 0, bool XT = false, int OCC = 0>
cudaError_t launch_t(const EprConsts& C, const SplatArgs& A, dim3 grid, size_t smem,
                     cudaStream_t stream)
{
    return epr_launch_kernel(C.pdl != 0, k_splat<NS, MODE, RESID, TH, TW, RC, XT, OCC>, grid,
                             dim3(splat_threads(NS)), smem, stream, C, A);
}

// Tiles whose one-line residual kernel has a six-blocks-per-SM variant.
template <int TH, int TW>
constexpr bool has_occ6() { return TH * TW < 64 * 64; }

template <int TH, int TW, int MODE>
cudaError_t launch_fx(const EprConsts& C, const SplatArgs& A, dim3 grid, size_t smem,
                      cudaStream_t stream)
{
    if (C.xt) return launch_t<0, MODE, false, TH, TW, 0, true>(C, A, grid, smem, stream);
    const bool r4 = MODE == ACC_FX2 && C.smax == 4;   // the default reach
    if (C.ns == 1)
        return r4 ? launch_t<1, MODE, false, TH, TW, MODE == ACC_FX2 ? 4 : 0>(C, A, grid, smem, stream)
                  : launch_t<1, MODE, false, TH, TW>(C, A, grid, smem, stream);
    return r4 ? launch_t<0, MODE, false, TH, TW, MODE == ACC_FX2 ? 4 : 0>(C, A, grid, smem, stream)
              : launch_t<0, MODE, false, TH, TW>(C, A, grid, smem, stream);
}

template <int TH, int TW>
cudaError_t launch_shape(const EprConsts& C, const SplatArgs& A, int resid, bool occ6, dim3 grid,
                         size_t smem, cudaStream_t stream)
{
    const bool mono = C.ns == 1;
    if (C.det)
        return A.fx_lo > 0 ? launch_fx<TH, TW, ACC_FX2>(C, A, grid, smem, stream)
                           : launch_fx<TH, TW, ACC_FX64>(C, A, grid, smem, stream);
    if (C.xt)   // x-dependent spectrum: the generic kernels with per-column constants
        return launch_t<0, ACC_F32, false, TH, TW, 0, true>(C, A, grid, smem, stream);
    if constexpr (has_occ6<TH, TW>()) {
        if (resid && mono && occ6 && C.smax == 3)
            return launch_t<1, ACC_F32, true, TH, TW, 3, false, 6>(C, A, grid, smem, stream);
        if (resid && mono && occ6 && C.smax == 4)
            return launch_t<1, ACC_F32, true, TH, TW, 4, false, 6>(C, A, grid, smem, stream);
    }
    if (resid && mono) {
        switch (C.smax) {
        case 3: return launch_t<1, ACC_F32, true, TH, TW, 3>(C, A, grid, smem, stream);
        case 4: return launch_t<1, ACC_F32, true, TH, TW, 4>(C, A, grid, smem, stream);
        case 6: return launch_t<1, ACC_F32, true, TH, TW, 6>(C, A, grid, smem, stream);
        default: return launch_t<1, ACC_F32, true, TH, TW>(C, A, grid, smem, stream);
        }
    }
    if (mono)
        return C.smax == 4 ? launch_t<1, ACC_F32, false, TH, TW, 4>(C, A, grid, smem, stream)
                           : launch_t<1, ACC_F32, false, TH, TW>(C, A, grid, smem, stream);
    if (C.ns == 8)   // the common polychromatic counts with an unrolled line loop
        return C.smax == 4 ? launch_t<8, ACC_F32, false, TH, TW, 4>(C, A, grid, smem, stream)
                           : launch_t<8, ACC_F32, false, TH, TW>(C, A, grid, smem, stream);
    if (C.ns == 4)
        return C.smax == 4 ? launch_t<4, ACC_F32, false, TH, TW, 4>(C, A, grid, smem, stream)
                           : launch_t<4, ACC_F32, false, TH, TW>(C, A, grid, smem, stream);
    switch (C.smax) {
    case 3: return launch_t<0, ACC_F32, false, TH, TW, 3>(C, A, grid, smem, stream);
    case 4: return launch_t<0, ACC_F32, false, TH, TW, 4>(C, A, grid, smem, stream);
    case 6: return launch_t<0, ACC_F32, false, TH, TW, 6>(C, A, grid, smem, stream);
    default: return launch_t<0, ACC_F32, false, TH, TW>(C, A, grid, smem, stream);
    }
}

template <int TH, int TW>
cudaError_t init_shape()
{
    cudaError_t e = cudaSuccess;
    auto allow = [&](auto kernel) { if (e == cudaSuccess) e = epr_allow_max_smem(kernel); };
    allow(k_splat<1, ACC_FX2, false, TH, TW, 4>);
    allow(k_splat<0, ACC_FX2, false, TH, TW, 4>);
    allow(k_splat<1, ACC_FX2, false, TH, TW>);
    allow(k_splat<0, ACC_FX2, false, TH, TW>);
    allow(k_splat<1, ACC_FX64, false, TH, TW>);
    allow(k_splat<0, ACC_FX64, false, TH, TW>);
    allow(k_splat<1, ACC_F32, true, TH, TW>);
    allow(k_splat<1, ACC_F32, true, TH, TW, 3>);
    allow(k_splat<1, ACC_F32, true, TH, TW, 4>);
    allow(k_splat<1, ACC_F32, true, TH, TW, 6>);
    allow(k_splat<1, ACC_F32, false, TH, TW, 4>);
    allow(k_splat<1, ACC_F32, false, TH, TW>);
    allow(k_splat<0, ACC_F32, false, TH, TW>);
    allow(k_splat<0, ACC_F32, false, TH, TW, 3>);
    allow(k_splat<0, ACC_F32, false, TH, TW, 4>);
    allow(k_splat<0, ACC_F32, false, TH, TW, 6>);
    allow(k_splat<8, ACC_F32, false, TH, TW, 4>);
    allow(k_splat<8, ACC_F32, false, TH, TW>);
    allow(k_splat<4, ACC_F32, false, TH, TW, 4>);
    allow(k_splat<4, ACC_F32, false, TH, TW>);
    allow(k_splat<0, ACC_FX2, false, TH, TW, 0, true>);
    allow(k_splat<0, ACC_FX64, false, TH, TW, 0, true>);
    allow(k_splat<0, ACC_F32, false, TH, TW, 0, true>);
    if constexpr (has_occ6<TH, TW>()) {
        allow(k_splat<1, ACC_F32, true, TH, TW, 3, false, 6>);
        allow(k_splat<1, ACC_F32, true, TH, TW, 4, false, 6>);
    }
    return e;
}

}  // namespace

#define EPR_SPLAT_DEFINE(TH, TW)                                                                 \
    cudaError_t epr_splat_launch_##TH##x##TW(const EprConsts& C, const SplatArgs& A, int resid,     \
                                             bool occ6, dim3 grid, size_t smem,                  \
                                             cudaStream_t stream)                               \
    {                                                                                            \
        return launch_shape<TH, TW>(C, A, resid, occ6, grid, smem, stream);                      \
    }                                                                                            \
    cudaError_t epr_splat_init_##TH##x##TW() { return init_shape<TH, TW>(); }
#endif  // EPR_SPLAT_KERNELS
