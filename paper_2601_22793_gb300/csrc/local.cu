// Local O(L^2) forward closure (arXiv 2601.22793, Eq. 1) in pixel units,
// and its diffraction-pressure term alone for the non-local model to second
// order, per spectral line, summed over lines (Eq. 5):
//   P_s = I - D_x(I u_x) - D_y(I u_y)                                    m = 1
//       + 1/2 [D_xx(I u_x^2) + 2 D_x D_y(I u_x u_y) + D_yy(I u_y^2)]
//       - eps^2/(4 p^4) [D_x(I D_x Q) + D_y(I D_y Q)]                      m = 2
// with I = f_s exp(-mu_s T), u = c_s G[T] and Q = (D_xx + D_yy) sqrt(I) /
// sqrt(I).  D_i: central differences, one-sided at the grid edges; D_ii:
// [1, -2, 1] with the edge value replicated.  (eps grad phi = p u and the
// physical derivative is D / p, which gives these pixel-unit forms.)
//
// A warp owns a strip of columns and marches down its rows.  Every
// intermediate field lives in registers, the last three rows of those that are
// differentiated along y, and horizontal neighbours come by warp shuffle, so
// there is no shared memory and no barrier.  The nested derivatives reach 3
// pixels (2 for m = 1): 26 (28) of the 32 lanes are output columns, and a
// strip of H rows computes H + 6.  221 (second-order term) and 304 (m = 2)
// thread instructions per pixel; the tile form this replaces staged every field
// in shared memory and spent 440 and 620, most of them on its index arithmetic,
// its barriers' phases and expm1.  47 and 58 % of the issue slots are used: what
// is left is the wait for the rows of T and P at 28 warps per SM.
// Stencils test the GLOBAL coordinate for the edge rules, so values computed
// outside the grid are never used by an in-grid output.  No atomics: the
// result is the same on every run.
//
// In a solve (D given) the kernel also forms the residual and its split over
// the lines, which would otherwise be a pass of its own over P and P_s.
#include "epr_internal.cuh"

namespace {

constexpr int kStencilThreads = 128;
constexpr int kStencilBlocks = 7;   // per SM: 72 registers a thread
constexpr int kStencilSlots = EPR_SMS * kStencilBlocks * (kStencilThreads / 32);   // resident warps

enum { ST_LOCAL1 = 1, ST_LOCAL2 = 2, ST_WKB1 = 3 };

struct StencilArgs {
    const float* T;
    const float* D;                  // solve: P <- D - P, P_s <- split residuals; else NULL
    float* P;                        // [B][ny][nx] out (ST_WKB1: the splat's P in, float mode)
    float* Ps;                       // [B][ns][ny][nx] (ns > 1), likewise, or NULL: not wanted
    const unsigned long long* Pq;    // ST_WKB1: fixed-point sums of the splat (DET)
    const unsigned long long* Psq;
    const EprProjState* st;
    int check_done;
    int H, strips;                   // rows and strips of a projection
};

// The sum of e^x - 1 over four arguments.  For |x| < 1/4 the Taylor series to
// x^8 / 8! (the first omitted term, x^9 / 9!, is below 4.3e-11 |x|), whose rounding is
// that of its last operations, as packed pairs; one test for all four.
__device__ __forceinline__ float2 expm1_taylor(float2 x)
{
    float2 p = fma2(x, both(1.f / 40320.f), both(1.f / 5040.f));
    p = fma2(x, p, both(1.f / 720.f));
    p = fma2(x, p, both(1.f / 120.f));
    p = fma2(x, p, both(1.f / 24.f));
    p = fma2(x, p, both(1.f / 6.f));
    p = fma2(x, p, both(0.5f));
    return fma2(mul2(x, x), p, x);
}
__device__ __noinline__ float expm1_sum4_any(float a, float b, float c, float d)
{
    return (expm1f(a) + expm1f(b)) + (expm1f(c) + expm1f(d));
}
__device__ __forceinline__ float expm1_sum4(float2 x, float2 y)
{
    const float big = fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(y.x), fabsf(y.y)));
    if (!(big < 0.25f)) return expm1_sum4_any(x.x, x.y, y.x, y.y);
    const float2 e = add2(expm1_taylor(x), expm1_taylor(y));   // a NaN argument stays one
    return e.x + e.y;
}

// Three consecutive rows of a field: m (row - 1), c (row), p (row + 1).
struct Rows3 {
    float m, c, p;
    __device__ __forceinline__ void push(float v)
    {
        m = c;
        c = p;
        p = v;
    }
};

template <int MODE, bool DET>
__global__ void __launch_bounds__(kStencilThreads, kStencilBlocks) k_stencil(const EprConsts C, const StencilArgs A)
{
    constexpr int HALO = MODE == ST_LOCAL1 ? 2 : 3, OUT = 32 - 2 * HALO;
    constexpr bool PRESSURE = MODE != ST_LOCAL1, LOCAL = MODE != ST_WKB1;
    const int nx = C.nx, ny = C.ny, ns = C.ns, b = blockIdx.z;
    epr_grid_wait();
    if (A.check_done && A.st[b].done) return;
    epr_grid_release();
    const int lane = threadIdx.x & 31;
    const int w = (blockIdx.x * kStencilThreads + threadIdx.x) >> 5;
    const int y0 = (w / A.strips) * A.H;
    if (y0 >= ny) return;   // a whole warp
    const int gx = (w % A.strips) * OUT - HALO + lane;
    const int y1 = min(y0 + A.H, ny);   // rows y0 .. y1 - 1
    const size_t npix = (size_t)nx * ny, pb = (size_t)b * npix;
    // this lane's column of each map; offsets within a map fit in an int
    const float* Tc = A.T + pb + min(max(gx, 0), nx - 1);
    const float* Dc = A.D ? A.D + pb + gx : nullptr;
    float* Pc = A.P + pb + gx;
    const bool xl = gx <= 0, xh = gx >= nx - 1;
    const float hsx = xl || xh ? 1.f : 0.5f;
    const bool out = lane >= HALO && lane < 32 - HALO && gx < nx;

    // horizontal neighbours, the edge value replicated
    auto left = [&](float f) { const float v = __shfl_up_sync(0xffffffffu, f, 1); return xl ? f : v; };
    auto right = [&](float f) { const float v = __shfl_down_sync(0xffffffffu, f, 1); return xh ? f : v; };
    auto dX = [&](float f) { return (right(f) - left(f)) * hsx; };
    auto dXX = [&](float f) { return left(f) - 2.f * f + right(f); };
    auto dY = [&](const Rows3& f, int y) {
        const bool lo = y == 0, hi = y == ny - 1;
        return ((hi ? f.c : f.p) - (lo ? f.c : f.m)) * (lo || hi ? 1.f : 0.5f);
    };
    auto dYY = [&](const Rows3& f, int y) {
        return (y == 0 ? f.c : f.m) - 2.f * f.c + (y == ny - 1 ? f.c : f.p);
    };
    auto ldT = [&](int y) { return __ldg(Tc + min(max(y, 0), ny - 1) * nx); };

    for (int s = 0; s < ns; ++s) {
        const float fs = line_const(C.f, s), mus = line_const(C.mu, s);
        const float cs = line_const(C.c, s), qc = line_const(C.qc, s);
        const float hm = -0.5f * mus;
        // Row yl of T arrives at step yl; the fields I, u, Q and the fluxes are
        // formed at row a = yl - 1, their first y derivatives and the flux of Q
        // at row b = yl - 2, and the derivative of that flux at row c = yl - 3.
        Rows3 t = {0.f, ldT(y0 - HALO), ldT(y0 - HALO + 1)};
        Rows3 Q = {}, AY = {}, BYY = {}, BXY = {}, CYQ = {};
        float Ib = 0.f, Ia = 0.f, Sc = 0.f, Sb = 0.f, Sa = 0.f;   // Sx: the terms known so far at row x
        float ahead = ldT(y0 - HALO + 2), ahead2 = ldT(y0 - HALO + 3);
        // what the output rows need besides: D on the last line, and the
        // prediction so far (the splat's, or the earlier lines')
        const bool lastD = A.D && s == ns - 1;
        const bool sofar = s > 0 || MODE == ST_WKB1;
        auto ldD = [&](int y) { return lastD && out && y < y1 ? __ldg(Dc + y * nx) : 0.f; };
        auto ldP = [&](int y) {
            if (!(sofar && out && y < y1)) return 0.f;
            return DET && s == 0 ? (float)A.Pq[pb + (size_t)y * nx + gx] * EPR_FX_INV : Pc[y * nx];
        };
        float d0 = 0.f, d1 = ldD(y0), p0 = 0.f, p1 = ldP(y0);   // rows yo, yo + 1
#pragma unroll 3
        for (int yl = y0 - HALO + 2; yl <= y1 - 1 + HALO; ++yl) {
            const int a = yl - 1, bb = yl - 2;
            t.push(ahead);   // rows a - 1, a, a + 1 after this push
            ahead = ahead2;
            ahead2 = ldT(yl + 2);
            const float T0 = t.c, Tl = left(T0), Tr = right(T0);
            const float Tu = a <= 0 ? T0 : t.m, Td = a >= ny - 1 ? T0 : t.p;
            Ib = Ia;
            Sc = Sb;
            Sb = Sa;
            Ia = fs * __expf(-mus * T0);
            Sa = LOCAL ? Ia : 0.f;
            if constexpr (LOCAL) {
                const float ux = cs * ((Tr - Tl) * hsx), uy = cs * dY(t, a);
                const float ax = Ia * ux, ay = Ia * uy;
                AY.push(ay);
                Sa -= dX(ax);
                if constexpr (PRESSURE) {
                    Sa += 0.5f * dXX(ax * ux);
                    BYY.push(ay * uy);
                    BXY.push(ax * uy);
                }
                Sb -= dY(AY, bb);
            }
            if constexpr (PRESSURE) {
                // Q = (D_xx + D_yy) sqrt(I) / sqrt(I).  With sqrt(I) = sqrt(f) e^(-mu T / 2)
                // each neighbour n contributes sqrt(I_n) / sqrt(I) - 1 = expm1(-mu (T_n - T) / 2)
                // (a replicated edge neighbour contributes 0): the same quotient
                // without the cancellation of second differences of a near-constant.
                const float q = expm1_sum4(mul2(both(hm), sub2(make_float2(Tl, Tr), both(T0))),
                                           mul2(both(hm), sub2(make_float2(Tu, Td), both(T0))));
                Q.push(Ia > 0.f ? q : 0.f);
                // the x derivatives of the two fluxes at row b are one
                float fx = -qc * (Ib * dX(Q.c));
                if constexpr (LOCAL) {
                    Sb += 0.5f * dYY(BYY, bb);
                    fx += dY(BXY, bb);
                }
                Sb += dX(fx);
                CYQ.push(Ib * dY(Q, bb));
            }
            const int yo = PRESSURE ? yl - 3 : bb;   // the row that is complete
            if (yo >= y0) {
                d0 = d1;
                p0 = p1;
                d1 = ldD(yo + 1);
                p1 = ldP(yo + 1);
            }
            const float p = PRESSURE ? Sc - qc * dY(CYQ, yo) : Sb;
            if (!out || yo < y0 || yo >= y1) continue;
            const float tot = p0 + p;   // the prediction of all lines so far
            const size_t o = (size_t)yo * nx + gx;
            if (ns > 1) {
                const size_t os = pb * ns + (size_t)s * npix + o;
                float ps = p;
                if (A.Ps) {
                    if constexpr (MODE == ST_WKB1) ps += DET ? (float)A.Psq[os] * EPR_FX_INV : A.Ps[os];
                    A.Ps[os] = ps;
                }
            }
            const float r = d0 - tot;
            Pc[yo * nx] = lastD ? r : tot;
            if (!lastD) continue;
            if (ns > 1) {   // this thread wrote every line's value of the pixel
                const bool pos = tot > 1e-30f;
                const float k = pos ? r / tot : r;
                for (int l = 0; l < ns; ++l) {
                    float* q = &A.Ps[pb * ns + (size_t)l * npix + o];
                    *q = k * (pos ? *q : line_const(C.f, l));
                }
            }
        }
    }
}

template <int MODE, bool DET>
cudaError_t launch_stencil(const EprConsts& C, StencilArgs& A, int batch, cudaStream_t stream)
{
    constexpr int OUT = MODE == ST_LOCAL1 ? 28 : 26;
    A.strips = (C.nx + OUT - 1) / OUT;
    // Strips that fill the resident warps a whole number of times.  One frame
    // of 2048 x 2048 (39 rows and one wave; 32 rows made 1.2), ten second-order
    // iterations: 1218 -> 1098 us; four of 1024 x 1024 (40 rows; 1.2 waves
    // before), 20 iterations of order 2: 2053 -> 1870 us.  At most 48 rows: 64
    // measured the same, 32 and 24 1.7 % slower per solve.
    A.H = epr_strip_rows(A.strips, C.ny, epr_rule_batch(C, batch), kStencilSlots, 4, 48);
    const int warps = A.strips * ((C.ny + A.H - 1) / A.H);
    const dim3 grid((warps * 32 + kStencilThreads - 1) / kStencilThreads, 1, batch);
    const cudaError_t e = epr_launch_kernel(C.pdl != 0, k_stencil<MODE, DET>, grid, dim3(kStencilThreads), 0,
                                            stream, C, A);
    epr_count_launch(1);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

// Second-order term of the non-local model, after the splat (one launch).
// fixed_point = 1 reads the splat's integer sums.  With D (a solve) the
// residual D - P and its split replace P and P_s.
cudaError_t epr_launch_wkb1(const EprConsts& C, const EprWork& W, const float* T, const float* D,
                            int fixed_point, int batch, int check_done, cudaStream_t stream)
{
    StencilArgs A = {};
    A.T = T;
    A.D = D;
    A.P = W.P;
    A.Ps = W.Ps;
    A.Pq = W.Pq;
    A.Psq = W.Psq;
    A.st = W.st;
    A.check_done = check_done;
    return fixed_point ? launch_stencil<ST_WKB1, true>(C, A, batch, stream)
                       : launch_stencil<ST_WKB1, false>(C, A, batch, stream);
}

// The local closure of order 1 or 2 (one launch); D as above.
cudaError_t epr_launch_local(const EprConsts& C, const EprWork& W, const float* T, const float* D, float* P,
                             float* Ps, int order, int batch, int check_done, cudaStream_t stream)
{
    StencilArgs A = {};
    A.T = T;
    A.D = D;
    A.P = P;
    A.Ps = Ps;
    A.st = W.st;
    A.check_done = check_done;
    return order >= 2 ? launch_stencil<ST_LOCAL2, false>(C, A, batch, stream)
                      : launch_stencil<ST_LOCAL1, false>(C, A, batch, stream);
}
