// Vector-Jacobian product of the non-local forward model (not in the paper:
// the analytic transpose of the transport of Eq. 3 with the shift of Eq. 2
// and the single-thickness intensity of Eq. 7), for calibration by gradient
// descent.  With gbar = dF/dP, per line s and source pixel with mapped point
// (x + u_x, y + u_y), corner values g00, g10, g01, g11 of gbar (0 outside
// the grid) and a = M_s^* gbar there:
//   Tbar     += -mu_s I_s a                                (through I_s)
//   vx, vy   += c_s ubar_x, c_s ubar_y with
//               ubar_x = I_s [(1-d_y)(g10 - g00) + d_y (g11 - g01)],
//               ubar_y = I_s [(1-d_x)(g01 - g00) + d_x (g11 - g10)]
//               (derivative of the bilinear weights; right derivative where a
//               mapped point crosses a pixel boundary)
//   cbar_s   += ubar . G[T],   mubar_s += -T I_s a         (scalars)
// then Tbar += G^T[vx, vy], the transpose of the numpy-gradient stencil.
// The host turns cbar, mubar into dF/dL, dF/ddelta_s, dF/dbeta_s.
//
// A warp marches down a strip of 30 output columns (32 lanes): vx of the
// neighbouring columns comes by warp shuffle and the last three rows of vy
// stay in registers, so G^T needs no maps of vx and vy and no second pass.
// The two-pass form it replaces also wrote and read vx, vy and Tbar and kept
// its per-line sums in local memory.  Bound by the latency of the gather's
// loads (four corners per line and pixel, from L1 and L2): long scoreboard is
// the top stall, half of the issue slots are used.  The corners of all lines
// are therefore loaded before the first is used, and the strips are cut so
// that every resident warp has one: 41.1 us where the two-pass form took 51.3
// (1536 x 1024, 3 lines; one line 22.7 and 38.0).
#include "epr_internal.cuh"

namespace {

constexpr int kVjpThreads = 256;
constexpr int kVjpMaxBlocks = 4 * EPR_SMS;   // per projection

constexpr int kVjpSlots = kVjpMaxBlocks * (kVjpThreads / 32);   // resident warps

struct VjpArgs {
    const float* T;
    const float* gbar;
    float* Tbar;
    double* part;        // [B][kVjpMaxBlocks][2 ns]  (cbar_s, mubar_s) per block
    int H;               // rows of a strip unit
    int strips, units;   // of one projection
};

// corners of gbar at a mapped point on the rim of the field or beyond it
// (0 outside the grid), and the fractions of the clamped shift
__device__ __noinline__ void vjp_corners(const float* G, int y, int x, float uy, float ux, int ny, int nx,
                                         float (&g)[4], float& dx, float& dy)
{
    const float lim = 2.f * (float)(nx > ny ? nx : ny);
    ux = fminf(fmaxf(ux, -lim), lim);
    uy = fminf(fmaxf(uy, -lim), lim);
    const float fx = floorf(ux), fy = floorf(uy);
    dx = ux - fx;
    dy = uy - fy;
    const int cx = x + (int)fx, cy = y + (int)fy;
    const bool x0 = (unsigned)cx < (unsigned)nx, x1 = (unsigned)(cx + 1) < (unsigned)nx;
    g[0] = g[1] = g[2] = g[3] = 0.f;
    if ((unsigned)cy < (unsigned)ny) {
        const float* r = G + (size_t)cy * nx + cx;
        if (x0) g[0] = __ldg(r);
        if (x1) g[1] = __ldg(r + 1);
    }
    if ((unsigned)(cy + 1) < (unsigned)ny) {
        const float* r = G + (size_t)(cy + 1) * nx + cx;
        if (x0) g[2] = __ldg(r);
        if (x1) g[3] = __ldg(r + 1);
    }
}

// A sum of floats with its rounding error beside it (Knuth's two-sum).  The terms
// of the scalars nearly cancel: with the lanes' sums added in plain float, dF/dbeta
// was off by 12 % more than in the two-pass form, whose threads each added
// fewer terms; without those roundings by 5 % less.  39.1 -> 41.1 us.
struct Pair {
    float s, c;
    __device__ __forceinline__ void add(float s2, float c2)
    {
        const float t = s + s2, b = t - s;
        c += c2 + ((s - (t - b)) + (s2 - b));
        s = t;
    }
};

// NSM: the line count up to 4 (the corner loads of every line are then issued
// together), a bound of it above (the sums stay in registers)
template <int NSM>
__global__ void __launch_bounds__(kVjpThreads, NSM <= 8 ? 4 : 2) k_vjp(const __grid_constant__ EprConsts C, const VjpArgs A)
{
    __shared__ double red[2 * NSM][kVjpThreads / 32];
    const int nx = C.nx, ny = C.ny, ns = C.ns, b = blockIdx.y;
    const size_t npix = (size_t)nx * ny, pb = (size_t)b * npix;
    const float* Tb = A.T + pb;
    const float* Gb = A.gbar + pb;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float cacc[NSM], macc[NSM];
#pragma unroll
    for (int s = 0; s < NSM; ++s) cacc[s] = macc[s] = 0.f;
    for (int w = blockIdx.x * (kVjpThreads / 32) + wid; w < A.units; w += gridDim.x * (kVjpThreads / 32)) {
        const int y0 = (w / A.strips) * A.H, y1 = min(y0 + A.H, ny);
        const int x = (w % A.strips) * 30 - 1 + lane;
        const bool on = x >= 0 && x < nx;                    // on the grid
        const bool own = on && lane >= 1 && lane < 31;       // an output column
        const int xc = min(max(x, 0), nx - 1);
        const float* Tc = Tb + xc;
        auto ldT = [&](int y) { return __ldg(Tc + (size_t)min(max(y, 0), ny - 1) * nx); };
        float tm = 0.f, tc = ldT(y0 - 2), tp = ldT(y0 - 1), ahead = ldT(y0);
        float vym = 0.f, vyc = 0.f, out = 0.f;   // v'_y of rows r - 2, r - 1; Tbar of row r - 1 so far
        for (int r = y0 - 1; r <= y1; ++r) {   // v of row r; row r - 1 is complete
            tm = tc;
            tc = tp;
            tp = ahead;
            ahead = ldT(r + 2);
            float l = __shfl_up_sync(0xffffffffu, tc, 1), h = __shfl_down_sync(0xffffffffu, tc, 1);
            // the halo lanes' outer neighbours
            if (lane == 0) l = __ldg(Tb + (size_t)min(max(r, 0), ny - 1) * nx + max(xc - 1, 0));
            if (lane == 31) h = __ldg(Tb + (size_t)min(max(r, 0), ny - 1) * nx + min(xc + 1, nx - 1));
            const bool xe = x == 0 || x == nx - 1, ye = r == 0 || r == ny - 1;
            const float sx = xe ? 1.f : 0.5f, sy = ye ? 1.f : 0.5f;
            const float gx = ((x == nx - 1 ? tc : h) - (x == 0 ? tc : l)) * sx;
            const float gy = ((r == ny - 1 ? tc : tp) - (r == 0 ? tc : tm)) * sy;
            float tb = 0.f, vx = 0.f, vy = 0.f;
            if (on && r >= 0 && r < ny) {
                const bool mine = own && r >= y0 && r < y1;   // counted in the sums once
                // the corners of up to four lines are on their way before the
                // first is used
                constexpr int K = NSM < 4 ? NSM : 4;
#pragma unroll
                for (int s0 = 0; s0 < NSM; s0 += K) {
                    if (NSM > 4 && s0 >= ns) break;
                    float g[K][4], dxs[K], dys[K];
#pragma unroll
                    for (int k = 0; k < K; ++k) {
                        if (NSM > 4 && s0 + k >= ns) break;
                        const float cs = C.c[s0 + k];
                        const float ux = cs * gx, uy = cs * gy;
                        int ix, iy;
                        const float2 d = floor_frac2(make_float2(ux, uy), ix, iy);
                        dxs[k] = d.x;
                        dys[k] = d.y;
                        const int cx = x + ix, cy = r + iy;
                        if ((unsigned)cx < (unsigned)(nx - 1) && (unsigned)cy < (unsigned)(ny - 1)) {
                            const float* q = Gb + (cy * nx + cx);
                            g[k][0] = __ldg(q);
                            g[k][1] = __ldg(q + 1);
                            g[k][2] = __ldg(q + nx);
                            g[k][3] = __ldg(q + nx + 1);
                        } else {
                            vjp_corners(Gb, r, x, uy, ux, ny, nx, g[k], dxs[k], dys[k]);
                        }
                    }
#pragma unroll
                    for (int k = 0; k < K; ++k) {
                        if (NSM > 4 && s0 + k >= ns) break;
                        const int s = s0 + k;
                        const float cs = C.c[s], dx = dxs[k], dy = dys[k];
                        const float m = C.mu[s], Is = C.f[s] * __expf(-m * tc), ci = cs * Is;
                        // the value and the slopes as weighted means of
                        // corners and differences: a value formed from
                        // differences of corners (g00 + dx (g10 - g00) + ..)
                        // takes 35.5 us where this takes 39.1 (1536 x 1024, 3
                        // lines), but carries the rounding of the largest corner
                        const float g00 = g[k][0], g10 = g[k][1], g01 = g[k][2], g11 = g[k][3];
                        const float wx = 1.f - dx, wy = 1.f - dy;
                        const float slx = wy * (g10 - g00) + dy * (g11 - g01);
                        const float sly = wx * (g01 - g00) + dx * (g11 - g10);
                        const float Ia = Is * (wy * (wx * g00 + dx * g10) + dy * (wx * g01 + dx * g11));
                        tb -= m * Ia;
                        vx += ci * slx;
                        vy += ci * sly;
                        if (mine) {
                            cacc[s] += Is * (slx * gx + sly * gy);
                            macc[s] -= tc * Ia;
                        }
                    }
                }
            }
            // G^T: with v' = v at the edges and v / 2 elsewhere, row and column
            // i add v'(i - 1) - v'(i + 1), where a neighbour beyond the grid is
            // minus the edge value
            const float vxs = vx * sx, vys = vy * sy;
            const float vl = __shfl_up_sync(0xffffffffu, vxs, 1), vh = __shfl_down_sync(0xffffffffu, vxs, 1);
            const float row = tb + ((x == 0 ? -vxs : vl) - (x == nx - 1 ? -vxs : vh));
            const int yo = r - 1;
            if (own && yo >= y0 && yo < y1)
                A.Tbar[pb + (size_t)yo * nx + x] =
                    out + ((yo == 0 ? -vyc : vym) - (yo == ny - 1 ? -vyc : vys));
            out = row;
            vym = vyc;
            vyc = vys;
        }
    }
    // deterministic block partials: warp shuffles, then warps in order
#pragma unroll
    for (int s = 0; s < NSM; ++s) {
        Pair c = {cacc[s], 0.f}, m = {macc[s], 0.f};
        for (int o = 16; o > 0; o >>= 1) {
            c.add(__shfl_down_sync(0xffffffffu, c.s, o), __shfl_down_sync(0xffffffffu, c.c, o));
            m.add(__shfl_down_sync(0xffffffffu, m.s, o), __shfl_down_sync(0xffffffffu, m.c, o));
        }
        if (lane == 0) {
            red[2 * s][wid] = (double)c.s + (double)c.c;
            red[2 * s + 1][wid] = (double)m.s + (double)m.c;
        }
    }
    __syncthreads();
    if (threadIdx.x < 2 * ns) {
        double acc = 0.0;
        for (int i = 0; i < kVjpThreads / 32; ++i) acc += red[threadIdx.x][i];
        A.part[((size_t)b * kVjpMaxBlocks + blockIdx.x) * 2 * ns + threadIdx.x] = acc;
    }
}

// sums[b][k] of the nblk block partials, in a fixed order: one block per
// scalar and projection
__global__ void __launch_bounds__(256) k_vjp_sum(const double* part, int nblk, int n, double* sums)
{
    __shared__ double red[32];
    const int k = blockIdx.x, b = blockIdx.y;
    double v = 0.0;
    for (int i = threadIdx.x; i < nblk; i += blockDim.x) v += part[((size_t)b * kVjpMaxBlocks + i) * n + k];
    const double t = block_sum_d(v, red);
    if (threadIdx.x == 0) sums[(size_t)b * n + k] = t;
}

}  // namespace

// Doubles of workspace: the block partials.
size_t epr_vjp_part_len(int ns, int batch) { return (size_t)batch * kVjpMaxBlocks * 2 * ns; }

// The gradient, and with `sums` ([batch][2 ns]: cbar_s, mubar_s; pinned host
// memory that the kernel writes itself) the scalars.
cudaError_t epr_launch_vjp(const EprConsts& C, const float* T, const float* gbar, float* Tbar,
                           double* part, double* sums, int batch, cudaStream_t stream)
{
    VjpArgs A;
    A.T = T;
    A.gbar = gbar;
    A.Tbar = Tbar;
    A.part = part;
    A.strips = (C.nx + 29) / 30;
    // a strip's rows are a serial chain of gathers, and each strip computes two
    // more rows than it writes.  1536 x 1024, 3 lines: 11 rows (one strip per
    // resident warp) 34.5 us, 22 rows 47.9 (both with the cheaper bilinear form)
    A.H = epr_strip_rows(A.strips, C.ny, epr_rule_batch(C, batch), kVjpSlots, 8, 32);
    A.units = A.strips * ((C.ny + A.H - 1) / A.H);
    int nblk = (A.units + kVjpThreads / 32 - 1) / (kVjpThreads / 32);
    if (nblk > kVjpMaxBlocks) nblk = kVjpMaxBlocks;
    const dim3 grid(nblk, batch), blk(kVjpThreads);
    if (C.ns == 1) k_vjp<1><<<grid, blk, 0, stream>>>(C, A);
    else if (C.ns == 2) k_vjp<2><<<grid, blk, 0, stream>>>(C, A);
    else if (C.ns == 3) k_vjp<3><<<grid, blk, 0, stream>>>(C, A);
    else if (C.ns == 4) k_vjp<4><<<grid, blk, 0, stream>>>(C, A);
    else if (C.ns <= 8) k_vjp<8><<<grid, blk, 0, stream>>>(C, A);
    else k_vjp<16><<<grid, blk, 0, stream>>>(C, A);
    epr_count_launch(1);
    if (sums) {
        k_vjp_sum<<<dim3(2 * C.ns, batch), 256, 0, stream>>>(part, nblk, 2 * C.ns, sums);
        epr_count_launch(1);
    }
    return cudaGetLastError();
}
