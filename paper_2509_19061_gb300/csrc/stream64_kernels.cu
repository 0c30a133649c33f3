// stream64_kernels.cu -- temporally blocked Jacobi by row streaming in FP64:
// fused Jacobi and RAS schedules that equal global Jacobi (overlap >= k - 1),
// on grids large enough to fill the GPU.  The FP32 form and the reasons for
// the traversal are in stream_kernels.cu.
//
// FP64 is bound by its pipe (two lanes per clock and SM), so what counts is
// the number of FP64 operations per cell and sweep: the stencil's 18 (square
// cells), four more per pass for the coefficients, and the halo.  A CTA is a
// chain of one warp per sweep over a strip of 64 columns (two per lane): warp
// 0 takes in the snapshot's row s in step s, forms its coefficients and writes
// them over the staged fields, runs the first sweep on row s - 1 and hands
// that row to warp 1, which runs the second sweep one step later, and so on;
// the last warp writes out.  One barrier a step.  A warp only runs the rows
// its successors still need.
//
// 100 sweeps of 1024^2 take 5.2 ms (20 Gcell-updates/s, 0.85 of the pipe for the
// operations and halo above) against 6.8 on 32 x 32 tiles, whose halo and
// per-tile coefficients cost more operations and whose phases leave the pipe
// idle in between; 40 sweeps of 4096^2 29.3 ms against 40.9.
#include <algorithm>

#include "internal.h"
#include "stencil.cuh"
#include "tma.h"

namespace stokes {

namespace {

constexpr int S8_COLS = 64;  // columns of a strip
constexpr int S8_MAX = 4;    // sweeps of a pass
constexpr long long S8_MIN_CELLS = 100000; // smallest grid
constexpr int S8_D = 10;     // staged rows
constexpr int S8_PF = S8_D - 2 * S8_MAX; // rows copied ahead
constexpr int S8_FIELDS = 9; // vx, vy, eta_c (2 eta_c / hx^2), eta_n (eta_n / h^2), bx, by, 1/dx, 1/dy (omega / diag), 2 eta_c / hy^2
constexpr int S8_ROW = S8_FIELDS * S8_COLS; // elements of a staged row
constexpr int S8_HAND = 2 * 2 * S8_COLS;    // a handed-over row: step parity, vx, vy
constexpr size_t S8_SMEM = (size_t)(S8_D * S8_ROW + (S8_MAX - 1) * S8_HAND) * sizeof(double);

struct Stream64 {
    GridDesc<double> g;
    const double *f[8];
    double omega;
    double *ox, *oy;
    int strips, rows, hl, own;
};

struct D2 {
    double a, b;
};
__device__ __forceinline__ D2 ld2(const double *p)
{
    const double2 v = *reinterpret_cast<const double2 *>(p);
    return {v.x, v.y};
}
__device__ __forceinline__ void st2(double *p, D2 v) { *reinterpret_cast<double2 *>(p) = make_double2(v.a, v.b); }
__device__ __forceinline__ D2 sub(D2 x, D2 y) { return {r_sub(x.a, y.a), r_sub(x.b, y.b)}; }
__device__ __forceinline__ D2 add(D2 x, D2 y) { return {r_add(x.a, y.a), r_add(x.b, y.b)}; }
__device__ __forceinline__ D2 mul(D2 x, D2 y) { return {r_mul(x.a, y.a), r_mul(x.b, y.b)}; }
__device__ __forceinline__ D2 mul(D2 x, double y) { return {r_mul(x.a, y), r_mul(x.b, y)}; }
__device__ __forceinline__ D2 fma(D2 x, double y, D2 z) { return {r_fma(x.a, y, z.a), r_fma(x.b, y, z.b)}; }
__device__ __forceinline__ D2 fma(D2 x, D2 y, D2 z) { return {r_fma(x.a, y.a, z.a), r_fma(x.b, y.b, z.b)}; }
// x - its west neighbour, its east neighbour - x, column by column
__device__ __forceinline__ D2 diff_west(D2 x)
{
    return {r_sub(x.a, __shfl_up_sync(0xffffffffu, x.b, 1)), r_sub(x.b, x.a)};
}
__device__ __forceinline__ D2 diff_east(D2 x)
{
    return {r_sub(x.b, x.a), r_sub(__shfl_down_sync(0xffffffffu, x.a, 1), x.b)};
}

// blockDim.x / 32 sweeps of strip blockIdx.x % strips, segment blockIdx.x / strips
template <bool SQ>
__global__ void __launch_bounds__(S8_MAX * 32, 4) k_stream64(const __grid_constant__ Stream64 a)
{
    extern __shared__ __align__(16) double smem8[];
    const int m = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = (int)threadIdx.x & 31;
    const int n = (int)blockDim.x >> 5; // sweeps; this warp runs sweep m + 1
    const int strip = (int)blockIdx.x % a.strips, seg = (int)blockIdx.x / a.strips;
    const int nx = a.g.nx, ny = a.g.ny, P = a.g.pitch;
    const int c0 = strip * a.own - a.hl + 2 * lane; // first of this lane's columns (even, may lie outside)
    const int y0 = seg * a.rows, y1 = min(y0 + a.rows, ny);
    const int jb = y0 - n; // first row loaded
    double *const ring = smem8 + 2 * lane;
    double *const hand = ring + S8_D * S8_ROW;

    // bytes of this lane's columns inside a row of nx (cell) or nx + 1 (node) columns
    const int bc = c0 < 0 ? 0 : max(0, min(2, nx - c0)) * 8;
    const int bn = c0 < 0 ? 0 : max(0, min(2, nx + 1 - c0)) * 8;
    const int cc = min(max(c0, 0), P - 2); // columns inside the rows for the copies that read nothing
    auto issue = [&](int j, int slot) {
        const long long at = (long long)min(max(j, 0), ny) * P + cc;
        const bool in0 = (unsigned)j < (unsigned)ny, in1 = (unsigned)j <= (unsigned)ny; // rows of the cells / of the nodes
        const int cr = in0 ? bc : 0, nr = in0 ? bn : 0, cn = in1 ? bc : 0, nn = in1 ? bn : 0;
        const int bytes[8] = {nr, cn, cr, nn, nr, cn, nr, cn};
        const uint32_t to = smem_addr(ring + slot * S8_ROW);
#pragma unroll
        for (int f = 0; f < 8; ++f) cp_async16z(to + f * S8_COLS * 8, a.f[f] + at, bytes[f]);
        cp_commit();
    };
    if (m == 0)
        for (int d = 0; d < S8_PF; ++d) issue(jb + d, d);

    const double ihx = a.g.ihx, ihy = a.g.ihy;
    const D2 zero = {0.0, 0.0};
    // at the last row taken in: velocity before this sweep, scaled shear, Tyy of the row before
    D2 vx = zero, vy = zero, sx = zero, sy = zero, ty = zero;
    const bool mine = 2 * lane >= a.hl && 2 * lane < a.hl + a.own && c0 < nx;
    // the rows this warp updates: those its successors and the output need
    const int r0 = y0 - (n - 1 - m), r1 = y1 + (n - 1 - m);
    const int steps = (y1 - y0) + 3 * n - 1; // the last sweep's row in step s is jb + s - 2 n + 1
    int slot = (S8_D * 2 - 2 * m) % S8_D;    // staged slot of the row taken in, jb + s - 2 m
    for (int s = 0; s < steps; ++s) {
        const int j = jb + s - 2 * m; // row taken in; the sweep updates row j - 1
        const int prev = slot == 0 ? S8_D - 1 : slot - 1;
        double *const in = ring + slot * S8_ROW;
        if (m == 0) {
            int to = slot + S8_PF;
            if (to >= S8_D) to -= S8_D;
            cp_wait<S8_PF - 1>();
            // the row's coefficients (coef_x, coef_y: doubling 1/h^2 is exact;
            // shear_sq, jacobi_weight) take the place of the fields they come from
            if (j <= r1) {
                const D2 ec = ld2(in + 2 * S8_COLS), en = ld2(in + 3 * S8_COLS);
                st2(in + 2 * S8_COLS, mul(ec, a.g.two_ihx2));
                if (!SQ) st2(in + 8 * S8_COLS, mul(ec, a.g.two_ihy2));
                if (SQ) st2(in + 3 * S8_COLS, mul(en, a.g.ihx2));
                st2(in + 6 * S8_COLS, mul(ld2(in + 6 * S8_COLS), a.omega));
                st2(in + 7 * S8_COLS, mul(ld2(in + 7 * S8_COLS), a.omega));
            }
            issue(j + S8_PF, to);
        }
        // (row r0 - 1 only leaves its velocity, row r0 its shear and Tyy)
        if (j >= r0 - 1 && j <= r1) {
            const double *const from = m == 0 ? in : hand + (m - 1) * S8_HAND + ((s - 1) & 1) * 2 * S8_COLS;
            const double *const cf = ring + prev * S8_ROW; // row j - 1
            const D2 ix = ld2(from), iy = ld2(from + S8_COLS);
            if (j >= r0) {
                const D2 en = ld2(in + 3 * S8_COLS);
                const D2 ax = ld2(cf + 2 * S8_COLS), ay = SQ ? ax : ld2(cf + 8 * S8_COLS);
                D2 sxn, syn;
                if (SQ) {
                    sxn = syn = mul(en, add(sub(ix, vx), diff_west(iy)));
                } else {
                    const D2 sh = mul(en, fma(sub(ix, vx), ihy, mul(diff_west(iy), ihx)));
                    sxn = mul(sh, ihy);
                    syn = mul(sh, ihx);
                }
                const D2 tyy = mul(ay, sub(iy, vy));
                if (j > r0) {
                    const D2 txx = mul(ax, diff_east(vx));
                    const D2 mx = add(diff_west(txx), sub(sxn, sx));
                    const D2 my = add(diff_east(sy), sub(tyy, ty));
                    const D2 nvx = fma(sub(ld2(cf + 4 * S8_COLS), mx), ld2(cf + 6 * S8_COLS), vx);
                    const D2 nvy = fma(sub(ld2(cf + 5 * S8_COLS), my), ld2(cf + 7 * S8_COLS), vy);
                    if (m < n - 1) {
                        double *const out = hand + m * S8_HAND + (s & 1) * 2 * S8_COLS;
                        st2(out, nvx);
                        st2(out + S8_COLS, nvy);
                    } else if (mine && j - 1 >= y0) { // the unknowns of the strip's own cells
                        const long long q = (long long)(j - 1) * P + c0;
                        const bool two = c0 + 1 < nx;
                        if (c0 >= 1 && two) st2(a.ox + q, nvx);
                        else if (c0 >= 1) a.ox[q] = nvx.a;
                        else if (two) a.ox[q + 1] = nvx.b;
                        if (j - 1 >= 1) {
                            if (two) st2(a.oy + q, nvy);
                            else a.oy[q] = nvy.a;
                        }
                    }
                }
                sx = sxn;
                sy = syn;
                ty = tyy;
            }
            vx = ix;
            vy = iy;
        }
        __syncthreads(); // this step's rows and coefficients are handed over
        slot = slot + 1 == S8_D ? 0 : slot + 1;
    }
    cp_wait<0>(); // no copy outlives the CTA
}

} // namespace

int stream64_passes(int nx, int ny, int sweeps, const RasRun &run)
{
    if (!run.allow_tma || run.pair_mode != 1 || sweeps < 2) return 0;
    // (40 sweeps: 256^2 377 us, 337 on 24 x 24 tiles; 384^2 470 and 544)
    if ((long long)nx * ny < S8_MIN_CELLS) return 0;
    return (sweeps + S8_MAX - 1) / S8_MAX;
}

cudaError_t launch_ras_stream64(const GridDesc<double> &g, const Coeffs<double> &c, double omega, int sweeps,
                                const double *vx, const double *vy, double *ox, double *oy, cudaStream_t s)
{
    if (!c.inv_dx || !c.inv_dy || sweeps < 1 || sweeps > S8_MAX) return cudaErrorInvalidValue;
    Stream64 a;
    a.g = g;
    a.omega = omega;
    a.ox = ox;
    a.oy = oy;
    const double *const f[8] = {vx, vy, c.eta_c, c.eta_n, c.bx, c.by, c.inv_dx, c.inv_dy};
    for (int q = 0; q < 8; ++q) a.f[q] = f[q];
    a.hl = sweeps <= 2 ? 2 : 4;
    a.own = S8_COLS - 2 * a.hl;
    a.strips = (g.nx + a.own - 1) / a.own;
    // chains per SM: more fill the FP64 pipe better, fewer have longer segments
    // and so fewer halo rows (40 sweeps with 2, 3, 4 a SM: 384^2 470, 579, 575
    // us; 768^2 1316, 1269, 1300; 2048^2 7947, 7655, 7533)
    const long long cells = (long long)g.nx * g.ny;
    const int per = cells >= 1000000 ? 4 : cells >= 400000 ? 3 : 2;
    const int segs = std::max(1, 152 * per / a.strips);
    a.rows = std::min(g.ny, std::max((g.ny + segs - 1) / segs, 8));
    const int ns = (g.ny + a.rows - 1) / a.rows;
    void (*const kern)(Stream64) = g.square ? k_stream64<true> : k_stream64<false>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S8_SMEM);
    if (e != cudaSuccess) return e;
    kern<<<a.strips * ns, sweeps * 32, S8_SMEM, s>>>(a);
    return cudaGetLastError();
}

} // namespace stokes
