// rbgs_kernels.cu -- red-black Gauss-Seidel by row streaming (Sec. 5 (i)), FP32,
// on grids large enough to fill the GPU; smaller grids and FP64 run
// k_rbgs_tile (sweep_kernels.cu).
//
// The half-sweeps vx red, vx black, vy red, vy black each read at most the
// adjacent rows, so a sweep can follow the rows: when row r arrives, vx red
// runs on row r - 1, vx black and vy red on row r - 2 and vy black on row
// r - 3, which is then final.  Every point reads what it reads in the in-place
// sweep, so the values are the same.  One warp runs one sweep on a strip of
// 128 columns (four per lane), holding the five rows of velocity it needs in
// registers; a second warp runs the next sweep four rows behind on the rows
// the first hands over in shared memory, and reads the coefficients from the
// same staged rows.  A tile of 32 x 32 cells staged a 40 x 40 window and met
// at four barriers a sweep: 47 us a sweep at 2000^2 and 629 at 8192^2; here 27 and
// 336, bound by issue (each value is formed by every sweep's own warp), where the eight
// fields read and two written per two sweeps take 12 us a sweep at the copy rate.
#include <algorithm>

#include "internal.h"
#include "stencil.cuh"
#include "tma.h"

namespace stokes {

namespace {

constexpr int RB_COLS = 128;  // columns of a strip
constexpr int RB_MAX = 2;     // sweeps of a pass, one warp each
// Smallest grid: at 512^2 the strips do not fill the SMs and the tiles are as
// fast (20 sweeps 171 us either way); 768^2 takes 253 us by tiles and 232 here,
// 1024^2 340 and 274, 2000^2 950 and 541.
constexpr long long RB_MIN_CELLS = 400000;
// Narrowest grid (a strip sweeps 128 columns however few there are): six sweeps
// of 32 x 25000 take 103 us by tiles and 142 here, of 48 x 16666 116 and 113.
constexpr int RB_MIN_NX = 48;
constexpr int RB_LAG = 4;     // rows from one sweep to the next (three, and one for the hand-over)
constexpr int RB_D = 12;      // staged rows
constexpr int RB_PF = RB_D - 1 - RB_LAG * RB_MAX; // rows copied ahead
constexpr int RB_FIELDS = 8;  // vx, vy; eta_c, eta_n, bx, by, 1/dx, 1/dy
constexpr int RB_CF = RB_FIELDS - 2;     // of them, the coefficients and b stay for RB_D rows,
constexpr int RB_DV = RB_PF + 1;         // the velocity until it is taken in
constexpr int RB_ROW = RB_CF * RB_COLS;
constexpr int RB_HAND = 2 * 2 * RB_COLS; // a handed-over row: step parity, vx, vy
constexpr int RB_CTAS = 4;               // per SM (a fifth would fit; shorter segments cost what it gains)
constexpr size_t RB_SMEM =
    (size_t)(RB_D * RB_ROW + RB_DV * 2 * RB_COLS + (RB_MAX - 1) * RB_HAND) * sizeof(float);
static_assert(RB_PF >= 2, "rows in flight");

struct RbArgs {
    GridDesc<float> g;
    const float *f[RB_FIELDS];
    float omega;
    float *ox, *oy;
    int strips, rows, hl, own;
};

// four adjacent columns of a row
struct Q4 {
    float e[4];
};
__device__ __forceinline__ Q4 ldq(const float *p)
{
    const float4 v = *reinterpret_cast<const float4 *>(p);
    return {{v.x, v.y, v.z, v.w}};
}
__device__ __forceinline__ void stq(float *p, const Q4 &v)
{
    *reinterpret_cast<float4 *>(p) = make_float4(v.e[0], v.e[1], v.e[2], v.e[3]);
}
// the last column of the lane to the west, the first of the lane to the east
__device__ __forceinline__ float west(const Q4 &v) { return __shfl_up_sync(0xffffffffu, v.e[3], 1); }
__device__ __forceinline__ float east(const Q4 &v) { return __shfl_down_sync(0xffffffffu, v.e[0], 1); }

// vx of the columns K, K + 2 of row j from its neighbours (gs_half's
// operations): rows j + 1 and j - 1 of vx, rows j + 1 and j of vy
template <int K, bool SQ>
__device__ __forceinline__ void half_x(const RbArgs &a, Q4 &v, const Q4 &vn, const Q4 &vs, const Q4 &yn, const Q4 &yc,
                                       const Q4 &ec, const Q4 &enn, const Q4 &enc, const Q4 &b, const Q4 &inv)
{
    const GridDesc<float> &g = a.g;
    // west of column 0 and east of column 3 lie in other lanes
    const float vw = K == 0 ? west(v) : 0.f, ecw = K == 0 ? west(ec) : 0.f;
    const float ynw = K == 0 ? west(yn) : 0.f, ycw = K == 0 ? west(yc) : 0.f, ve = K == 1 ? east(v) : 0.f;
    float nv[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = K + 2 * h, w = c > 0 ? c - 1 : 0, e = c < 3 ? c + 1 : 3;
        const float vc = v.e[c];
        const float txx_c = flux_n(coef_x(g, ec.e[c]), c < 3 ? v.e[e] : ve, vc);
        const float txx_w = flux_n(coef_x(g, c > 0 ? ec.e[w] : ecw), vc, c > 0 ? v.e[w] : vw);
        const float sx_n = shear_x<SQ ? 1 : 0>(g, enn.e[c], vn.e[c], vc, yn.e[c], c > 0 ? yn.e[w] : ynw);
        const float sx_c = shear_x<SQ ? 1 : 0>(g, enc.e[c], vc, vs.e[c], yc.e[c], c > 0 ? yc.e[w] : ycw);
        nv[h] = jacobi_update(vc, b.e[c], m_x(txx_c, txx_w, sx_n, sx_c), jacobi_weight(a.omega, inv.e[c]));
    }
    v.e[K] = nv[0];
    v.e[K + 2] = nv[1];
}

// vy of the columns K, K + 2 of row j: rows j + 1 and j - 1 of vy, rows j and j - 1 of vx
template <int K, bool SQ>
__device__ __forceinline__ void half_y(const RbArgs &a, Q4 &v, const Q4 &vn, const Q4 &vs, const Q4 &xc, const Q4 &xs,
                                       const Q4 &ec, const Q4 &ecs, const Q4 &enc, const Q4 &b, const Q4 &inv)
{
    const GridDesc<float> &g = a.g;
    const float vw = K == 0 ? west(v) : 0.f, ve = K == 1 ? east(v) : 0.f;
    const float xce = K == 1 ? east(xc) : 0.f, xse = K == 1 ? east(xs) : 0.f, ene = K == 1 ? east(enc) : 0.f;
    float nv[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = K + 2 * h, w = c > 0 ? c - 1 : 0, e = c < 3 ? c + 1 : 3;
        const float vc = v.e[c];
        const float tyy_c = flux_n(coef_y(g, ec.e[c]), vn.e[c], vc);
        const float tyy_s = flux_n(coef_y(g, ecs.e[c]), vc, vs.e[c]);
        const float sy_e = shear_y<SQ ? 1 : 0>(g, c < 3 ? enc.e[e] : ene, c < 3 ? xc.e[e] : xce,
                                               c < 3 ? xs.e[e] : xse, c < 3 ? v.e[e] : ve, vc);
        const float sy_c = shear_y<SQ ? 1 : 0>(g, enc.e[c], xc.e[c], xs.e[c], vc, c > 0 ? v.e[w] : vw);
        nv[h] = jacobi_update(vc, b.e[c], m_y(sy_e, sy_c, tyy_c, tyy_s), jacobi_weight(a.omega, inv.e[c]));
    }
    v.e[K] = nv[0];
    v.e[K + 2] = nv[1];
}

// blockDim.x / 32 sweeps of strip blockIdx.x % strips, segment blockIdx.x / strips
template <bool SQ>
__global__ void __launch_bounds__(RB_MAX * 32, RB_CTAS) k_rbgs_stream(const __grid_constant__ RbArgs a)
{
    extern __shared__ __align__(16) float rb_smem[];
    const int m = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = (int)threadIdx.x & 31;
    const int n = (int)blockDim.x >> 5; // sweeps
    const int strip = (int)blockIdx.x % a.strips, seg = (int)blockIdx.x / a.strips;
    const int nx = a.g.nx, ny = a.g.ny, P = a.g.pitch;
    const int c0 = strip * a.own - a.hl + 4 * lane; // a multiple of four; may lie outside
    const int y0 = seg * a.rows, y1 = min(y0 + a.rows, ny);
    // A sweep's output row j reads rows j - 4 .. j + 3 of its input.  One row
    // less below would do for rows that only the next sweep reads.
    const int jb = y0 - 4 * n;
    float *const ring = rb_smem + 4 * lane;
    float *const vel = ring + RB_D * RB_ROW; // vx, vy of RB_DV rows
    float *const hand = vel + RB_DV * 2 * RB_COLS;

    const int bc = c0 < 0 ? 0 : max(0, min(4, nx - c0)) * 4;     // bytes inside a row of cells
    const int bn = c0 < 0 ? 0 : max(0, min(4, nx + 1 - c0)) * 4; // of nodes
    const int cc = min(max(c0, 0), P - 4);
    auto issue = [&](int j, int slot, int vslot) {
        const long long at = (long long)min(max(j, 0), ny) * P + cc;
        const bool in0 = (unsigned)j < (unsigned)ny, in1 = (unsigned)j <= (unsigned)ny;
        const int cr = in0 ? bc : 0, nr = in0 ? bn : 0, cn = in1 ? bc : 0, nn = in1 ? bn : 0;
        const int bytes[RB_FIELDS] = {nr, cn, cr, nn, nr, cn, nr, cn};
        const uint32_t to = smem_addr(ring + slot * RB_ROW), tov = smem_addr(vel + vslot * 2 * RB_COLS);
#pragma unroll
        for (int f = 0; f < RB_FIELDS; ++f)
            cp_async16z(f < 2 ? tov + f * RB_COLS * 4 : to + (f - 2) * RB_COLS * 4, a.f[f] + at, bytes[f]);
        cp_commit();
    };
    if (m == 0)
        for (int d = 0; d < RB_PF; ++d) issue(jb + d, d, d);

    const Q4 zero = {{0.f, 0.f, 0.f, 0.f}};
    Q4 x0 = zero, x1 = zero, x2 = zero, x3 = zero, x4 = zero; // vx of rows r .. r - 4
    Q4 z0 = zero, z1 = zero, z2 = zero, z3 = zero, z4 = zero; // vy
    const bool mine = 4 * lane >= a.hl && 4 * lane < a.hl + a.own && c0 < nx;
    // step s: sweep m + 1 takes in row jb + s - 4 m and finishes the row three below
    const int steps = (y1 - y0) + 4 * n + 4 * (n - 1) + 3;
    int slot = (RB_D - (RB_LAG * m) % RB_D) % RB_D; // staged slot of the row taken in
    auto back = [&](int d) { // the staged row d rows below
        int q = slot - d;
        return ring + (q < 0 ? q + RB_D : q) * RB_ROW;
    };
    for (int s = 0; s < steps; ++s) {
        const int r = jb + s - RB_LAG * m;
        if (m == 0) {
            int to = slot + RB_PF;
            if (to >= RB_D) to -= RB_D;
            cp_wait<RB_PF - 1>();
            __syncwarp();
            issue(r + RB_PF, to, (s + RB_PF) % RB_DV);
        }
        if (s >= RB_LAG * m) {
            const float *const from = m == 0 ? vel + s % RB_DV * 2 * RB_COLS : hand + (m - 1) * RB_HAND + ((s - 1) & 1) * 2 * RB_COLS;
            x4 = x3;
            x3 = x2;
            x2 = x1;
            x1 = x0;
            z4 = z3;
            z3 = z2;
            z2 = z1;
            z1 = z0;
            x0 = ldq(from);
            z0 = ldq(from + RB_COLS);
            const float *const p0 = back(0), *const p1 = back(1), *const p2 = back(2), *const p3 = back(3);
            const Q4 en0 = ldq(p0 + 1 * RB_COLS), en1 = ldq(p1 + 1 * RB_COLS), en2 = ldq(p2 + 1 * RB_COLS);
            const Q4 ec1 = ldq(p1 + 0 * RB_COLS), ec2 = ldq(p2 + 0 * RB_COLS), ec3 = ldq(p3 + 0 * RB_COLS);
            // red: column + row even; c0 is even, so the first red column of a
            // lane is 0 in even rows and 1 in odd ones
            const bool odd = r & 1; // row r - 2 likewise, rows r - 1 and r - 3 the other way
            {
                const Q4 b = ldq(p1 + 2 * RB_COLS), iv = ldq(p1 + 4 * RB_COLS);
                if (odd) half_x<0, SQ>(a, x1, x0, x2, z0, z1, ec1, en0, en1, b, iv); // vx red, row r - 1 even
                else half_x<1, SQ>(a, x1, x0, x2, z0, z1, ec1, en0, en1, b, iv);
            }
            {
                const Q4 b = ldq(p2 + 2 * RB_COLS), iv = ldq(p2 + 4 * RB_COLS);
                if (odd) half_x<0, SQ>(a, x2, x1, x3, z1, z2, ec2, en1, en2, b, iv); // vx black, row r - 2 odd
                else half_x<1, SQ>(a, x2, x1, x3, z1, z2, ec2, en1, en2, b, iv);
            }
            {
                const Q4 b = ldq(p2 + 3 * RB_COLS), iv = ldq(p2 + 5 * RB_COLS);
                if (odd) half_y<1, SQ>(a, z2, z1, z3, x2, x3, ec2, ec3, en2, b, iv); // vy red, row r - 2 odd
                else half_y<0, SQ>(a, z2, z1, z3, x2, x3, ec2, ec3, en2, b, iv);
            }
            {
                const Q4 b = ldq(p3 + 3 * RB_COLS), iv = ldq(p3 + 5 * RB_COLS);
                const Q4 en3 = ldq(p3 + 1 * RB_COLS), ec4 = ldq(back(4) + 0 * RB_COLS);
                if (odd) half_y<1, SQ>(a, z3, z2, z4, x3, x4, ec3, ec4, en3, b, iv); // vy black, row r - 3 even
                else half_y<0, SQ>(a, z3, z2, z4, x3, x4, ec3, ec4, en3, b, iv);
            }
            const int j = r - 3; // final
            if (m < n - 1) {
                float *const out = hand + m * RB_HAND + (s & 1) * 2 * RB_COLS;
                stq(out, x3);
                stq(out + RB_COLS, z3);
            } else if (mine && j >= y0 && j < y1) { // the unknowns of the strip's own cells
                const long long q = (long long)j * P + c0;
                if (c0 >= 1 && c0 + 4 <= nx) {
                    stq(a.ox + q, x3);
                } else {
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        if (c0 + c >= 1 && c0 + c < nx) a.ox[q + c] = x3.e[c];
                }
                if (j >= 1) {
                    if (c0 + 4 <= nx) {
                        stq(a.oy + q, z3);
                    } else {
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            if (c0 + c < nx) a.oy[q + c] = z3.e[c];
                    }
                }
            }
        }
        __syncthreads(); // this step's rows are handed over
        slot = slot + 1 == RB_D ? 0 : slot + 1;
    }
    cp_wait<0>(); // no copy outlives the CTA
}

} // namespace

int rbgs_stream_passes(int nx, int ny, int sweeps, const RasRun &run)
{
    // One sweep, or two on the smaller grids, gain less than the copy back that an
    // odd pass count costs: 8192^2 one sweep 1014 us, 962 by tiles; two at 640^2
    // 28.4 and 26.4, at 1024^2 37.9 and 39.7.
    const long long least = sweeps == 2 ? 2 * RB_MIN_CELLS : RB_MIN_CELLS;
    if (!run.allow_tma || run.pair_mode != 1 || sweeps < 2 || nx < RB_MIN_NX || (long long)nx * ny < least)
        return 0;
    return (sweeps + RB_MAX - 1) / RB_MAX;
}

cudaError_t launch_rbgs_stream(const GridDesc<float> &g, const Coeffs<float> &c, float omega, int sweeps,
                               const float *vx, const float *vy, float *ox, float *oy, cudaStream_t s)
{
    if (!c.inv_dx || !c.inv_dy || sweeps < 1 || sweeps > RB_MAX) return cudaErrorInvalidValue;
    RbArgs a;
    a.g = g;
    a.omega = omega;
    a.ox = ox;
    a.oy = oy;
    const float *const f[RB_FIELDS] = {vx, vy, c.eta_c, c.eta_n, c.bx, c.by, c.inv_dx, c.inv_dy};
    for (int q = 0; q < RB_FIELDS; ++q) a.f[q] = f[q];
    a.hl = 4 * sweeps; // a sweep reads four columns to either side
    a.own = RB_COLS - 2 * a.hl;
    a.strips = (g.nx + a.own - 1) / a.own;
    const int segs = std::max(1, 152 * RB_CTAS / a.strips); // one wave
    a.rows = std::max(8, (g.ny + segs - 1) / segs);
    const int ns = (g.ny + a.rows - 1) / a.rows;
    void (*const kern)(RbArgs) = g.square ? k_rbgs_stream<true> : k_rbgs_stream<false>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RB_SMEM);
    if (e != cudaSuccess) return e;
    kern<<<a.strips * ns, sweeps * 32, RB_SMEM, s>>>(a);
    return cudaGetLastError();
}

} // namespace stokes
