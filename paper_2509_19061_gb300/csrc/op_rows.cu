// op_rows.cu -- the velocity operator in FP64 by row-marching warps: M v + G p
// (stokes_apply_operator) and the residual b - M v of the solves.
//
// Both are bound by the FP64 pipe (two lanes per clock and SM), so the layout
// is the one with the fewest FP64 operations per cell: a warp owns a strip of
// 60 columns (two per lane; lanes 0 and 31 carry the neighbour columns and own
// none) and marches up a band of rows, each flux is formed once, by the lane
// and in the row it belongs to, and its neighbours' come by shuffles and from
// the row before.  M v takes 16 operations a cell (square cells) and 1/15 for
// the carried columns, a thread per unknown twice the fluxes: M v + G p at
// 2000^2 took 487 us and takes 200, the residual at 4096^2 1883 and 708 (0.76
// of the FP64 pipe).  The next row's loads are issued before the current row's
// arithmetic, which hides them.  (The energy sums in this form measured 345 us
// at 2000^2 with spills and 378 without, against 352 tile by tile, and q = M p
// of the outer CG must keep the order of its inner products, whose last bits
// FP32 sweeps amplify; both stay tile by tile.)
//
// Operations and their order are those of stencil.cuh, so M v has the bits of
// the other kernels.
#include <algorithm>

#include "internal.h"
#include "stencil.cuh"

namespace stokes {

namespace {

constexpr int OR_WARPS = 4, OR_THREADS = OR_WARPS * 32;
constexpr int OR_OWN = 60; // columns of a strip
// Smaller grids leave most SMs idle, where a thread per unknown (twice the
// operations, all in parallel) is sooner done than a warp's rows in turn.
constexpr long long OR_MIN_CELLS = 100000;

constexpr int OR_BLOCKS = 4; // blocks an SM

enum { OR_APPLY, OR_RESID };


struct OpRows {
    GridDesc<double> g;
    const double *ec, *en;
    const double *vx, *vy;
    const double *p;       // OR_APPLY: pressure or NULL
    const double *bx, *by; // OR_RESID
    double *ox, *oy;
    int strips, rows;
};

__device__ __forceinline__ double up1(double v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ double dn1(double v) { return __shfl_down_sync(0xffffffffu, v, 1); }

struct D2 {
    double e[2];
};

// two columns of row j of a field of rows x cols entries, zero outside
__device__ __forceinline__ D2 ld2(const double *__restrict__ f, const GridDesc<double> &g, int j, int c, int rows,
                                  int cols)
{
    D2 r = {{0.0, 0.0}};
    if (j >= 0 && j < rows && c >= 0 && c < g.pitch) {
        const double2 v = *reinterpret_cast<const double2 *>(f + (size_t)j * g.pitch + c);
        if (c < cols) r.e[0] = v.x;
        if (c + 1 < cols) r.e[1] = v.y;
    }
    return r;
}

// the two columns' entries below `cols`
__device__ __forceinline__ void st2(double *__restrict__ f, const GridDesc<double> &g, int j, int c, int cols, D2 v)
{
    double *const p = f + (size_t)j * g.pitch + c;
    if (c + 1 < cols) *reinterpret_cast<double2 *>(p) = make_double2(v.e[0], v.e[1]);
    else if (c < cols) p[0] = v.e[0];
}

// what row j reads: vx, vy, eta_n of the row above, the rest of row j
struct OpRow {
    D2 vx, vy, en, ec, bx, by, p;
};

template <int MODE, bool SQ>
__device__ __forceinline__ void op_band(const OpRows &o, int strip, int j0, int j1)
{
    const GridDesc<double> &g = o.g;
    const int lane = (int)threadIdx.x & 31, c0 = strip * OR_OWN - 2 + 2 * lane;
    const int nx = g.nx, ny = g.ny, cx = nx + 1, cy = nx;
    const bool own = lane >= 1 && lane <= 30;
    const bool hasp = MODE == OR_APPLY && o.p;
    auto load = [&](int j) {
        OpRow r;
        r.vx = ld2(o.vx, g, j + 1, c0, ny, cx);
        r.vy = ld2(o.vy, g, j + 1, c0, ny + 1, cy);
        r.en = ld2(o.en, g, j + 1, c0, ny + 1, cx);
        r.ec = ld2(o.ec, g, j, c0, ny, cy);
        if (MODE == OR_RESID) {
            r.bx = ld2(o.bx, g, j, c0, ny, cx);
            r.by = ld2(o.by, g, j, c0, ny + 1, cy);
        }
        if (hasp) r.p = ld2(o.p, g, j, c0, ny, cy);
        return r;
    };
    // coefficients of Txx and Tyy (coef_x, coef_y: doubling eta_c or 1/h^2 is exact) and the scaled shear
    auto ax_of = [&](const OpRow &r, int k) { return r_mul(r.ec.e[k], g.two_ihx2); };
    auto ay_of = [&](const OpRow &r, int k) { return r_mul(r.ec.e[k], g.two_ihy2); };
    auto shear2 = [&](double en, double vxc, double vxs, double vyc, double vyw, double &sx, double &sy) {
        if (SQ) {
            sx = sy = shear_sq(r_mul(en, g.ihx2), vxc, vxs, vyc, vyw);
        } else {
            const double sh = shear(g, en, vxc, vxs, vyc, vyw);
            sx = r_mul(sh, g.ihy);
            sy = r_mul(sh, g.ihx);
        }
    };
    // state at row j: velocity, scaled shear at its nodes, Tyy and p of the row before
    D2 vx, vy, sx, sy, ty, ps = {{0.0, 0.0}};
    {
        const OpRow r = load(j0 - 1); // vx, vy, eta_n of row j0
        const D2 vxs = ld2(o.vx, g, j0 - 1, c0, ny, cx), vys = ld2(o.vy, g, j0 - 1, c0, ny + 1, cy);
        vx = r.vx;
        vy = r.vy;
        const double vyw = up1(vy.e[1]);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            ty.e[k] = flux_n(SQ ? ax_of(r, k) : ay_of(r, k), vy.e[k], vys.e[k]);
            shear2(r.en.e[k], vx.e[k], vxs.e[k], vy.e[k], k ? vy.e[0] : vyw, sx.e[k], sy.e[k]);
        }
        if (hasp) ps = r.p;
    }
    OpRow cur = load(j0);
    for (int j = j0; j < j1; ++j) {
        OpRow nxt = cur;
        if (j + 1 < j1) nxt = load(j + 1);
        D2 sxn, syn, tyy, txx, dx, dy;
        const double vyw = up1(cur.vy.e[1]), vxe = dn1(vx.e[0]);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            shear2(cur.en.e[k], cur.vx.e[k], vx.e[k], cur.vy.e[k], k ? cur.vy.e[0] : vyw, sxn.e[k], syn.e[k]);
            const double ax = ax_of(cur, k), ay = SQ ? ax : ay_of(cur, k);
            dx.e[k] = r_sub(k ? vxe : vx.e[1], vx.e[k]);
            dy.e[k] = r_sub(cur.vy.e[k], vy.e[k]);
            txx.e[k] = r_mul(ax, dx.e[k]);
            tyy.e[k] = r_mul(ay, dy.e[k]);
        }
        const double txw = up1(txx.e[1]), sye = dn1(sy.e[0]);
        const double pw = hasp ? up1(cur.p.e[1]) : 0.0;
        D2 rx = {{0.0, 0.0}}, ry = {{0.0, 0.0}};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int c = c0 + k;
            const bool ux = j < ny && c >= 1 && c <= nx - 1, uy = j >= 1 && j <= ny - 1 && c >= 0 && c < nx;
            const double mx = m_x(txx.e[k], k ? txx.e[0] : txw, sxn.e[k], sx.e[k]);
            const double my = m_y(k ? sye : sy.e[1], sy.e[k], tyy.e[k], ty.e[k]);
            const double px = hasp ? r_sub(cur.p.e[k], k ? cur.p.e[0] : pw) : 0.0;
            const double py = hasp ? r_sub(cur.p.e[k], ps.e[k]) : 0.0;
            if (MODE == OR_APPLY) {
                if (ux) rx.e[k] = hasp ? r_fma(-px, g.ihx, mx) : mx;
                if (uy) ry.e[k] = hasp ? r_fma(-py, g.ihy, my) : my;
            } else {
                if (ux) rx.e[k] = r_sub(cur.bx.e[k], mx);
                if (uy) ry.e[k] = r_sub(cur.by.e[k], my);
            }
        }
        if (own && c0 >= 0) {
            if (MODE == OR_APPLY) { // every entry of the buffers, zero off the unknowns
                st2(o.ox, g, j, c0, g.pitch, rx);
                st2(o.oy, g, j, c0, g.pitch, ry);
            } else { // the fields' own extents
                if (j < ny) st2(o.ox, g, j, c0, cx, rx);
                st2(o.oy, g, j, c0, cy, ry);
            }
        }
        vx = cur.vx;
        vy = cur.vy;
        sx = sxn;
        sy = syn;
        ty = tyy;
        if (hasp) ps = cur.p;
        cur = nxt;
    }
}

template <int MODE, bool SQ>
__global__ void __launch_bounds__(OR_THREADS, OR_BLOCKS) k_op_rows(const __grid_constant__ OpRows o)
{
    const int warp = (int)threadIdx.x >> 5;
    const int bands = (o.g.ny + o.rows) / o.rows; // of rows 0 .. ny
    for (int t = (int)blockIdx.x * OR_WARPS + warp; t < o.strips * bands; t += (int)gridDim.x * OR_WARPS) {
        const int j0 = t / o.strips * o.rows;
        op_band<MODE, SQ>(o, t % o.strips, j0, min(j0 + o.rows, o.g.ny + 1));
    }
}

// bands of one warp each, as many as one wave holds but at least four rows;
// columns 0 .. cols - 1
template <int MODE>
cudaError_t run(OpRows &o, int cols, cudaStream_t s)
{
    o.strips = (cols + OR_OWN - 1) / OR_OWN;
    const int bands = std::max(1, std::min(152 * OR_BLOCKS * OR_WARPS / o.strips, (o.g.ny + 1 + 3) / 4));
    o.rows = (o.g.ny + 1 + bands - 1) / bands;
    const long long items = (long long)o.strips * ((o.g.ny + o.rows) / o.rows);
    const int nb = (int)std::min<long long>((items + OR_WARPS - 1) / OR_WARPS, 152 * OR_BLOCKS);
    if (o.g.square) k_op_rows<MODE, true><<<nb, OR_THREADS, 0, s>>>(o);
    else k_op_rows<MODE, false><<<nb, OR_THREADS, 0, s>>>(o);
    return cudaGetLastError();
}

} // namespace

bool op_rows_takes(int nx, int ny) { return (long long)nx * ny >= OR_MIN_CELLS; }

cudaError_t op_rows_apply(const GridDesc<double> &g, const double *ec, const double *en, const double *vx,
                          const double *vy, const double *p, double *ox, double *oy, cudaStream_t s)
{
    OpRows o{};
    o.g = g;
    o.ec = ec;
    o.en = en;
    o.vx = vx;
    o.vy = vy;
    o.p = p;
    o.ox = ox;
    o.oy = oy;
    return run<OR_APPLY>(o, g.pitch, s);
}

cudaError_t op_rows_residual(const GridDesc<double> &g, const double *ec, const double *en, const double *bx,
                             const double *by, const double *vx, const double *vy, double *rx, double *ry,
                             cudaStream_t s)
{
    OpRows o{};
    o.g = g;
    o.ec = ec;
    o.en = en;
    o.vx = vx;
    o.vy = vy;
    o.bx = bx;
    o.by = by;
    o.ox = rx;
    o.oy = ry;
    return run<OR_RESID>(o, g.nx + 1, s);
}

} // namespace stokes
