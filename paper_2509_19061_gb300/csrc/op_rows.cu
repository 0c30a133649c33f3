// op_rows.cu -- the velocity operator by row-marching warps: in FP64 M v + G p
// (stokes_apply_operator) and the residual b - M v of the solves, in either
// precision the residual of a multigrid level with its restriction.
//
// FP64 is bound by its pipe (two lanes per clock and SM), so the layout is the
// one with the fewest operations per cell: a warp owns a strip of 60 columns
// (two per lane; lanes 0 and 31 carry the neighbour columns and own none) and
// marches up a band of rows, each flux is formed once, by the lane and in the
// row it belongs to, and its neighbours' come by shuffles and from the row
// before.  M v takes 16 operations a cell (square cells) and 1/15 for the
// carried columns, a thread per unknown twice the fluxes: M v + G p at 2000^2
// took 487 us and takes 183, the residual at 4096^2 1883 and 641 (0.84 of the
// FP64 pipe).  The next row's loads are issued before the current row's
// arithmetic, which hides them.  (The energy sums in this form measured 345 us
// at 2000^2 with spills and 378 without, against 352 tile by tile, and q = M p
// of the outer CG must keep the order of its inner products, whose last bits
// FP32 sweeps amplify; both stay tile by tile.)
//
// The restriction reads a level's residual at fixed offsets: 2 I of the fine
// columns is a lane's first, and the coarse sums gather their fine rows in
// ascending order, so they accumulate as the march passes and the residual
// never goes to memory.  FP32 is bound by its loads.  All levels of a V-cycle on
// 4096^2: 149 us, 328 as a residual and a restriction a level.
//
// Operations and their order are those of stencil.cuh, so M v has the bits of
// the other kernels.  G p is subtracted by one fused multiply-add, where k_apply
// rounds the product first: M v + G p may differ from it in the last bit.
#include <algorithm>

#include "batch.h"
#include "internal.h"
#include "stencil.cuh"

namespace stokes {

namespace {

constexpr int OR_WARPS = 4, OR_THREADS = OR_WARPS * 32;
constexpr int OR_OWN = 60; // columns of a strip
// Smaller grids leave most SMs idle, where a thread per unknown (twice the
// operations, all in parallel) is sooner done than a warp's rows in turn.
constexpr long long OR_MIN_CELLS = 100000;

template <typename T>
constexpr int OR_BLOCKS = sizeof(T) == 4 ? 6 : 4; // blocks an SM

enum { OR_APPLY, OR_RESID, OR_RESTRICT };

template <typename T>
struct OpRows {
    GridDesc<T> g;
    const T *ec, *en;
    const T *vx, *vy;
    const T *p;       // OR_APPLY: pressure or NULL
    const T *bx, *by; // OR_RESID, OR_RESTRICT
    T *ox, *oy;       // OR_RESTRICT: the coarse right-hand side
    int cp;           // OR_RESTRICT: its pitch
    int strips, rows; // rows of a band (OR_RESTRICT: coarse rows)
};

template <typename T>
__device__ __forceinline__ T up1(T v) { return __shfl_up_sync(0xffffffffu, v, 1); }
template <typename T>
__device__ __forceinline__ T dn1(T v) { return __shfl_down_sync(0xffffffffu, v, 1); }

template <typename T>
struct V2 {
    T e[2];
};
template <typename T>
struct alignas(2 * sizeof(T)) Mem2 {
    T x, y;
};

// Two columns of row j of a field of `rows` rows, at the nearest entry where
// that lies outside.  The load stands under no condition and its value under
// none until it is used, so a row's loads are all in flight together: with a
// zero selected beside each load, the next one waited for it, and a level of
// six rows took 20 us of memory latencies.
template <typename T>
__device__ __forceinline__ V2<T> ld2(const T *__restrict__ f, const GridDesc<T> &g, int j, int c, int rows)
{
    const int jc = min(max(j, 0), rows - 1), cc = min(max(c, 0), (int)g.pitch - 2);
    const Mem2<T> v = *reinterpret_cast<const Mem2<T> *>(f + (size_t)jc * g.pitch + cc);
    return {{v.x, v.y}};
}

// the two columns' entries below `cols`
template <typename T>
__device__ __forceinline__ void st2(T *__restrict__ f, const GridDesc<T> &g, int j, int c, int cols, V2<T> v)
{
    T *const p = f + (size_t)j * g.pitch + c;
    if (c + 1 < cols) *reinterpret_cast<Mem2<T> *>(p) = Mem2<T>{v.e[0], v.e[1]};
    else if (c < cols) p[0] = v.e[0];
}

// what row j reads: vx, vy, eta_n of the row above, the rest of row j
template <typename T>
struct OpRow {
    V2<T> vx, vy, en, ec, bx, by, p;
};

// b = P^T r / 4 of a lane's coarse column I as the fine rows pass: the sums of
// mg_point.cuh's restrict_point, in its order
template <typename T>
struct Restrict {
    T a, n, y; // vx toward the coarse row being finished and the next one, vy
};

// s += w * (fine vx row's columns 2I - 1, 2I, 2I + 1 at 1/2, 1, 1/2)
template <typename T>
__device__ __forceinline__ T add_x(T s, T w, T west, V2<T> r)
{
    s = r_add(s, r_mul(r_mul(w, T(0.5)), west));
    s = r_add(s, r_mul(w, r.e[0]));
    return r_add(s, r_mul(r_mul(w, T(0.5)), r.e[1]));
}

// s += w * (fine vy row's columns 2I - 1 .. 2I + 2 at 1/4, 3/4, 3/4, 1/4, mirrored at the walls)
template <typename T>
__device__ __forceinline__ T add_y(T s, T w, T west, V2<T> r, T east, int I, int ncx)
{
    if (I >= 1) s = r_add(s, r_mul(r_mul(w, T(0.25)), west));
    s = r_add(s, r_mul(r_mul(w, I == 0 ? T(1) : T(0.75)), r.e[0]));
    s = r_add(s, r_mul(r_mul(w, I == ncx - 1 ? T(1) : T(0.75)), r.e[1]));
    if (I + 1 <= ncx - 1) s = r_add(s, r_mul(r_mul(w, T(0.25)), east));
    return s;
}

// fine row j of the band that owns coarse rows J0 .. J1 - 1; zero off the coarse unknowns
template <typename T>
__device__ __forceinline__ void restrict_row(const OpRows<T> &o, Restrict<T> &q, int j, int J0, int J1, int I,
                                             bool own, V2<T> rx, V2<T> ry)
{
    const int ncx = o.g.nx >> 1, ncy = o.g.ny >> 1, J = j >> 1;
    const T wx = up1(rx.e[1]), wy = up1(ry.e[1]), ey = dn1(ry.e[0]);
    const T c34 = T(0.75), c14 = T(0.25);
    auto out_x = [&](int Jc, T s) {
        if (own && Jc >= J0 && Jc < J1 && I <= ncx)
            o.ox[(size_t)Jc * o.cp + I] = I >= 1 && I <= ncx - 1 ? r_mul(c14, s) : T(0);
    };
    auto out_y = [&](int Jc, T s) {
        if (own && Jc >= J0 && Jc < J1 && I < ncx)
            o.oy[(size_t)Jc * o.cp + I] = Jc >= 1 && Jc <= ncy - 1 ? r_mul(c14, s) : T(0);
    };
    if (j & 1) {
        q.a = add_x(q.a, J == ncy - 1 ? T(1) : c34, wx, rx);
        if (J == ncy - 1) out_x(J, q.a);
        q.n = add_x(T(0), c14, wx, rx);
        out_y(J, add_y(q.y, T(0.5), wy, ry, ey, I, ncx));
        q.y = add_y(T(0), T(0.5), wy, ry, ey, I, ncx);
    } else {
        if (J >= 1 && J <= ncy - 1) out_x(J - 1, add_x(q.a, c14, wx, rx));
        q.a = add_x(J == 0 ? T(0) : q.n, J == 0 ? T(1) : c34, wx, rx);
        if (J == ncy) out_y(J, T(0));
        q.y = add_y(q.y, T(1), wy, ry, ey, I, ncx);
    }
}

// rows j0 .. j1 - 1 of a strip (OR_RESTRICT: of the band that owns coarse rows J0 .. J1 - 1)
template <int MODE, bool SQ, typename T>
__device__ __forceinline__ void op_band(const OpRows<T> &o, int strip, int j0, int j1, int J0, int J1)
{
    const GridDesc<T> &g = o.g;
    const int lane = (int)threadIdx.x & 31, c0 = strip * OR_OWN - 2 + 2 * lane;
    const int nx = g.nx, ny = g.ny, cx = nx + 1, cy = nx;
    const bool in0 = c0 >= 0 && c0 < cy, in1 = c0 + 1 >= 0 && c0 + 1 < cy;
    const bool own = lane >= 1 && lane <= 30;
    const bool hasp = MODE == OR_APPLY && o.p;
    auto load = [&](int j) {
        OpRow<T> r;
        r.vx = ld2(o.vx, g, j + 1, c0, ny);
        r.vy = ld2(o.vy, g, j + 1, c0, ny + 1);
        r.en = ld2(o.en, g, j + 1, c0, ny + 1);
        r.ec = ld2(o.ec, g, j, c0, ny);
        if (MODE != OR_APPLY) {
            r.bx = ld2(o.bx, g, j, c0, ny);
            r.by = ld2(o.by, g, j, c0, ny + 1);
        }
        if (hasp) r.p = ld2(o.p, g, j, c0, ny);
        return r;
    };
    // The nodes on the walls (eta_n = 0) read velocities beyond them, which must
    // be numbers: vx of rows -1 and ny, vy of columns -1 and nx.  What else lies
    // outside reaches no unknown.
    auto inside = [&](OpRow<T> &r, int j) {
        if (j + 1 >= ny) r.vx = {{T(0), T(0)}};
        r.vy = {{in0 ? r.vy.e[0] : T(0), in1 ? r.vy.e[1] : T(0)}};
    };
    // coefficients of Txx and Tyy (coef_x, coef_y: doubling eta_c or 1/h^2 is exact) and the scaled shear
    auto ax_of = [&](const OpRow<T> &r, int k) { return r_mul(r.ec.e[k], g.two_ihx2); };
    auto ay_of = [&](const OpRow<T> &r, int k) { return r_mul(r.ec.e[k], g.two_ihy2); };
    auto shear2 = [&](T en, T vxc, T vxs, T vyc, T vyw, T &sx, T &sy) {
        if (SQ) {
            sx = sy = shear_sq(r_mul(en, g.ihx2), vxc, vxs, vyc, vyw);
        } else {
            const T sh = shear(g, en, vxc, vxs, vyc, vyw);
            sx = r_mul(sh, g.ihy);
            sy = r_mul(sh, g.ihx);
        }
    };
    // FP32 levels of a few rows wait for memory only, so row j0 is in flight with
    // the rows before it (the smallest levels: 6.3 us, 5.1 so and with bands of one
    // coarse row); FP64 keeps the registers.
    OpRow<T> cur;
    if (sizeof(T) == 4) cur = load(j0);
    // state at row j: velocity, scaled shear at its nodes, Tyy and p of the row before
    V2<T> vx, vy, sx, sy, ty, ps = {{T(0), T(0)}};
    {
        OpRow<T> r = load(j0 - 1); // vx, vy, eta_n of row j0
        V2<T> vxs = ld2(o.vx, g, j0 - 1, c0, ny), vys = ld2(o.vy, g, j0 - 1, c0, ny + 1);
        inside(r, j0 - 1);
        if (j0 == 0) vxs = {{T(0), T(0)}};
        vx = r.vx;
        vy = r.vy;
        const T vyw = up1(vy.e[1]);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            ty.e[k] = flux_n(SQ ? ax_of(r, k) : ay_of(r, k), vy.e[k], vys.e[k]);
            shear2(r.en.e[k], vx.e[k], vxs.e[k], vy.e[k], k ? vy.e[0] : vyw, sx.e[k], sy.e[k]);
        }
        if (hasp) ps = r.p;
    }
    Restrict<T> acc = {T(0), T(0), T(0)};
    if (sizeof(T) == 8) cur = load(j0);
    for (int j = j0; j < j1; ++j) {
        OpRow<T> nxt = cur;
        if (j + 1 < j1) nxt = load(j + 1);
        inside(cur, j);
        V2<T> sxn, syn, tyy, txx, dx, dy;
        const T vyw = up1(cur.vy.e[1]), vxe = dn1(vx.e[0]);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            shear2(cur.en.e[k], cur.vx.e[k], vx.e[k], cur.vy.e[k], k ? cur.vy.e[0] : vyw, sxn.e[k], syn.e[k]);
            const T ax = ax_of(cur, k), ay = SQ ? ax : ay_of(cur, k);
            dx.e[k] = r_sub(k ? vxe : vx.e[1], vx.e[k]);
            dy.e[k] = r_sub(cur.vy.e[k], vy.e[k]);
            txx.e[k] = r_mul(ax, dx.e[k]);
            tyy.e[k] = r_mul(ay, dy.e[k]);
        }
        const T txw = up1(txx.e[1]), sye = dn1(sy.e[0]);
        const T pw = hasp ? up1(cur.p.e[1]) : T(0);
        V2<T> rx = {{T(0), T(0)}}, ry = {{T(0), T(0)}};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int c = c0 + k;
            const bool ux = j < ny && c >= 1 && c <= nx - 1, uy = j >= 1 && j <= ny - 1 && c >= 0 && c < nx;
            const T mx = m_x(txx.e[k], k ? txx.e[0] : txw, sxn.e[k], sx.e[k]);
            const T my = m_y(k ? sye : sy.e[1], sy.e[k], tyy.e[k], ty.e[k]);
            const T px = hasp ? r_sub(cur.p.e[k], k ? cur.p.e[0] : pw) : T(0);
            const T py = hasp ? r_sub(cur.p.e[k], ps.e[k]) : T(0);
            if (MODE == OR_APPLY) {
                if (ux) rx.e[k] = hasp ? r_fma(-px, g.ihx, mx) : mx;
                if (uy) ry.e[k] = hasp ? r_fma(-py, g.ihy, my) : my;
            } else {
                if (ux) rx.e[k] = r_sub(cur.bx.e[k], mx);
                if (uy) ry.e[k] = r_sub(cur.by.e[k], my);
            }
        }
        if (MODE == OR_RESTRICT) {
            restrict_row(o, acc, j, J0, J1, c0 >> 1, own && c0 >= 0, rx, ry);
        } else if (own && c0 >= 0) {
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

template <int MODE, bool SQ, typename T>
__global__ void __launch_bounds__(OR_THREADS, OR_BLOCKS<T>) k_op_rows(const __grid_constant__ OpRows<T> o)
{
    const int warp = (int)threadIdx.x >> 5, ny = o.g.ny;
    const int nrow = MODE == OR_RESTRICT ? ny / 2 + 1 : ny + 1; // rows 0 .. ny, of the coarse level or this one
    const int bands = (nrow + o.rows - 1) / o.rows;
    for (int t = (int)blockIdx.x * OR_WARPS + warp; t < o.strips * bands; t += (int)gridDim.x * OR_WARPS) {
        const int r0 = t / o.strips * o.rows, r1 = min(r0 + o.rows, nrow);
        if (MODE == OR_RESTRICT) // the fine rows 2 J - 1 .. 2 J + 2 of each
            op_band<MODE, SQ>(o, t % o.strips, max(2 * r0 - 1, 0), min(2 * r1, ny) + 1, r0, r1);
        else op_band<MODE, SQ>(o, t % o.strips, r0, r1, 0, 0);
    }
}

// The residual and its restriction of every instance of a batch, in FP32: 24
// launches over 64 instances of 64^2 to 1024^2 took 1012 us for the residuals, a
// thread per unknown, and 525 for the restrictions, and take 666 here.
static_assert(OR_BATCH_COLS == OR_OWN && OR_BATCH_WARPS == OR_WARPS, "a block's strip and warps");
__global__ void __launch_bounds__(OR_THREADS, OR_BLOCKS<float>)
    k_op_rows_batch(const BLevel<float> *__restrict__ tab, const BSeg *__restrict__ m, int nseg,
                    const int *__restrict__ active)
{
    const BSeg sg = m[seg_of(m, nseg, (int)blockIdx.x)];
    if (active && !active[sg.inst]) return;
    const BLevel<float> &l = tab[sg.inst];
    OpRows<float> o;
    o.g = l.g;
    o.ec = l.ec;
    o.en = l.en;
    o.vx = l.vx;
    o.vy = l.vy;
    o.p = nullptr;
    o.bx = l.bx;
    o.by = l.by;
    o.ox = l.cbx;
    o.oy = l.cby;
    o.cp = l.cp;
    const int lb = (int)blockIdx.x - sg.block_begin, strip = lb % sg.bxb;
    const int r0 = (lb / sg.bxb * OR_WARPS + (int)threadIdx.x / 32) * OR_BATCH_ROWS, nrow = o.g.ny / 2 + 1;
    if (r0 >= nrow) return; // (the whole warp)
    const int r1 = min(r0 + OR_BATCH_ROWS, nrow), j0 = max(2 * r0 - 1, 0), j1 = min(2 * r1, o.g.ny) + 1;
    if (o.g.square) op_band<OR_RESTRICT, true>(o, strip, j0, j1, r0, r1);
    else op_band<OR_RESTRICT, false>(o, strip, j0, j1, r0, r1);
}

// bands of one warp each, as many as one wave holds but at least four rows
// (one coarse row); columns 0 .. cols - 1
template <int MODE, typename T>
cudaError_t run(OpRows<T> &o, int cols, cudaStream_t s)
{
    o.strips = (cols + OR_OWN - 1) / OR_OWN;
    const int nrow = MODE == OR_RESTRICT ? o.g.ny / 2 + 1 : o.g.ny + 1, least = MODE == OR_RESTRICT ? 1 : 4;
    const int bands = std::max(1, std::min(152 * OR_BLOCKS<T> * OR_WARPS / o.strips, (nrow + least - 1) / least));
    o.rows = (nrow + bands - 1) / bands;
    const long long items = (long long)o.strips * ((nrow + o.rows - 1) / o.rows);
    const int nb = (int)std::min<long long>((items + OR_WARPS - 1) / OR_WARPS, 152 * OR_BLOCKS<T>);
    if (o.g.square) k_op_rows<MODE, true, T><<<nb, OR_THREADS, 0, s>>>(o);
    else k_op_rows<MODE, false, T><<<nb, OR_THREADS, 0, s>>>(o);
    return cudaGetLastError();
}

} // namespace

bool op_rows_takes(int nx, int ny) { return (long long)nx * ny >= OR_MIN_CELLS; }

cudaError_t op_rows_apply(const GridDesc<double> &g, const double *ec, const double *en, const double *vx,
                          const double *vy, const double *p, double *ox, double *oy, cudaStream_t s)
{
    OpRows<double> o{};
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
    OpRows<double> o{};
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

template <typename T>
cudaError_t op_rows_restrict(const GridDesc<T> &g, const T *ec, const T *en, const T *bx, const T *by, const T *vx,
                             const T *vy, T *cbx, T *cby, int cpitch, cudaStream_t s)
{
    OpRows<T> o{};
    o.g = g;
    o.ec = ec;
    o.en = en;
    o.vx = vx;
    o.vy = vy;
    o.bx = bx;
    o.by = by;
    o.ox = cbx;
    o.oy = cby;
    o.cp = cpitch;
    return run<OR_RESTRICT>(o, g.nx + 1, s);
}
template cudaError_t op_rows_restrict<float>(const GridDesc<float> &, const float *, const float *, const float *,
                                             const float *, const float *, const float *, float *, float *, int,
                                             cudaStream_t);
template cudaError_t op_rows_restrict<double>(const GridDesc<double> &, const double *, const double *,
                                              const double *, const double *, const double *, const double *,
                                              double *, double *, int, cudaStream_t);

cudaError_t batch_residual_restrict(const BLevel<float> *tab, const BSeg *map, int nseg, int nblocks,
                                    const int *active, cudaStream_t s)
{
    if (nblocks > 0) k_op_rows_batch<<<nblocks, OR_THREADS, 0, s>>>(tab, map, nseg, active);
    return cudaGetLastError();
}

} // namespace stokes
