// gstencil.cuh -- the velocity operator evaluated at one point from global
// memory (used by the global-memory smoothers, the residual, the energy norm
// and the multigrid kernels).  Same arithmetic as stencil.cuh.
#pragma once
#include "internal.h"
#include "stencil.cuh"

namespace stokes {

// (M v)_x and diag(M)_x at vx unknown (j, i), 1 <= i <= nx-1, 0 <= j < ny.
// Rows outside the vx extent (j = -1, j = ny) enter only through a zero
// eta_n and are read as zero.
// MASK: eta_n is the caller's raw array, so boundary nodes are zeroed here
// (the library's own copy already holds zeros there).
template <typename T, bool MASK = false, int SQM = 2>
__device__ __forceinline__ void op_x(const GridDesc<T> &g, const T *__restrict__ eta_c, const T *__restrict__ eta_n,
                                     const T *__restrict__ vx, const T *__restrict__ vy, int j, int i, T &m, T &d,
                                     T &vc)
{
    const size_t P = (size_t)g.pitch;
    const size_t q = (size_t)j * P + (size_t)i;
    vc = vx[q];
    const T vE = vx[q + 1], vW = vx[q - 1];
    const T vN = j + 1 < g.ny ? vx[q + P] : T(0);
    const T vS = j > 0 ? vx[q - P] : T(0);
    const T ecC = eta_c[q], ecW = eta_c[q - 1];
    const T enN = (MASK && j + 1 == g.ny) ? T(0) : eta_n[q + P];
    const T enS = (MASK && j == 0) ? T(0) : eta_n[q];
    const T txx_c = flux_n(coef_x(g, ecC), vE, vc);
    const T txx_w = flux_n(coef_x(g, ecW), vc, vW);
    const T sx_n = shear_x<SQM>(g, enN, vN, vc, vy[q + P], vy[q + P - 1]);
    const T sx_c = shear_x<SQM>(g, enS, vc, vS, vy[q], vy[q - 1]);
    m = m_x(txx_c, txx_w, sx_n, sx_c);
    d = diag_x(g, ecC, ecW, enN, enS);
}

// (M v)_y and diag(M)_y at vy unknown (j, i), 1 <= j <= ny-1, 0 <= i < nx.
template <typename T, bool MASK = false, int SQM = 2>
__device__ __forceinline__ void op_y(const GridDesc<T> &g, const T *__restrict__ eta_c, const T *__restrict__ eta_n,
                                     const T *__restrict__ vx, const T *__restrict__ vy, int j, int i, T &m, T &d,
                                     T &vc)
{
    const size_t P = (size_t)g.pitch;
    const size_t q = (size_t)j * P + (size_t)i;
    vc = vy[q];
    const T vN = vy[q + P], vS = vy[q - P];
    const T vE = i + 1 < g.nx ? vy[q + 1] : T(0);
    const T vW = i > 0 ? vy[q - 1] : T(0);
    const T ecC = eta_c[q], ecS = eta_c[q - P];
    const T enE = (MASK && i + 1 == g.nx) ? T(0) : eta_n[q + 1];
    const T enW = (MASK && i == 0) ? T(0) : eta_n[q];
    const T tyy_c = flux_n(coef_y(g, ecC), vN, vc);
    const T tyy_s = flux_n(coef_y(g, ecS), vc, vS);
    const T sy_e = shear_y<SQM>(g, enE, vx[q + 1], vx[q + 1 - P], vE, vc);
    const T sy_c = shear_y<SQM>(g, enW, vx[q], vx[q - P], vc, vW);
    m = m_y(sy_e, sy_c, tyy_c, tyy_s);
    d = diag_y(g, ecC, ecS, enE, enW);
}

template <typename T>
__device__ __forceinline__ bool vx_unknown(const GridDesc<T> &g, int j, int i)
{
    return j < g.ny && i >= 1 && i <= g.nx - 1;
}
template <typename T>
__device__ __forceinline__ bool vy_unknown(const GridDesc<T> &g, int j, int i)
{
    return i < g.nx && j >= 1 && j <= g.ny - 1;
}
template <typename T>
__device__ __forceinline__ bool vx_wall(const GridDesc<T> &g, int j, int i)
{
    return j < g.ny && (i == 0 || i == g.nx);
}
template <typename T>
__device__ __forceinline__ bool vy_wall(const GridDesc<T> &g, int j, int i)
{
    return i < g.nx && (j == 0 || j == g.ny);
}

// ---- tiled operator apply with shared fluxes --------------------------------
// q = M p on the 32 x 8 cell tile at (i0, j0), plus (<p, q>, <p, r>) over its
// unknowns added to (s0, s1).  Every flux of the tile and a one-cell halo
// (sigma'xx / hx at cells, sigma'yy / hy at cells, the shear at nodes scaled
// by 1/hy and by 1/hx) is computed once into shared memory and M p assembled
// from them: about half the arithmetic of evaluating the stencil per unknown,
// which computes each flux twice.  ax, ay (nullable): the cell coefficients
// 2 eta_c / hx^2 and 2 eta_c / hy^2 precomputed by coef_x / coef_y, which
// saves their evaluation per flux.  The operands and helpers are those of
// op_x / op_y (library eta_n with zero boundary nodes; rows and columns
// outside a field read as zero), so q is the same bit for bit.  Called by all
// 256 threads of the block; tid is the caller's linear thread index (0 .. 255).
constexpr int AT_X = 32, AT_Y = 8;

template <typename T>
struct ApplyTile {
    T txx[AT_Y][AT_X + 1];     // cells (j0 + a, i0 - 1 + b)
    T tyy[AT_Y + 1][AT_X];     // cells (j0 - 1 + a, i0 + b)
    T sx[AT_Y + 1][AT_X + 1];  // nodes (j0 + a, i0 + b): shear / hy
    T sy[AT_Y + 1][AT_X + 1];  // the same nodes: shear / hx
};

// What one thread of a tile reads: the velocity at its cell and next to it, its
// flux coefficients (or eta_c) and eta_n, and h, what its share of the halo reads.
// All of a tile's loads stand under no condition on their values (at the nearest
// entry where one lies outside), so they are in flight together, and a loop over
// tiles issues the next tile's before it uses the current one's fluxes: with a loop
// over each kind of flux and a zero selected at each load, a tile waited six times
// in turn for memory.
template <typename T>
struct TileLoad {
    T vxc, vxe, vxs, vyc, vyn, vyw, cx, cy, e, h[5];
};

// The halo's row of Tyy, row and column of nodes and column of Txx go to one warp
// each (a warp is a row of the tile).
template <typename T>
__device__ __forceinline__ TileLoad<T> tile_load(const GridDesc<T> &g, const T *__restrict__ ec,
                                                 const T *__restrict__ en, const T *__restrict__ ax,
                                                 const T *__restrict__ ay, const T *__restrict__ px,
                                                 const T *__restrict__ py, int i0, int j0, int tid)
{
    const int tx = tid % AT_X, ty = tid / AT_X, j = j0 + ty, i = i0 + tx;
    // the velocity components', cell and node fields' entries nearest to (j, i)
    auto at = [&](int jj, int ii, int rows, int cols) {
        return (size_t)min(max(jj, 0), rows - 1) * g.pitch + (size_t)min(max(ii, 0), cols - 1);
    };
    auto vx_at = [&](int jj, int ii) { return px[at(jj, ii, g.ny, g.nx + 1)]; };
    auto vy_at = [&](int jj, int ii) { return py[at(jj, ii, g.ny + 1, g.nx)]; };
    auto node_at = [&](int jj, int ii) { return en[at(jj, ii, g.ny + 1, g.nx + 1)]; };
    auto cx_at = [&](int jj, int ii) { return (ax ? ax : ec)[at(jj, ii, g.ny, g.nx)]; };
    auto cy_at = [&](int jj, int ii) { return (ax ? ay : ec)[at(jj, ii, g.ny, g.nx)]; };
    TileLoad<T> l;
    l.vxc = vx_at(j, i);
    l.vxe = vx_at(j, i + 1);
    l.vxs = vx_at(j - 1, i);
    l.vyc = vy_at(j, i);
    l.vyn = vy_at(j + 1, i);
    l.vyw = vy_at(j, i - 1);
    l.cx = cx_at(j, i);
    l.cy = g.square ? l.cx : cy_at(j, i); // (square cells: the same number)
    l.e = node_at(j, i);
    if (ty == 0) {
        l.h[0] = cy_at(j0 - 1, i);
        l.h[1] = vy_at(j0 - 1, i);
    } else if (ty == 3) {
        l.h[0] = cx_at(j0 + tx, i0 - 1);
        l.h[1] = vx_at(j0 + tx, i0);
        l.h[2] = vx_at(j0 + tx, i0 - 1);
    } else if (ty <= 2) {
        const int jn = ty == 1 ? j0 + AT_Y : j0 + tx, in = ty == 1 ? i : i0 + AT_X;
        l.h[0] = node_at(jn, in);
        l.h[1] = vx_at(jn, in);
        l.h[2] = vx_at(jn - 1, in);
        l.h[3] = vy_at(jn, in);
        l.h[4] = vy_at(jn, in - 1);
    }
    return l;
}

// The fluxes of the tile at (i0, j0) and its halo into shared memory, ending with
// a barrier; `made`: the loads hold flux coefficients, not eta_c.
template <typename T>
__device__ __forceinline__ void tile_flux(const GridDesc<T> &g, const TileLoad<T> &l, bool made, int i0, int j0,
                                          int tid, ApplyTile<T> &sm)
{
    const int tx = tid % AT_X, ty = tid / AT_X, j = j0 + ty, i = i0 + tx;
    auto is_cell = [&](int jj, int ii) { return jj >= 0 && jj < g.ny && ii >= 0 && ii < g.nx; };
    auto cfx = [&](T c) { return made ? c : coef_x(g, c); };
    auto cfy = [&](T c) { return made ? c : coef_y(g, c); };
    // node (jj, ii) from vx of rows jj, jj - 1 and vy of columns ii, ii - 1, zero outside
    auto node = [&](int jj, int ii, T e, T vxc, T vxs, T vyc, T vyw, int a, int b) {
        T sx = T(0), sy = T(0);
        if (jj <= g.ny && ii <= g.nx)
            shear_xy(g, e, jj < g.ny ? vxc : T(0), jj > 0 ? vxs : T(0), ii < g.nx ? vyc : T(0), ii > 0 ? vyw : T(0),
                     sx, sy);
        sm.sx[a][b] = sx;
        sm.sy[a][b] = sy;
    };
    const bool cell = is_cell(j, i);
    const T kx = cfx(l.cx);
    sm.txx[ty][tx + 1] = cell ? flux_n(kx, l.vxe, l.vxc) : T(0);
    sm.tyy[ty + 1][tx] = cell ? flux_n(g.square ? kx : cfy(l.cy), l.vyn, l.vyc) : T(0);
    node(j, i, l.e, l.vxc, l.vxs, l.vyc, l.vyw, ty, tx);
    if (ty == 0) {
        sm.tyy[0][tx] = is_cell(j0 - 1, i) ? flux_n(cfy(l.h[0]), l.vyc, l.h[1]) : T(0);
    } else if (ty == 3) {
        if (tx < AT_Y) sm.txx[tx][0] = is_cell(j0 + tx, i0 - 1) ? flux_n(cfx(l.h[0]), l.h[1], l.h[2]) : T(0);
    } else if (ty == 1) {
        node(j0 + AT_Y, i, l.h[0], l.h[1], l.h[2], l.h[3], l.h[4], AT_Y, tx);
    } else if (ty == 2 && tx <= AT_Y) {
        node(j0 + tx, i0 + AT_X, l.h[0], l.h[1], l.h[2], l.h[3], l.h[4], tx, AT_X);
    }
    __syncthreads();
}

template <typename T>
__device__ __forceinline__ void flux_tile_stage(const GridDesc<T> &g, const T *__restrict__ ec,
                                                const T *__restrict__ en, const T *__restrict__ ax,
                                                const T *__restrict__ ay, const T *__restrict__ px,
                                                const T *__restrict__ py, int i0, int j0, int tid, ApplyTile<T> &sm)
{
    const TileLoad<T> l = tile_load(g, ec, en, ax, ay, px, py, i0, j0, tid);
    tile_flux(g, l, ax != nullptr, i0, j0, tid, sm);
}

// M v at the tile's cell (ty, tx), from the staged fluxes
template <typename T>
__device__ __forceinline__ T tile_mx(const ApplyTile<T> &sm, int ty, int tx)
{
    return m_x(sm.txx[ty][tx + 1], sm.txx[ty][tx], sm.sx[ty + 1][tx], sm.sx[ty][tx]);
}
template <typename T>
__device__ __forceinline__ T tile_my(const ApplyTile<T> &sm, int ty, int tx)
{
    return m_y(sm.sy[ty][tx + 1], sm.sy[ty][tx], sm.tyy[ty + 1][tx], sm.tyy[ty][tx]);
}

// The entry of cell (j, i), or the last column's or row's nearest to it: every
// field holds it, and an unknown at (j, i) is never moved.
template <typename T>
__device__ __forceinline__ size_t inner_entry(const GridDesc<T> &g, int j, int i)
{
    return (size_t)min(j, g.ny - 1) * g.pitch + min(i, g.nx - 1);
}

// q = M p at the tile's cell of this thread, and its terms of <p, q> and <p, r>
// (p = (pxq, pyq), r = (rxq, ryq) there)
template <typename T>
__device__ __forceinline__ void apply_dot_cell(const GridDesc<T> &g, T pxq, T pyq, T rxq, T ryq, T *__restrict__ qx,
                                               T *__restrict__ qy, int i0, int j0, int tid, const ApplyTile<T> &sm,
                                               double &s0, double &s1)
{
    const int tx = tid % AT_X, ty = tid / AT_X, j = j0 + ty, i = i0 + tx;
    const size_t q = (size_t)j * g.pitch + i;
    if (j < g.ny && i <= g.nx) {
        T m = T(0);
        if (vx_unknown(g, j, i)) {
            m = tile_mx(sm, ty, tx);
            s0 = fma((double)pxq, (double)m, s0);
            s1 = fma((double)pxq, (double)rxq, s1);
        }
        qx[q] = m;
    }
    if (j <= g.ny && i < g.nx) {
        T m = T(0);
        if (vy_unknown(g, j, i)) {
            m = tile_my(sm, ty, tx);
            s0 = fma((double)pyq, (double)m, s0);
            s1 = fma((double)pyq, (double)ryq, s1);
        }
        qy[q] = m;
    }
}

} // namespace stokes
