// mg_point.cuh -- per-point arithmetic of the multigrid transfer operators,
// shared by the single-instance and the batched kernels.  Prolongation P:
// bilinear in the staggered coordinates, mirror ghosts for the tangential
// direction, zero walls; restriction R = P^T / 4 (gather form).
#pragma once
#include "internal.h"
#include "stencil.cuh"

namespace stokes {

template <typename T>
struct alignas(2 * sizeof(T)) FinePair {
    T e[2];
};

// fine += P coarse at the unknowns of the 2 x 2 fine cells of coarse cell (J, I)
// (both components).  In the cell-centred direction a fine point takes 3/4 of its
// coarse cell and 1/4 of the nearer neighbour, mirrored at the walls; in the
// node-centred one the coinciding point, or half of each side.  The four cells
// share the coarse values (12 loads for 8 points, 24 a point at a time) and the
// fine rows move as pairs, at even columns of an even pitch.  All levels of a
// V-cycle on 4096^2: 79 us, 148 a point at a time.
template <typename T>
__device__ __forceinline__ void prolong_cell(int fp, int ncx, int ncy, int cp, const T *__restrict__ cx,
                                             const T *__restrict__ cy, T *__restrict__ fx, T *__restrict__ fy, int J,
                                             int I)
{
    const T c34 = T(0.75), c14 = T(0.25), c12 = T(0.5);
    const int W = I > 0 ? I - 1 : 0, E = I < ncx - 1 ? I + 1 : I; // mirrored at the walls
    const int S = J > 0 ? J - 1 : 0, N = J < ncy - 1 ? J + 1 : J;
    const size_t c = (size_t)J * cp, q = (size_t)(2 * J) * fp + 2 * I;
    FinePair<T> *const px[2] = {(FinePair<T> *)(fx + q), (FinePair<T> *)(fx + q + fp)};
    FinePair<T> *const py[2] = {(FinePair<T> *)(fy + q), (FinePair<T> *)(fy + q + fp)};
    const FinePair<T> x0 = *px[0], x1 = *px[1], y0 = *py[0], y1 = *py[1];
    // vx: cell-centred in y, node-centred in x
    const T xc[2] = {cx[c + I], cx[c + I + 1]};
    const T xo[2][2] = {{cx[(size_t)S * cp + I], cx[(size_t)S * cp + I + 1]},
                        {cx[(size_t)N * cp + I], cx[(size_t)N * cp + I + 1]}};
    // vy: node-centred in y, cell-centred in x
    const T yc[2][3] = {{cy[c + W], cy[c + I], cy[c + E]}, {cy[c + cp + W], cy[c + cp + I], cy[c + cp + E]}};
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        T s = r_add(T(0), r_mul(c34, xc[0]));
        const T even = r_add(s, r_mul(c14, xo[r][0]));
        s = r_add(T(0), r_mul(r_mul(c34, c12), xc[0]));
        s = r_add(s, r_mul(r_mul(c34, c12), xc[1]));
        s = r_add(s, r_mul(r_mul(c14, c12), xo[r][0]));
        const T odd = r_add(s, r_mul(r_mul(c14, c12), xo[r][1]));
        const FinePair<T> x = r ? x1 : x0;
        const FinePair<T> v = {{r_add(x.e[0], even), r_add(x.e[1], odd)}};
        if (I > 0) *px[r] = v;
        else px[r]->e[1] = v.e[1];
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        if (r == 0 && J == 0) continue; // the wall
        const T w = r ? c12 : T(1);
        FinePair<T> v = r ? y1 : y0;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            T s = r_add(T(0), r_mul(r_mul(w, c34), yc[0][1]));
            s = r_add(s, r_mul(r_mul(w, c14), yc[0][2 * k]));
            if (r) {
                s = r_add(s, r_mul(r_mul(w, c34), yc[1][1]));
                s = r_add(s, r_mul(r_mul(w, c14), yc[1][2 * k]));
            }
            v.e[k] = r_add(v.e[k], s);
        }
        *py[r] = v;
    }
}

// coarse b = P^T r / 4 at coarse point (J, I) (both components; zero off the
// coarse unknowns)
template <typename T>
__device__ __forceinline__ void restrict_point(int nfx, int nfy, int fp, int ncx, int ncy, int cp,
                                               const T *__restrict__ rx, const T *__restrict__ ry,
                                               T *__restrict__ bx, T *__restrict__ by, int J, int I)
{
    const size_t cq = (size_t)J * cp + I;
    const T c34 = T(0.75), c14 = T(0.25), c12 = T(0.5);
    if (J < ncy) { // vx
        T s = T(0);
        if (I >= 1 && I <= ncx - 1) {
            // fine rows (cell-centred in y) and their weights toward coarse row J
            int rows[4];
            T wr[4];
            int nr = 0;
            if (J >= 1) { rows[nr] = 2 * J - 1; wr[nr++] = c14; }
            rows[nr] = 2 * J; wr[nr++] = J == 0 ? T(1) : c34;
            rows[nr] = 2 * J + 1; wr[nr++] = J == ncy - 1 ? T(1) : c34;
            if (J + 1 <= ncy - 1) { rows[nr] = 2 * J + 2; wr[nr++] = c14; }
            for (int a = 0; a < nr; ++a) {
                const T *row = rx + (size_t)rows[a] * fp;
                s = r_add(s, r_mul(r_mul(wr[a], c12), row[2 * I - 1]));
                s = r_add(s, r_mul(wr[a], row[2 * I]));
                s = r_add(s, r_mul(r_mul(wr[a], c12), row[2 * I + 1]));
            }
            s = r_mul(c14, s);
        }
        bx[cq] = s;
    }
    if (I < ncx) { // vy
        T s = T(0);
        if (J >= 1 && J <= ncy - 1) {
            int cols[4];
            T wc[4];
            int nc = 0;
            if (I >= 1) { cols[nc] = 2 * I - 1; wc[nc++] = c14; }
            cols[nc] = 2 * I; wc[nc++] = I == 0 ? T(1) : c34;
            cols[nc] = 2 * I + 1; wc[nc++] = I == ncx - 1 ? T(1) : c34;
            if (I + 1 <= ncx - 1) { cols[nc] = 2 * I + 2; wc[nc++] = c14; }
            const int rows[3] = {2 * J - 1, 2 * J, 2 * J + 1};
            const T wr[3] = {c12, T(1), c12};
            for (int a = 0; a < 3; ++a) {
                const T *row = ry + (size_t)rows[a] * fp;
                for (int b = 0; b < nc; ++b) s = r_add(s, r_mul(r_mul(wr[a], wc[b]), row[cols[b]]));
            }
            s = r_mul(c14, s);
        }
        by[cq] = s;
    }
}

} // namespace stokes
