// mg_kernels.cu -- kernels of the geometric-multigrid V-cycle used for the
// velocity solve of the inexact Uzawa method (Sec. 3.2, configuration in
// Sec. 6.2): coarse viscosity, residual, restriction, prolongation, precision
// casts and the dense FP64 coarsest solve.
//
// Transfer operators (the paper does not state them): bilinear prolongation
// P in the staggered coordinates with mirror ghosts for the tangential
// direction and zero walls; restriction R = P^T / 4.
#include "../../include/stokes.h"
#include "gstencil.cuh"
#include "internal.h"
#include "mg.h"
#include "mg_point.cuh"

namespace stokes {

namespace {

constexpr int BX = 32, BY = 8;
inline dim3 grid2d(int w, int h) { return dim3((unsigned)((w + BX - 1) / BX), (unsigned)((h + BY - 1) / BY)); }

// coarse eta_c = mean of the four children; coarse eta_n at an interior node =
// full-weighting mean of the 3 x 3 fine nodes around the coincident node
// (4 centre, 2 edges, 1 corners, over 16), 0 on boundary nodes.  Injecting
// eta_n would make the coarse operator too soft next to stiff inclusions.
template <typename T>
__global__ void k_coarsen_eta(int ncx, int ncy, int fp, int cp, const T *__restrict__ fec, const T *__restrict__ fen,
                              T *__restrict__ cec, T *__restrict__ cen)
{
    const int I = blockIdx.x * BX + threadIdx.x, J = blockIdx.y * BY + threadIdx.y;
    if (I > ncx || J > ncy) return;
    const size_t cq = (size_t)J * cp + I, f0 = (size_t)(2 * J) * fp + 2 * I;
    if (I < ncx && J < ncy) {
        const T s = r_add(r_add(r_add(fec[f0], fec[f0 + 1]), fec[f0 + fp]), fec[f0 + fp + 1]);
        cec[cq] = r_mul(T(0.25), s);
    }
    T v = T(0);
    if (I >= 1 && I <= ncx - 1 && J >= 1 && J <= ncy - 1) {
        const T centre = fen[f0];
        const T edges = r_add(r_add(r_add(fen[f0 - fp], fen[f0 + fp]), fen[f0 - 1]), fen[f0 + 1]);
        const T corners = r_add(r_add(r_add(fen[f0 - fp - 1], fen[f0 - fp + 1]), fen[f0 + fp - 1]), fen[f0 + fp + 1]);
        v = r_mul(r_add(r_add(r_mul(T(4), centre), r_mul(T(2), edges)), corners), T(0.0625));
    }
    cen[cq] = v;
}

template <typename Ts, typename Td>
__global__ void k_cast(size_t n, const Ts *__restrict__ s, Td *__restrict__ d)
{
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
        d[t] = (Td)s[t];
}

// r = b - M v at unknowns, zero elsewhere (rows up to ny, columns up to nx)
template <typename T>
__global__ void k_residual(GridDesc<T> g, const T *__restrict__ ec, const T *__restrict__ en,
                           const T *__restrict__ bx, const T *__restrict__ by, const T *__restrict__ vx,
                           const T *__restrict__ vy, T *__restrict__ rx, T *__restrict__ ry)
{
    const int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y;
    if (i > g.nx || j > g.ny) return;
    const size_t q = (size_t)j * g.pitch + i;
    T m, d, vc;
    if (j < g.ny) {
        T r = T(0);
        if (vx_unknown(g, j, i)) {
            op_x(g, ec, en, vx, vy, j, i, m, d, vc);
            r = r_sub(bx[q], m);
        }
        rx[q] = r;
    }
    if (i < g.nx) {
        T r = T(0);
        if (vy_unknown(g, j, i)) {
            op_y(g, ec, en, vx, vy, j, i, m, d, vc);
            r = r_sub(by[q], m);
        }
        ry[q] = r;
    }
}

// fine += P coarse at the fine unknowns
template <typename T>
__global__ void __launch_bounds__(BX *BY) k_prolong_add(int fp, int ncx, int ncy, int cp, const T *__restrict__ cx,
                                                        const T *__restrict__ cy, T *__restrict__ fx,
                                                        T *__restrict__ fy)
{
    const int I = blockIdx.x * BX + threadIdx.x, J = blockIdx.y * BY + threadIdx.y;
    if (I < ncx && J < ncy) prolong_cell(fp, ncx, ncy, cp, cx, cy, fx, fy, J, I);
}

// coarse b = P^T r / 4 at the coarse unknowns (gather form), zero elsewhere
template <typename T>
__global__ void k_restrict(int nfx, int nfy, int fp, int ncx, int ncy, int cp, const T *__restrict__ rx,
                           const T *__restrict__ ry, T *__restrict__ bx, T *__restrict__ by)
{
    const int I = blockIdx.x * BX + threadIdx.x, J = blockIdx.y * BY + threadIdx.y;
    if (I > ncx || J > ncy) return;
    restrict_point(nfx, nfy, fp, ncx, ncy, cp, rx, ry, bx, by, J, I);
}

// ---- dense coarsest solve --------------------------------------------------
// Unknown numbering: vx unknowns row-major (j, i = 1..nx-1), then vy unknowns
// row-major (j = 1..ny-1, i).
__device__ __forceinline__ void unknown_pos(int u, int nx, int ny, int &comp, int &j, int &i)
{
    const int nvx = ny * (nx - 1);
    if (u < nvx) {
        comp = 0;
        j = u / (nx - 1);
        i = u - j * (nx - 1) + 1;
    } else {
        u -= nvx;
        comp = 1;
        j = u / nx + 1;
        i = u - (j - 1) * nx;
    }
}

// A[r][c] = -(M e_c)_r in FP64 from the level's viscosity (boundary nodes of
// eta_n hold zero)
// (one job per blockIdx.y)
template <typename T>
__global__ void k_assemble(const DenseJob *__restrict__ jobs)
{
    const DenseJob &jb = jobs[blockIdx.y];
    const int nx = jb.nx, ny = jb.ny, pitch = jb.pitch, n = jb.n;
    const double ihx = jb.ihx, ihy = jb.ihy;
    const T *__restrict__ ec = (const T *)jb.ec;
    const T *__restrict__ en = (const T *)jb.en;
    double *__restrict__ A = jb.A;
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long)n * n) return;
    const int r = (int)(t / n), c = (int)(t - (long)r * n);
    int rc, rj, ri, cc, cj, ci;
    unknown_pos(r, nx, ny, rc, rj, ri);
    unknown_pos(c, nx, ny, cc, cj, ci);
    // value of the unit vector e_c at (component, j, i)
    auto ux = [&](int j, int i) { return (cc == 0 && cj == j && ci == i) ? 1.0 : 0.0; };
    auto uy = [&](int j, int i) { return (cc == 1 && cj == j && ci == i) ? 1.0 : 0.0; };
    auto EC = [&](int j, int i) { return (double)ec[(size_t)j * pitch + i]; };
    auto EN = [&](int j, int i) { return (double)en[(size_t)j * pitch + i]; };
    double m;
    if (rc == 0) {
        const int j = rj, i = ri;
        const double txe = 2.0 * EC(j, i) * (ux(j, i + 1) - ux(j, i)) * ihx;
        const double txw = 2.0 * EC(j, i - 1) * (ux(j, i) - ux(j, i - 1)) * ihx;
        const double sn = EN(j + 1, i) * ((ux(j + 1, i) - ux(j, i)) * ihy + (uy(j + 1, i) - uy(j + 1, i - 1)) * ihx);
        const double ss = EN(j, i) * ((ux(j, i) - ux(j - 1, i)) * ihy + (uy(j, i) - uy(j, i - 1)) * ihx);
        m = (txe - txw) * ihx + (sn - ss) * ihy;
    } else {
        const int j = rj, i = ri;
        const double tyn = 2.0 * EC(j, i) * (uy(j + 1, i) - uy(j, i)) * ihy;
        const double tys = 2.0 * EC(j - 1, i) * (uy(j, i) - uy(j - 1, i)) * ihy;
        const double se = EN(j, i + 1) * ((ux(j, i + 1) - ux(j - 1, i + 1)) * ihy + (uy(j, i + 1) - uy(j, i)) * ihx);
        const double sw = EN(j, i) * ((ux(j, i) - ux(j - 1, i)) * ihy + (uy(j, i) - uy(j, i - 1)) * ihx);
        m = (se - sw) * ihx + (tyn - tys) * ihy;
    }
    A[(size_t)r * n + c] = -m;
}

// The dense factorisation -M = L L^T, W = L^{-1}, (-M)^{-1} = W^T W of one
// coarsest level (n <= 1024) is bound by the FP64 pipe's latency and rate (two
// FP64 lanes per clock and SM) and by its chain of n square roots and
// divisions, not by bytes (n^2 doubles stay in L2).  One CTA per matrix kept
// one SM's FP64 pipe for the whole n^3 / 6: 12.4 ms for L and 12.5 ms for W at
// n = 480.  Blocked by 32 columns the work spreads over the SMs and only the
// chain stays serial: 0.71 and 0.43 ms (and 0.065 for W^T W, from 0.157).  Every
// entry is still formed by the same operations in
// the same order (its updates in ascending k, then its division), so the
// factors have the bits of the unblocked algorithm.
constexpr int DN_B = 32;  // block columns
constexpr int DN_ER = 16; // rows below the diagonal block per panel CTA

// Panel kb: the diagonal block's factor (formed by every CTA, from the
// trailing matrix in A) and DN_ER rows of the block column below it, into the
// lower triangle of `L` (the job's Ainv buffer, free until k_gram).  The
// diagonal block and the CTA's rows go through the columns together.  What
// bounds it is the chain of one update, a square root and a division per
// column, so two warps run that and nothing else, and the other six bring the
// column before into the columns after it meanwhile: 40 us a panel, 50 with
// all warps in each phase in turn.  `status` is set to 1 if a pivot is not
// positive.  Grid: (row groups, jobs).
__global__ void __launch_bounds__(256) k_chol_panel(const DenseJob *__restrict__ jobs, int kb)
{
    const DenseJob &jb = jobs[blockIdx.y];
    const int n = jb.n, k0 = kb * DN_B;
    if (k0 >= n) return;
    const int r0 = k0 + DN_B + (int)blockIdx.x * DN_ER; // first row of this CTA below the block
    if (blockIdx.x > 0 && r0 >= n) return;
    const double *__restrict__ A = jb.A;
    double *__restrict__ L = jb.Ainv;
    constexpr int ROWS = DN_B + DN_ER;
    __shared__ double P[ROWS][DN_B + 1]; // the trailing columns; rows 0..31: the diagonal block
    __shared__ double F[ROWS][DN_B + 1]; // the finished columns
    __shared__ int bad;
    const int nb = min(DN_B, n - k0), tid = (int)threadIdx.x, lane = tid & 31, w = tid >> 5;
    auto row_of = [&](int q) { return q < DN_B ? k0 + q : r0 + (q - DN_B); };
    for (int e = tid; e < ROWS * DN_B; e += 256) {
        const int q = e / DN_B, c = e % DN_B, i = row_of(q);
        P[q][c] = (i < n && c < nb && (q >= DN_B || c <= q)) ? A[(size_t)i * n + k0 + c] : 0.0;
    }
    if (tid == 0) bad = 0;
    const int rows = r0 < n ? DN_B + min(DN_ER, n - r0) : DN_B;
    __syncthreads();
    for (int k = 0; k < nb; ++k) {
        if (w < 2) { // one thread per row of column k: its last update, the square root, the division
            if (tid < rows && tid >= k) {
                double d = P[k][k], x = P[tid][k];
                if (k > 0) {
                    const double l = F[k][k - 1];
                    d = fma(-l, l, d);
                    x = fma(-F[tid][k - 1], l, x);
                }
                if (tid == k && !(d > 0.0)) bad = 1;
                const double piv = d > 0.0 ? sqrt(d) : 1.0;
                F[tid][k] = tid == k ? piv : x / piv;
            }
        } else if (k > 0) { // column k - 1 into the columns after k
            for (int c = k + 1 + w - 2; c < nb; c += 6)
                if (lane >= c) P[lane][c] = fma(-F[lane][k - 1], F[c][k - 1], P[lane][c]);
            const int q = DN_B + lane % DN_ER;
            for (int c = k + 1 + 2 * (w - 2) + lane / DN_ER; c < nb; c += 12)
                P[q][c] = fma(-F[q][k - 1], F[c][k - 1], P[q][c]);
        }
        __syncthreads();
    }
    const int q0 = blockIdx.x == 0 ? 0 : DN_B;
    for (int e = tid + q0 * DN_B; e < rows * DN_B; e += 256) {
        const int q = e / DN_B, c = e % DN_B, i = row_of(q);
        if (i < n && c < nb && (q >= DN_B || c <= q)) L[(size_t)i * n + k0 + c] = F[q][c];
    }
    if (bad && tid == 0 && blockIdx.x == 0) *jb.status = 1;
}

// Trailing update of panel kb: A[i][j] -= sum_k L[i][k] L[j][k] over the
// panel's columns in ascending k, one 16 x 16 tile of the lower triangle per
// CTA (one entry per thread; 16 x 16 keeps all SMs busy until the trailing
// matrix is small).  Grid: (tiles of the largest trailing triangle, jobs).
__global__ void __launch_bounds__(256) k_chol_update(const DenseJob *__restrict__ jobs, int kb)
{
    const DenseJob &jb = jobs[blockIdx.y];
    const int n = jb.n, k0 = kb * DN_B, t0 = k0 + DN_B;
    if (t0 >= n) return;
    const double *__restrict__ L = jb.Ainv;
    double *__restrict__ A = jb.A;
    // tile (I, J), J <= I, of the lower triangle numbered row by row
    const int b = (int)blockIdx.x;
    int I = (int)((sqrtf(8.f * (float)b + 1.f) - 1.f) * 0.5f);
    while ((I + 1) * (I + 2) / 2 <= b) ++I;
    while (I * (I + 1) / 2 > b) --I;
    const int J = b - I * (I + 1) / 2;
    const int i0 = t0 + 16 * I, j0 = t0 + 16 * J;
    if (i0 >= n) return;
    __shared__ double Li[16][DN_B + 1], Lj[16][DN_B + 1];
    const int tid = (int)threadIdx.x;
    for (int e = tid; e < 16 * DN_B; e += 256) {
        const int q = e / DN_B, c = e % DN_B;
        Li[q][c] = i0 + q < n ? L[(size_t)(i0 + q) * n + k0 + c] : 0.0;
        Lj[q][c] = j0 + q < n ? L[(size_t)(j0 + q) * n + k0 + c] : 0.0;
    }
    __syncthreads();
    const int i = i0 + tid / 16, j = j0 + tid % 16;
    if (i >= n || j > i) return;
    double a = A[(size_t)i * n + j];
#pragma unroll 8
    for (int c = 0; c < DN_B; ++c) a = fma(-Li[tid / 16][c], Lj[tid % 16][c], a);
    A[(size_t)i * n + j] = a;
}

// W = L^{-1} (lower triangle; zero above), C columns per CTA, one thread per
// (row of the current 32-row block, column): the block's sums over the rows
// above it from 32 x 32 tiles of L (ascending m), then the block's forward
// substitution.  The columns' finished part stays in shared memory.  C = 4
// spreads one matrix over n / 4 CTAs (chain-bound); C = 16 uses the lanes of
// the divisions better and is for many matrices at once (FP64-rate-bound).
// Grid: (column groups, jobs); dynamic shared memory n_max x C doubles.
template <int C>
__global__ void __launch_bounds__(DN_B *C) k_tri_inverse(const DenseJob *__restrict__ jobs)
{
    extern __shared__ __align__(16) double Wc[]; // [row][C]
    const DenseJob &jb = jobs[blockIdx.y];
    const int n = jb.n, c0 = (int)blockIdx.x * C;
    if (c0 >= n) return;
    const double *__restrict__ L = jb.Ainv;
    double *__restrict__ W = jb.W;
    __shared__ double T[DN_B][DN_B + 1];
    const int tid = (int)threadIdx.x, r = tid / C, q = tid % C, c = c0 + q;
    const int b0 = c0 / DN_B, nblk = (n + DN_B - 1) / DN_B;
    auto load_tile = [&](int I, int K) { // rows of block I, columns of block K, zero outside the triangle
        for (int e = tid; e < DN_B * DN_B; e += DN_B * C) {
            const int i = I * DN_B + e / DN_B, m = K * DN_B + e % DN_B;
            T[e / DN_B][e % DN_B] = (i < n && m <= i) ? L[(size_t)i * n + m] : 0.0;
        }
    };
    if (c < n)
        for (int i = r; i < b0 * DN_B; i += DN_B) W[(size_t)i * n + c] = 0.0;
    for (int I = b0; I < nblk; ++I) {
        double s = 0.0;
        for (int K = b0; K < I; ++K) {
            __syncthreads();
            load_tile(I, K);
            __syncthreads();
            const double *wk = Wc + (size_t)K * DN_B * C + q;
#pragma unroll 4
            for (int m = 0; m < DN_B; ++m) s = fma(T[r][m], wk[m * C], s);
        }
        __syncthreads();
        load_tile(I, I);
        __syncthreads();
        const int i0 = I * DN_B, nr = min(DN_B, n - i0);
        for (int t = 0; t < nr; ++t) {
            if (r == t) {
                const int i = i0 + t;
                double w = 0.0;
                if (c < n && i == c) w = 1.0 / T[t][t];
                else if (c < n && i > c) w = -s / T[t][t];
                Wc[(size_t)i * C + q] = w;
                if (c < n) W[(size_t)i * n + c] = w;
            }
            __syncthreads();
            if (r > t && i0 + t >= c) s = fma(T[r][t], Wc[(size_t)(i0 + t) * C + q], s);
        }
    }
}

// Ainv = W^T W, one 16 x 16 tile of the lower triangle per CTA (an entry per
// thread, ascending m from the tile's first row) stored to both triangles
// (the products commute, so the mirrored entry has the same bits).  Grid:
// (tiles of the largest triangle, jobs).
__global__ void __launch_bounds__(256) k_gram(const DenseJob *__restrict__ jobs)
{
    const DenseJob &jb = jobs[blockIdx.y];
    const int n = jb.n;
    const double *__restrict__ W = jb.W;
    double *__restrict__ Ainv = jb.Ainv;
    const int b = (int)blockIdx.x;
    int I = (int)((sqrtf(8.f * (float)b + 1.f) - 1.f) * 0.5f);
    while ((I + 1) * (I + 2) / 2 <= b) ++I;
    while (I * (I + 1) / 2 > b) --I;
    const int J = b - I * (I + 1) / 2;
    const int i0 = 16 * I, j0 = 16 * J;
    if (i0 >= n) return;
    __shared__ double Wi[DN_B][16], Wj[DN_B][16];
    const int tid = (int)threadIdx.x, ti = tid / 16, tj = tid % 16;
    double s = 0.0;
    for (int m0 = i0; m0 < n; m0 += DN_B) { // W[m][i] = 0 for m < i, and j <= i
        __syncthreads();
        for (int e = tid; e < DN_B * 16; e += 256) {
            const int m = m0 + e / 16, q = e % 16;
            Wi[e / 16][q] = (m < n && i0 + q < n) ? W[(size_t)m * n + i0 + q] : 0.0;
            Wj[e / 16][q] = (m < n && j0 + q < n) ? W[(size_t)m * n + j0 + q] : 0.0;
        }
        __syncthreads();
#pragma unroll 8
        for (int m = 0; m < DN_B; ++m) s = fma(Wi[m][ti], Wj[m][tj], s);
    }
    const int i = i0 + ti, j = j0 + tj;
    if (i >= n || j > i) return;
    Ainv[(size_t)i * n + j] = s;
    Ainv[(size_t)j * n + i] = s;
}

// x = -Ainv b (solution of M x = b) from and to the level's fields, one warp per
// row of the matrix; every CTA gathers b itself, which saves the launches that
// packed b and unpacked x (12 us in three, 5.3 in one, at 480 unknowns).
constexpr int DS_THREADS = 256, DS_MAX = 1024; // (the largest coarsest level)
template <typename T>
__global__ void __launch_bounds__(DS_THREADS) k_dense_solve(int nx, int ny, int pitch, int n,
                                                            const double *__restrict__ Ainv,
                                                            const T *__restrict__ bx, const T *__restrict__ by,
                                                            T *__restrict__ vx, T *__restrict__ vy)
{
    __shared__ double b[DS_MAX];
    const int row = blockIdx.x * (DS_THREADS / 32) + threadIdx.x / 32, lane = threadIdx.x & 31;
    const double *const A = Ainv + (size_t)min(row, n - 1) * n;
    constexpr int AHEAD = 16; // of a lane's entries, in flight while b is gathered
    double a[AHEAD];
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) a[k] = A[min(lane + 32 * k, n - 1)];
    int comp, j, i;
    for (int u = (int)threadIdx.x; u < n; u += DS_THREADS) {
        unknown_pos(u, nx, ny, comp, j, i);
        b[u] = (double)(comp == 0 ? bx : by)[(size_t)j * pitch + i];
    }
    __syncthreads();
    if (row >= n) return;
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < AHEAD; ++k)
        if (lane + 32 * k < n) s += a[k] * b[lane + 32 * k];
    for (int c = lane + 32 * AHEAD; c < n; c += 32) s += A[c] * b[c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane > 0) return;
    unknown_pos(row, nx, ny, comp, j, i);
    (comp == 0 ? vx : vy)[(size_t)j * pitch + i] = (T)-s;
}

} // namespace

// ---------------------------------------------------------------------------
template <typename T>
cudaError_t mg_coarsen_eta(const MgLevel &f, const MgLevel &c, cudaStream_t s)
{
    k_coarsen_eta<T><<<grid2d(c.nx + 1, c.ny + 1), dim3(BX, BY), 0, s>>>(
        c.nx, c.ny, f.pitch, c.pitch, (const T *)f.ec, (const T *)f.en, (T *)c.ec, (T *)c.en);
    return cudaGetLastError();
}

template <typename Ts, typename Td>
cudaError_t mg_cast(size_t n, const void *src, void *dst, cudaStream_t s)
{
    k_cast<Ts, Td><<<1216, 256, 0, s>>>(n, (const Ts *)src, (Td *)dst);
    return cudaGetLastError();
}

template <typename T>
cudaError_t mg_residual(const MgLevel &l, cudaStream_t s)
{
    const GridDesc<T> g = make_grid<T>(l.nx, l.ny, l.pitch, l.hx, l.hy);
    if constexpr (sizeof(T) == 8)
        if (op_rows_takes(l.nx, l.ny))
            return op_rows_residual(g, (const T *)l.ec, (const T *)l.en, (const T *)l.bx, (const T *)l.by,
                                    (const T *)l.vx, (const T *)l.vy, (T *)l.rx, (T *)l.ry, s);
    k_residual<T><<<grid2d(l.nx + 1, l.ny + 1), dim3(BX, BY), 0, s>>>(g, (const T *)l.ec, (const T *)l.en,
                                                                       (const T *)l.bx, (const T *)l.by,
                                                                       (const T *)l.vx, (const T *)l.vy, (T *)l.rx,
                                                                       (T *)l.ry);
    return cudaGetLastError();
}

template <typename T>
cudaError_t mg_residual_restrict(const MgLevel &f, const MgLevel &c, cudaStream_t s)
{
    if (mg_restrict_fused<T>(f.nx, f.ny))
        return op_rows_restrict(make_grid<T>(f.nx, f.ny, f.pitch, f.hx, f.hy), (const T *)f.ec, (const T *)f.en,
                                (const T *)f.bx, (const T *)f.by, (const T *)f.vx, (const T *)f.vy, (T *)c.bx,
                                (T *)c.by, c.pitch, s);
    if constexpr (sizeof(T) == 8) {
        const cudaError_t e = mg_residual<T>(f, s);
        if (e != cudaSuccess) return e;
        k_restrict<T><<<grid2d(c.nx + 1, c.ny + 1), dim3(BX, BY), 0, s>>>(f.nx, f.ny, f.pitch, c.nx, c.ny, c.pitch,
                                                                           (const T *)f.rx, (const T *)f.ry, (T *)c.bx,
                                                                           (T *)c.by);
        return cudaGetLastError();
    } else {
        return cudaErrorInvalidValue; // (FP32 levels always take the fused form)
    }
}

template <typename T>
cudaError_t mg_prolong_add(const MgLevel &f, const MgLevel &c, cudaStream_t s)
{
    k_prolong_add<T><<<grid2d(c.nx, c.ny), dim3(BX, BY), 0, s>>>(f.pitch, c.nx, c.ny, c.pitch, (const T *)c.vx,
                                                                 (const T *)c.vy, (T *)f.vx, (T *)f.vy);
    return cudaGetLastError();
}

template <typename T>
cudaError_t mg_dense_setup_many(const DenseJob *jobs, int count, int nmax, cudaStream_t s)
{
    const long nn = (long)nmax * nmax;
    const int nblk = (nmax + DN_B - 1) / DN_B;
    auto tiles16 = [](int rows) { const int t = (rows + 15) / 16; return (unsigned)(t * (t + 1) / 2); };
    // four columns per CTA while that leaves at most four CTAs an SM (480
    // unknowns: 120 CTAs a matrix), where the chain bounds it; sixteen beyond,
    // where the FP64 rate does and a division wants full warps
    const bool many = (long)count * ((nmax + 3) / 4) > 4L * 152;
    const int cols = many ? 16 : 4;
    const size_t wsm = (size_t)nblk * DN_B * cols * sizeof(double);
    cudaError_t e = cudaFuncSetAttribute(many ? k_tri_inverse<16> : k_tri_inverse<4>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wsm);
    if (e != cudaSuccess) return e;
    for (int j0 = 0; j0 < count; j0 += 65535) {
        const int c = count - j0 < 65535 ? count - j0 : 65535;
        const DenseJob *jb = jobs + j0;
        k_assemble<T><<<dim3((unsigned)((nn + 255) / 256), c), 256, 0, s>>>(jb);
        for (int kb = 0; kb < nblk; ++kb) {
            const int below = nmax - (kb + 1) * DN_B; // rows below the diagonal block
            k_chol_panel<<<dim3((unsigned)(below > 0 ? (below + DN_ER - 1) / DN_ER : 1), c), 256, 0, s>>>(jb, kb);
            if (below > 0) k_chol_update<<<dim3(tiles16(below), c), 256, 0, s>>>(jb, kb);
        }
        const dim3 gi((unsigned)((nmax + cols - 1) / cols), c);
        if (many) k_tri_inverse<16><<<gi, DN_B * 16, wsm, s>>>(jb);
        else k_tri_inverse<4><<<gi, DN_B * 4, wsm, s>>>(jb);
        k_gram<<<dim3(tiles16(nmax), c), 256, 0, s>>>(jb);
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t mg_dense_setup(const MgLevel &l, int n, double *A, double *W, double *Ainv, int *status,
                           cudaStream_t s)
{
    DenseJob h;
    h.nx = l.nx;
    h.ny = l.ny;
    h.pitch = l.pitch;
    h.n = n;
    h.ihx = 1.0 / l.hx;
    h.ihy = 1.0 / l.hy;
    h.ec = l.ec;
    h.en = l.en;
    h.A = A;
    h.W = W;
    h.Ainv = Ainv;
    h.status = status;
    // a one-entry job table in stream-ordered memory, freed after the kernels
    DenseJob *d = nullptr;
    cudaError_t e = cudaMallocAsync((void **)&d, sizeof(DenseJob), s);
    if (e != cudaSuccess) return e;
    e = cudaMemcpyAsync(d, &h, sizeof(DenseJob), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = mg_dense_setup_many<T>(d, 1, n, s);
    const cudaError_t e2 = cudaStreamSynchronize(s);
    cudaFreeAsync(d, s);
    return e != cudaSuccess ? e : e2;
}

template <typename T>
cudaError_t mg_dense_solve(const MgLevel &l, int n, const double *Ainv, cudaStream_t s)
{
    if (n > DS_MAX) return cudaErrorInvalidValue;
    k_dense_solve<T><<<(n + DS_THREADS / 32 - 1) / (DS_THREADS / 32), DS_THREADS, 0, s>>>(
        l.nx, l.ny, l.pitch, n, Ainv, (const T *)l.bx, (const T *)l.by, (T *)l.vx, (T *)l.vy);
    return cudaGetLastError();
}

#define INST(T)                                                                                                    \
    template cudaError_t mg_coarsen_eta<T>(const MgLevel &, const MgLevel &, cudaStream_t);                        \
    template cudaError_t mg_residual<T>(const MgLevel &, cudaStream_t);                                            \
    template cudaError_t mg_residual_restrict<T>(const MgLevel &, const MgLevel &, cudaStream_t);                  \
    template cudaError_t mg_prolong_add<T>(const MgLevel &, const MgLevel &, cudaStream_t);                        \
    template cudaError_t mg_dense_setup<T>(const MgLevel &, int, double *, double *, double *, int *,              \
                                           cudaStream_t);                                                          \
    template cudaError_t mg_dense_setup_many<T>(const DenseJob *, int, int, cudaStream_t);                         \
    template cudaError_t mg_dense_solve<T>(const MgLevel &, int, const double *, cudaStream_t);
INST(float)
INST(double)
#undef INST
template cudaError_t mg_cast<double, float>(size_t, const void *, void *, cudaStream_t);
template cudaError_t mg_cast<float, double>(size_t, const void *, void *, cudaStream_t);
template cudaError_t mg_cast<double, double>(size_t, const void *, void *, cudaStream_t);
template cudaError_t mg_cast<float, float>(size_t, const void *, void *, cudaStream_t);

} // namespace stokes
