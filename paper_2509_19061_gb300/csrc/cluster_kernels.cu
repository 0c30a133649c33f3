// cluster_kernels.cu -- all sweeps of a small grid's damped Jacobi in one
// launch: Jacobi in any schedule, and RAS schedules that equal it (overlap >=
// k - 1), on the coarse levels of a V-cycle and on small grids.
//
// Such a grid is bound by latency: the tile kernels take a launch for every k
// sweeps (6 to 10 us each for 4 to 8 sweeps of 64^2 to 256^2 cells), and one
// CTA holding a whole level leaves 151 SMs idle (in FP64, whose pipe runs two
// lanes per clock and SM, 4.7 us a sweep at 32^2).  Here a thread-block cluster
// of up to 16 CTAs holds the grid in registers, a band of rows per CTA.  A
// sweep reads its neighbours' values from shared memory and writes the band's
// first and last row into the neighbour CTAs' shared memory (two buffers, by
// sweep parity); one cluster barrier ends it.  The grid is read and written
// once, in place.
//
// Per sweep: the fluxes of every cell (Txx, Tyy, the shear at its node), a
// CTA barrier, the updates, the cluster barrier.  Operations and their order
// are those of stencil.cuh, so the values are those of the other kernels.
//
// Measured, 40 sweeps (tile kernel, 32 x 32 tiles, k = 4, against this one):
// FP64 64^2 415 and 85 us, 32^2 329 and 52; FP32 64^2 66 and 28, 128^2 66 and
// 40.  A sweep costs 0.45 us at the least, most of it the cluster barrier; an FP64
// sweep of 64^2 takes 2.1, of which the FP64 pipes of the 16 SMs take 1.1.
#include <algorithm>
#include <atomic>
#include <mutex>

#include <cooperative_groups.h>

#include "internal.h"
#include "stencil.cuh"

namespace stokes {

namespace {

namespace cg = cooperative_groups;

constexpr int CL_MAX_CTAS = 16;
constexpr int CL_MAX_COLS = 256;
constexpr int CL_MAX_THREADS = 512;
constexpr size_t CL_MAX_SMEM = (size_t)200 * 1024;

template <typename T>
struct ClusterArgs {
    GridDesc<T> g;
    Coeffs<T> c;
    T omega;
    T *vx, *vy;
    int sweeps;
    int band; // rows per CTA
    int cols; // thread columns: nx rounded up to 32
};

// elements of one plane row: columns -1 .. cols
__host__ __device__ constexpr int cl_pitch(int cols) { return cols + 2; }
// Vx, Vy, Txx, Sy, Tyy, Sx of the band, then the rows before and after it: two buffers of vx, vy each
__host__ __device__ constexpr int cl_elems(int cols, int band) { return cl_pitch(cols) * (6 * band + 8); }

// R rows of one column per thread; thread (column, row group)
template <typename T, int R, bool SQ>
__global__ void __launch_bounds__(CL_MAX_THREADS) k_jacobi_cluster(const __grid_constant__ ClusterArgs<T> a)
{
    extern __shared__ __align__(16) unsigned char cl_raw[];
    cg::cluster_group cluster = cg::this_cluster();
    const GridDesc<T> &g = a.g;
    const int nx = g.nx, ny = g.ny, rank = (int)cluster.block_rank(), ranks = (int)cluster.num_blocks();
    const int W = cl_pitch(a.cols), B = a.band;
    T *const sm = reinterpret_cast<T *>(cl_raw) + 1; // column -1 is element -1 of a row
    T *const Vx = sm, *const Vy = sm + B * W, *const Fx = sm + 2 * B * W, *const Fs = sm + 3 * B * W;
    T *const Fy = sm + 4 * B * W, *const Fn = sm + 5 * B * W; // Tyy and Sx, for the row groups above and below
    T *const H = sm + 6 * B * W; // [buffer][0: row before, 1: row after][vx, vy]
    auto halo = [&](int buf, int side, int comp) { return H + ((buf * 2 + side) * 2 + comp) * W; };
    const int j0 = rank * B, nb = max(0, min(B, ny - j0)); // this CTA's rows
    const int i = (int)threadIdx.x % a.cols, rg = (int)threadIdx.x / a.cols;
    const size_t P = (size_t)g.pitch;
    const bool col = i < nx;

    // field value at (j, i), zero outside its rows x columns
    auto at = [&](const T *__restrict__ f, int j, int ii, int rows, int cols) {
        return (j >= 0 && j < rows && ii >= 0 && ii < cols) ? f[(size_t)j * P + (size_t)ii] : T(0);
    };
    // everything to zero first (columns outside the grid, rows after the last)
    for (int e = (int)threadIdx.x; e < cl_elems(a.cols, B); e += (int)blockDim.x) sm[e - 1] = T(0);
    __syncthreads();
    T vx[R], vy[R], ax[R], ay[R], en[R], bx[R], by[R], wx[R], wy[R];
    bool ux[R], uy[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int lr = rg * R + r, j = j0 + lr;
        const bool in = lr < nb && col;
        vx[r] = in ? at(a.vx, j, i, ny, nx + 1) : T(0);
        vy[r] = in ? at(a.vy, j, i, ny + 1, nx) : T(0);
        const T ec = in ? at(a.c.eta_c, j, i, ny, nx) : T(0), e = in ? at(a.c.eta_n, j, i, ny + 1, nx + 1) : T(0);
        ax[r] = coef_x(g, ec);
        ay[r] = coef_y(g, ec);
        en[r] = SQ ? r_mul(e, g.ihx2) : e; // shear_sq takes eta_n / h^2
        bx[r] = in ? a.c.bx[(size_t)j * P + i] : T(0);
        by[r] = in ? a.c.by[(size_t)j * P + i] : T(0);
        ux[r] = in && i >= 1; // i <= nx - 1, j <= ny - 1
        uy[r] = in && j >= 1;
        wx[r] = ux[r] ? jacobi_weight(a.omega, a.c.inv_dx[(size_t)j * P + i]) : T(0);
        wy[r] = uy[r] ? jacobi_weight(a.omega, a.c.inv_dy[(size_t)j * P + i]) : T(0);
        if (in) {
            Vx[lr * W + i] = vx[r];
            Vy[lr * W + i] = vy[r];
            if (i == nx - 1) Vx[lr * W + nx] = at(a.vx, j, nx, ny, nx + 1); // the east wall
        }
    }
    // coefficients of the rows before and after the band, and those rows' first values
    T ay_before = T(0), en_after = T(0);
    if (nb > 0) {
        if (rg == 0) ay_before = coef_y(g, at(a.c.eta_c, j0 - 1, i, ny, nx));
        const T e = at(a.c.eta_n, j0 + nb, i, ny + 1, nx + 1);
        en_after = SQ ? r_mul(e, g.ihx2) : e;
        for (int e2 = (int)threadIdx.x; e2 <= nx; e2 += (int)blockDim.x) {
            halo(0, 0, 0)[e2] = at(a.vx, j0 - 1, e2, ny, nx + 1);
            halo(0, 0, 1)[e2] = at(a.vy, j0 - 1, e2, ny + 1, nx);
            halo(0, 1, 0)[e2] = at(a.vx, j0 + nb, e2, ny, nx + 1);
            halo(0, 1, 1)[e2] = at(a.vy, j0 + nb, e2, ny + 1, nx);
            if (j0 + nb >= ny) { // the wall row after the last band stays
                halo(1, 1, 1)[e2] = at(a.vy, ny, e2, ny + 1, nx);
            }
        }
    }
    // where the neighbours keep this band's first and last row
    const bool lo = rank > 0 && nb > 0, hi = rank + 1 < ranks && j0 + B < ny;
    T *const to_lo = lo ? cluster.map_shared_rank(H, rank - 1) : nullptr;
    T *const to_hi = hi ? cluster.map_shared_rank(H, rank + 1) : nullptr;
    cluster.sync(); // every CTA has read its part of the grid and zeroed its buffers
    auto shear2 = [&](T e, T vxc, T vxs, T vyc, T vyw, T &sx, T &sy) {
        if (SQ) {
            sx = sy = shear_sq(e, vxc, vxs, vyc, vyw);
        } else {
            const T sh = shear(g, e, vxc, vxs, vyc, vyw);
            sx = r_mul(sh, g.ihy);
            sy = r_mul(sh, g.ihx);
        }
    };
    for (int s = 0; s < a.sweeps; ++s) {
        const int buf = s & 1;
        T txx[R], tyy[R], sx[R], sy[R], ty_before = T(0), sx_after = T(0);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int lr = rg * R + r, q = lr * W + i;
            txx[r] = tyy[r] = sx[r] = sy[r] = T(0);
            if (lr < nb && col) {
                const bool first = lr == 0, last = lr == nb - 1;
                const T vxs = first ? halo(buf, 0, 0)[i] : r > 0 ? vx[r > 0 ? r - 1 : 0] : Vx[q - W];
                const T vyn = last ? halo(buf, 1, 1)[i] : r < R - 1 ? vy[r < R - 1 ? r + 1 : r] : Vy[q + W];
                txx[r] = flux_n(ax[r], Vx[q + 1], vx[r]);
                tyy[r] = flux_n(SQ ? ax[r] : ay[r], vyn, vy[r]);
                shear2(en[r], vx[r], vxs, vy[r], Vy[q - 1], sx[r], sy[r]);
                Fx[q] = txx[r];
                Fs[q] = sy[r];
                if (r == R - 1) Fy[q] = tyy[r];
                if (r == 0) Fn[q] = sx[r];
                if (first) ty_before = flux_n(ay_before, vy[r], halo(buf, 0, 1)[i]);
                if (last) {
                    T sya;
                    shear2(en_after, halo(buf, 1, 0)[i], vx[r], vyn, halo(buf, 1, 1)[i - 1], sx_after, sya);
                }
            }
        }
        __syncthreads();
        const bool more = s + 1 < a.sweeps;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int lr = rg * R + r, q = lr * W + i;
            if (lr < nb && col) {
                const bool first = lr == 0, last = lr == nb - 1;
                const T sxn = last ? sx_after : r < R - 1 ? sx[r < R - 1 ? r + 1 : r] : Fn[q + W];
                const T tys = first ? ty_before : r > 0 ? tyy[r > 0 ? r - 1 : 0] : Fy[q - W];
                if (ux[r]) vx[r] = jacobi_update(vx[r], bx[r], m_x(txx[r], Fx[q - 1], sxn, sx[r]), wx[r]);
                if (uy[r]) vy[r] = jacobi_update(vy[r], by[r], m_y(Fs[q + 1], sy[r], tyy[r], tys), wy[r]);
                if (more) {
                    Vx[q] = vx[r];
                    Vy[q] = vy[r];
                    const int nbuf = buf ^ 1;
                    if (first && lo) { // the row after the band below
                        to_lo[((nbuf * 2 + 1) * 2 + 0) * W + i] = vx[r];
                        to_lo[((nbuf * 2 + 1) * 2 + 1) * W + i] = vy[r];
                    }
                    if (last && hi) { // the row before the band above
                        to_hi[((nbuf * 2 + 0) * 2 + 0) * W + i] = vx[r];
                        to_hi[((nbuf * 2 + 0) * 2 + 1) * W + i] = vy[r];
                    }
                }
            }
        }
        if (more) cluster.sync();
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int lr = rg * R + r;
        const size_t q = (size_t)(j0 + lr) * P + i;
        if (ux[r]) a.vx[q] = vx[r];
        if (uy[r]) a.vy[q] = vy[r];
    }
}

template <typename T>
struct ClusterPlan {
    int ctas, band, cols, rows, threads; // rows: per thread
    size_t smem;
};

// `most`: CTAs of the largest cluster
template <typename T>
bool cluster_plan(int nx, int ny, int most, ClusterPlan<T> *p)
{
    if (nx > CL_MAX_COLS || ny < 2) return false;
    // FP64 wants every SM it can get; FP32 CTAs of at least 256 cells, below
    // which the barrier dominates
    const int cells = nx * ny, per = sizeof(T) == 8 ? 32 : 256;
    int c = 1;
    while (c * 2 <= most && c * 2 <= ny / 2 && cells >= c * 2 * per) c *= 2;
    p->ctas = c;
    p->band = (ny + c - 1) / c;
    p->cols = (nx + 31) / 32 * 32;
    p->rows = 1;
    while (p->rows < 8 && p->cols * ((p->band + p->rows - 1) / p->rows) > CL_MAX_THREADS) p->rows *= 2;
    p->threads = p->cols * ((p->band + p->rows - 1) / p->rows);
    p->smem = (size_t)cl_elems(p->cols, p->band) * sizeof(T);
    return p->threads <= CL_MAX_THREADS && p->smem <= CL_MAX_SMEM;
}

template <typename T, int R>
void (*pick_cluster(bool square))(ClusterArgs<T>)
{
    return square ? k_jacobi_cluster<T, R, true> : k_jacobi_cluster<T, R, false>;
}

// CTAs of the largest cluster that the current device runs of the largest CTA
// used here (one an SM, so it does not depend on the kernel): 16 where a GPC
// has that many SMs free for one client, else less; 0 if none.  Asked once per
// device.
int cluster_limit()
{
    static std::atomic<int> known[16]; // limit + 1
    static std::mutex asking; // (a launch of the same kernel sets its attribute after its own call here)
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    const bool cached = dev >= 0 && dev < 16;
    if (cached)
        if (const int k = known[dev].load(std::memory_order_relaxed)) return k - 1;
    std::lock_guard<std::mutex> lock(asking);
    if (cached)
        if (const int k = known[dev].load(std::memory_order_relaxed)) return k - 1;
    const auto kern = k_jacobi_cluster<float, 1, true>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CL_MAX_SMEM);
    cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    int c = CL_MAX_CTAS;
    for (; c > 0; c /= 2) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)c);
        cfg.blockDim = dim3(CL_MAX_THREADS);
        cfg.dynamicSmemBytes = CL_MAX_SMEM;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)c;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess && n > 0) break;
    }
    cudaGetLastError();
    if (cached) known[dev].store(c + 1, std::memory_order_relaxed);
    return c;
}

int most_ctas(const RasRun &run) { return run.max_cluster > 0 ? std::min(run.max_cluster, CL_MAX_CTAS) : cluster_limit(); }

} // namespace

template <typename T>
int cluster_ctas(int nx, int ny, const RasRun &run)
{
    ClusterPlan<T> p;
    return cluster_plan<T>(nx, ny, most_ctas(run), &p) ? p.ctas : 0;
}

template <typename T>
bool cluster_takes(int nx, int ny, int sweeps, const RasRun &run)
{
    // (other options ask for a tile kernel, a negative wait limit for its way out)
    if (!run.allow_tma || run.pair_mode != 1 || run.wait_limit < 0) return false;
    // FP64: a sweep takes cells / 16 x 9 cycles of each SM's pipe (2.1 us at
    // 64^2 in all, 115 us for 40 sweeps of 72 x 64), which soon is more than the
    // tile kernels on all SMs need.  FP32: 40 sweeps of 256^2 take 121 us, 66 on
    // tiles.  Narrow bands of many rows per thread are slower too (18 x 250 in
    // FP64: 141 us, 85 for as many cells in 64 rows).
    if ((long long)nx * ny > (sizeof(T) == 8 ? 4608 : 16384)) return false;
    ClusterPlan<T> p;
    if (sweeps < 2) return false;
    const int most = most_ctas(run); // (no cluster to be had: the tiles)
    return most > 0 && cluster_plan<T>(nx, ny, most, &p);
}

template <typename T>
cudaError_t launch_jacobi_cluster(const GridDesc<T> &g, const Coeffs<T> &c, T omega, int sweeps, T *vx, T *vy,
                                  const RasRun &run, cudaStream_t s)
{
    ClusterPlan<T> p;
    if (!c.inv_dx || !c.inv_dy || !cluster_plan<T>(g.nx, g.ny, most_ctas(run), &p)) return cudaErrorInvalidValue;
    ClusterArgs<T> a;
    a.g = g;
    a.c = c;
    a.omega = omega;
    a.vx = vx;
    a.vy = vy;
    a.sweeps = sweeps;
    a.band = p.band;
    a.cols = p.cols;
    const bool sq = g.square != 0;
    void (*const kern)(ClusterArgs<T>) = p.rows == 1   ? pick_cluster<T, 1>(sq)
                                         : p.rows == 2 ? pick_cluster<T, 2>(sq)
                                         : p.rows == 4 ? pick_cluster<T, 4>(sq)
                                                       : pick_cluster<T, 8>(sq);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem);
    if (e == cudaSuccess && p.ctas > 8) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.ctas);
    cfg.blockDim = dim3((unsigned)p.threads);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)p.ctas;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

template int cluster_ctas<float>(int, int, const RasRun &);
template int cluster_ctas<double>(int, int, const RasRun &);
template bool cluster_takes<float>(int, int, int, const RasRun &);
template bool cluster_takes<double>(int, int, int, const RasRun &);
template cudaError_t launch_jacobi_cluster<float>(const GridDesc<float> &, const Coeffs<float> &, float, int, float *,
                                                  float *, const RasRun &, cudaStream_t);
template cudaError_t launch_jacobi_cluster<double>(const GridDesc<double> &, const Coeffs<double> &, double, int,
                                                   double *, double *, const RasRun &, cudaStream_t);

} // namespace stokes
