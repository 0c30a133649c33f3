// smooth.cu -- schedules of the five smoothers of Sec. 5 over the kernels:
// sweep loops, RAS outer iterations with their tile shifts (Algorithm 2),
// and the ping-pong between the caller's velocity and a scratch pair.
#include "../../include/stokes.h"
#include "internal.h"

namespace stokes {

namespace {

// global Jacobi in any traversal: fused Jacobi, and RAS with overlap >= k - 1
bool any_traversal(const SmoothSpec &p)
{
    return (p.variant == STOKES_RAS && p.overlap >= p.k - 1) || p.variant == STOKES_JACOBI_FUSED;
}

// passes of a row-streaming kernel for this smoothing, 0 if none takes it: red-
// black Gauss-Seidel's own; else a RAS schedule with overlap >= k - 1 is global
// Jacobi in any traversal, and fused Jacobi's sweeps need not each cross the
// grid before the next begins (20 sweeps of 4001 x 2999: 408 us, 1822 us as 20
// passes of k_jacobi_rows).  Separate-pass and blocked Jacobi keep their passes.
// A strip sweeps 128 (FP64: 64) columns however few the grid has, where a tile's
// window narrows with it: RAS on narrower grids keeps its tiles (24 FP32 sweeps
// of 12 x 66666 198 us, 219 streamed, of 20 x 40000 351 and 150; eight FP64
// sweeps of 24 x 33333 673 and 783, of 32 x 25000 918 and 596).  Fused Jacobi
// streams at any width (FP64, 5 x 60000: 2292 us as passes, 1423).
constexpr int STREAM_MIN_NX32 = 20, STREAM_MIN_NX64 = 32;
template <typename T>
int stream_passes_of(int nx, int ny, const SmoothSpec &p, const RasRun &run)
{
    if constexpr (sizeof(T) == 4)
        if (p.variant == STOKES_RBGS) return rbgs_stream_passes(nx, ny, p.sweeps, run);
    if (!any_traversal(p)) return 0;
    if (p.variant == STOKES_RAS && nx < (sizeof(T) == 4 ? STREAM_MIN_NX32 : STREAM_MIN_NX64)) return 0;
    if constexpr (sizeof(T) == 4) return stream_passes((long long)nx * ny, p.sweeps, run);
    else return stream64_passes(nx, ny, p.sweeps, run);
}

// The tiles of an FP32 RAS schedule that equals global Jacobi, on grids between
// the cluster's and the row streaming's: the given tiles, shifts and k change no
// value there, so they are chosen for this GPU.  Windows are 64 columns wide (two
// per lane of the pair kernel) and of 5 rows a warp, a pass runs up to eight
// sweeps, split evenly, on tiles cut at zero.  Such a grid has few tiles and a
// launch takes the time of one times the waves: about 32 rows' worth of setup and
// the window's rows (8.9 us with 50 rows and eight sweeps, 11.4 with 80; 32 x 32
// tiles with k = 4 6.5 for four), so the window height with the least product is
// taken.  With the middle levels' tiles as given: 512^2 Uzawa (32 x 32, k = 4)
// 25.0 ms, now 24.1; 8 CG cycles of 1024^2 (48 x 32, k = 8) 7.28 and 7.11.
// Given tiles that run the sweeps in one pass of one wave stay where their
// windows are narrower still, up to 48 columns (one a thread), and the sweeps
// at most four (four sweeps of 200^2 on 32 x 32 tiles 14.4 us, 16.5 on chosen
// ones; at 500^2, two waves, 18.5 and 16.5).
constexpr long long FREE_MAX_CELLS = 600000; // where the row streaming starts
template <typename T>
SmoothSpec tiles_of(int nx, int ny, const SmoothSpec &p, const RasRun &run)
{
    if (sizeof(T) != 4 || p.variant != STOKES_RAS || p.sweeps < 1 || !any_traversal(p) || !run.allow_tma ||
        run.pair_mode != 1 || p.k > 8 || nx < 64 || ny < 40 || (long long)nx * ny >= FREE_MAX_CELLS)
        return p;
    const long long given = (long long)((nx + p.ti - 1) / p.ti + 1) * ((ny + p.tj - 1) / p.tj + 1); // (shifted)
    if (p.sweeps <= p.k && p.sweeps <= 4 && given <= 152 && p.ti + 2 * p.overlap + 2 <= 48) return p;
    SmoothSpec q = p;
    const int passes = (p.sweeps + 7) / 8;
    q.k = (p.sweeps + passes - 1) / passes;
    q.overlap = q.k - 1;
    q.shift_mode = STOKES_SHIFT_NONE;
    q.ti = 64 - 2 * q.k;
    long long best = 0;
    for (int rows : {40, 50, 65, 80}) {
        const int tj = rows - 2 * q.k;
        const long long tiles = (long long)((nx + q.ti - 1) / q.ti) * ((ny + tj - 1) / tj);
        const long long cost = (tiles + 151) / 152 * (32 + rows);
        if (best == 0 || cost < best) {
            best = cost;
            q.tj = tj;
        }
    }
    return q;
}

} // namespace

// (passes: one per sweep, per outer iteration of RAS or per pass of a
// row-streaming kernel)
template <typename T>
SmoothPlan smooth_plan(int nx, int ny, const SmoothSpec &p, const RasRun &run)
{
    SmoothPlan n{false, 0, tiles_of<T>(nx, ny, p, run), p.sweeps};
    if (p.sweeps <= 0) {
        n.passes = 0;
    } else if (any_traversal(p) && cluster_takes<T>(nx, ny, p.sweeps, run)) {
        n.cluster = true;
        n.passes = 1;
    } else if ((n.stream = stream_passes_of<T>(nx, ny, p, run)) > 0) {
        n.passes = n.stream;
    } else if (p.variant == STOKES_RAS) {
        n.passes = (p.sweeps + n.tiles.k - 1) / n.tiles.k;
    }
    return n;
}

template <typename T>
int smooth_buffers(const GridDesc<T> &g, const Coeffs<T> &k, T *vx, T *vy, T *sx, T *sy, const SmoothSpec &p,
                   const RasRun &run, cudaStream_t s, LaunchHook &hook, bool *swapped, T *tx, T *ty,
                   bool zero_walls)
{
    if (swapped) *swapped = false;
    const T omega = (T)p.omega;
    int st = STOKES_OK;
#define LAUNCH(kind, nk, expr)                                                                                     \
    do {                                                                                                           \
        st = hook.run((kind), (nk), [&]() { return (expr); });                                                     \
        if (st != STOKES_OK) return st;                                                                            \
    } while (0)
    if (p.sweeps == 0) return STOKES_OK;
    const SmoothPlan plan = smooth_plan<T>(g.nx, g.ny, p, run);
    const SmoothSpec &q = plan.tiles; // what the tile launches run
    const int n_pass = plan.passes, n_stream = plan.stream;
    const bool cluster = plan.cluster;
    const int kind = p.variant == STOKES_RAS    ? STOKES_K_RAS
                     : p.variant == STOKES_RBGS ? STOKES_K_RBGS
                                                : STOKES_K_JACOBI;
    if ((cluster || n_stream > 0 || q.shift_mode != p.shift_mode) && p.variant == STOKES_RAS &&
        p.shift_mode == STOKES_SHIFT_LIST)
        for (int t = 0; t < (p.sweeps + p.k - 1) / p.k; ++t) // the shifts change nothing, but bad ones stay refused
            if (p.shifts[2 * t] < 0 || p.shifts[2 * t] >= p.ti || p.shifts[2 * t + 1] < 0 || p.shifts[2 * t + 1] >= p.tj)
                return STOKES_ERR_ARG;
    if (cluster) {
        LAUNCH(kind, 1, launch_jacobi_cluster<T>(g, k, omega, p.sweeps, vx, vy, run, s));
        return STOKES_OK;
    }
    // ping-pong between (vx, vy) and the scratch pair; the scratch walls take
    // the Dirichlet values of (vx, vy).  With a second scratch pair (tx, ty)
    // and an odd number n >= 3 of passes, pass 1 goes from (vx, vy) to (sx, sy),
    // passes 2 .. n-1 alternate between the two scratch pairs and pass n
    // writes (vx, vy): the result lands in place without a copy back.
    const bool three = tx && ty && !swapped && n_pass >= 3 && (n_pass & 1);
    T *ax = vx, *ay = vy, *bx = sx, *by = sy;
    if (!zero_walls) LAUNCH(STOKES_K_COPY, 1, launch_copy_walls<T>(g, vx, vy, sx, sy, s));
    if (three) LAUNCH(STOKES_K_COPY, 1, launch_copy_walls<T>(g, vx, vy, tx, ty, s));
    int passes = 0;
    // after pass `passes` (1-based) wrote (bx, by): the source and target of the next
    auto advance = [&]() {
        T *nx_ = bx, *ny_ = by;
        if (!three) {
            bx = ax;
            by = ay;
        } else if (passes == n_pass - 1) {
            bx = vx;
            by = vy;
        } else {
            bx = (nx_ == sx) ? tx : sx;
            by = (ny_ == sy) ? ty : sy;
        }
        ax = nx_;
        ay = ny_;
    };
    if (n_stream > 0) {
        for (int t = 0; t < n_stream; ++t) {
            const int ks = p.sweeps / n_stream + (t < p.sweeps % n_stream ? 1 : 0);
            if constexpr (sizeof(T) == 8) {
                LAUNCH(kind, 1, launch_ras_stream64(g, k, omega, ks, ax, ay, bx, by, s));
            } else if (p.variant == STOKES_RBGS) {
                LAUNCH(kind, 1, launch_rbgs_stream(g, k, omega, ks, ax, ay, bx, by, s));
            } else {
                LAUNCH(kind, 1, launch_ras_stream(g, k, omega, ks, ax, ay, bx, by, s));
            }
            ++passes;
            advance();
        }
    } else if (p.variant == STOKES_RAS) {
        for (int t = 0; t < n_pass; ++t) {
            const int ks = (t == n_pass - 1) ? q.sweeps - (n_pass - 1) * q.k : q.k;
            int si = 0, sj = 0;
            if (q.shift_mode == STOKES_SHIFT_SPLITMIX) {
                si = (int)(splitmix64(q.seed, 2u * (uint64_t)t) % (uint64_t)q.ti);
                sj = (int)(splitmix64(q.seed, 2u * (uint64_t)t + 1u) % (uint64_t)q.tj);
            } else if (q.shift_mode == STOKES_SHIFT_LIST) {
                si = q.shifts[2 * t];
                sj = q.shifts[2 * t + 1];
                if (si < 0 || si >= q.ti || sj < 0 || sj >= q.tj) return STOKES_ERR_ARG;
            }
            const TileGrid tg = make_tiles(g.nx, g.ny, q.ti, q.tj, si, sj);
            LAUNCH(STOKES_K_RAS, 1, launch_ras<T>(g, k, omega, tg, ks, q.overlap, ax, ay, bx, by, run, s));
            ++passes;
            advance();
        }
    } else {
        for (int it = 0; it < p.sweeps; ++it) {
            if (p.variant == STOKES_RBGS) {
                LAUNCH(STOKES_K_RBGS, 1, launch_rbgs_sweep<T>(g, k, omega, ax, ay, bx, by, s));
            } else if (p.variant == STOKES_JACOBI_BLOCKED) {
                const TileGrid tg = make_tiles(g.nx, g.ny, p.ti, p.tj, 0, 0);
                LAUNCH(STOKES_K_RAS, 1, launch_ras<T>(g, k, omega, tg, 1, 0, ax, ay, bx, by, run, s));
            } else {
                const int fused = p.variant == STOKES_JACOBI_FUSED;
                LAUNCH(STOKES_K_JACOBI, fused ? 1 : 2, launch_jacobi<T>(g, k, omega, ax, ay, bx, by, fused, s));
            }
            ++passes;
            advance();
        }
    }
    if ((passes & 1) && !three) {
        if (swapped)
            *swapped = true; // the result stays in (sx, sy); the caller swaps its pointers
        else
            LAUNCH(STOKES_K_COPY, 1, launch_copy_velocity<T>(g, ax, ay, vx, vy, s));
    }
#undef LAUNCH
    return STOKES_OK;
}

template SmoothPlan smooth_plan<float>(int, int, const SmoothSpec &, const RasRun &);
template SmoothPlan smooth_plan<double>(int, int, const SmoothSpec &, const RasRun &);
template int smooth_buffers<float>(const GridDesc<float> &, const Coeffs<float> &, float *, float *, float *,
                                   float *, const SmoothSpec &, const RasRun &, cudaStream_t, LaunchHook &, bool *,
                                   float *, float *, bool);
template int smooth_buffers<double>(const GridDesc<double> &, const Coeffs<double> &, double *, double *, double *,
                                    double *, const SmoothSpec &, const RasRun &, cudaStream_t, LaunchHook &, bool *,
                                    double *, double *, bool);

} // namespace stokes
