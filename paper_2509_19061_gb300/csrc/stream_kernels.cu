// stream_kernels.cu -- temporally blocked Jacobi by row streaming, the FP32
// path of fused Jacobi and of RAS schedules that equal global Jacobi
// (overlap >= k - 1, Sec. 4.3) on grids large enough to fill the GPU.
//
// Such a schedule's result does not depend on its tiles, so any traversal that
// performs the same sweeps gives the same values.  The tile kernels sweep the
// halo of every tile again (48 x 64 cells owned of a 64 x 80 window, 40 % of
// the arithmetic, for k = 8) and meet at a barrier each sweep.  Here a strip of
// 128 columns (four adjacent columns per lane, as two packed FP32 pairs) is
// marched up row by row with all sweeps of a pass in flight: when row j
// arrives, sweep 1 updates row j - 1, sweep 2 row j - 2, ..., the last sweep
// row j - n, which is written out.  A sweep keeps its last row's velocity,
// shear and Tyy in registers, and a warp the coefficients of as many rows as
// it has sweeps in flight, in a ring indexed at compile time (the row loop is
// unrolled over it).  There is no halo along y but the 2 n rows a segment
// starts and ends with; what is swept in vain are the n columns at either side
// of a strip (12.5 % for n = 8).
//
// Two warps share a strip: the front warp runs the first KL sweeps and hands
// their rows over in shared memory, the back warp runs the others (KL, or
// KL - 1 for an odd n), one row behind.  Half the sweeps per warp halve the
// registers, which pays for four columns per lane: two independent chains of
// arithmetic, half the shuffles and half the spare columns of a two-column
// form with all sweeps in one warp (648 us a pass of 7.7 sweeps at 8192^2,
// against 470 here and 915 for the pair kernel's 48 x 64 tiles).
//
// Bounds (8192^2, 100 sweeps in 13 passes): 40 bytes a cell and pass (eight
// fields read, two written) take 400 us at the measured copy rate, the packed
// arithmetic about 360 us of the FMA pipe; 470 us is 0.85 of that copy rate.
// On the way: the rows' loads and copies at the end of a step instead of its
// start 564 us; register copies left by a ring of KL slots under state that
// rotates through KL + 1 another 100 us.
//
// The front warp copies each row's eight fields into a ring of ST_D rows by
// cp.async (16 bytes a lane, zero-filled outside each field's extent); the
// back warp reads the coefficients of its rows there again.  Their only
// synchronisation is one barrier of the two warps per row.  A cell outside
// the unknowns has weight zero (its 1/diag is zero), so walls and the outside
// keep their values while the fields are finite.  Where a field overflows, the
// product of zero and infinity beside a wall is not zero, and the walls in
// memory must not take it: row 0 of vy is not stored, and the west wall's entry
// of vx, which shares a 16-byte store with three unknowns, is the one taken in,
// kept in shared memory until its row is written (100 sweeps of 8192^2 7.10 ms,
// 7.06 with computed walls stored; 20 of 4001 x 2999 410 us and 406.  The strip
// at the wall is on the critical path of its wave: leaving the entry out by
// smaller stores took 7.46 to 7.72 ms, loading it from memory again 7.97).
#include <algorithm>

#include "f32x2.cuh"
#include "internal.h"
#include "tma.h"

namespace stokes {

namespace {

constexpr int ST_COLS = 128;     // columns of a strip
constexpr int ST_PAIRS = 4;      // strips (pairs of warps) per CTA
constexpr int ST_THREADS = ST_PAIRS * 64;
constexpr int ST_ROW = ST_FIELDS * ST_COLS;           // elements of a staged row
constexpr int ST_MIN_SWEEPS = 3, ST_MAX_SWEEPS = 8;   // sweeps of a pass
constexpr long long ST_MIN_CELLS = 600000;            // smallest grid
constexpr int ST_WALLS = 16; // rows (a power of two above the rows in flight) whose west wall is kept

// barrier of the two warps of a pair
__device__ __forceinline__ void pair_sync(int pair)
{
    asm volatile("bar.sync %0, 64;" ::"r"(pair + 1) : "memory");
}

// four adjacent columns as two packed pairs
struct alignas(16) f4 {
    f2 a, b;
};
__device__ __forceinline__ f4 ld4(const float *p)
{
    return *reinterpret_cast<const f4 *>(p);
}
// 16-byte global stores of a row of vx and vy by the lanes whose `on` is set,
// without a branch; vy only if row > 0
__device__ __forceinline__ void st4_both(float *px, f4 x, float *py, f4 y, bool on, int row)
{
    asm volatile("{\n\t.reg .pred p, r;\n\tsetp.ne.s32 p, %6, 0;\n\t@p st.global.v2.b64 [%0], {%1, %2};\n\t"
                 "setp.gt.and.s32 r, %7, 0, p;\n\t@r st.global.v2.b64 [%3], {%4, %5};\n\t}" ::"l"(px),
                 "l"(x.a.u), "l"(x.b.u), "l"(py), "l"(y.a.u), "l"(y.b.u), "r"((int)on), "r"(row)
                 : "memory");
}
// shared store, and load over v, of the lanes whose `on` is set, without a branch
__device__ __forceinline__ void sts_if(uint32_t p, float v, bool on)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p st.shared.f32 [%0], %1;\n\t}" ::"r"(p), "f"(v),
                 "r"((int)on)
                 : "memory");
}
__device__ __forceinline__ float lds_if(uint32_t p, float v, bool on)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p ld.shared.f32 %0, [%1];\n\t}"
                 : "+f"(v)
                 : "r"(p), "r"((int)on)
                 : "memory");
    return v;
}
__device__ __forceinline__ f4 operator+(f4 x, f4 y) { return {add2(x.a, y.a), add2(x.b, y.b)}; }
__device__ __forceinline__ f4 operator-(f4 x, f4 y) { return {sub2(x.a, y.a), sub2(x.b, y.b)}; }
__device__ __forceinline__ f4 mul4(f4 x, f4 y) { return {mul2(x.a, y.a), mul2(x.b, y.b)}; }
__device__ __forceinline__ f4 mul4(f4 x, f2 y) { return {mul2(x.a, y), mul2(x.b, y)}; }
// a product that is not fused into the addition it feeds (see mul2r)
__device__ __forceinline__ f4 mul4r(f4 x, f4 y) { return {mul2r(x.a, y.a), mul2r(x.b, y.b)}; }
__device__ __forceinline__ f4 mul4r(f4 x, f2 y) { return {mul2r(x.a, y), mul2r(x.b, y)}; }
__device__ __forceinline__ f4 fma4(f4 x, f4 y, f4 z) { return {fma2(x.a, y.a, z.a), fma2(x.b, y.b, z.b)}; }
__device__ __forceinline__ f4 fma4(f4 x, f2 y, f4 z) { return {fma2(x.a, y, z.a), fma2(x.b, y, z.b)}; }
// x - its west neighbour and its east neighbour - x, column by column: scalar
// halves, which need no register moves to pair the neighbours up
__device__ __forceinline__ f4 diff_west(f4 x)
{
    const float c0 = f2lo(x.a), c1 = f2hi(x.a), c2 = f2lo(x.b), c3 = f2hi(x.b);
    return {pk(__fsub_rn(c0, __shfl_up_sync(0xffffffffu, c3, 1)), __fsub_rn(c1, c0)),
            pk(__fsub_rn(c2, c1), __fsub_rn(c3, c2))};
}
__device__ __forceinline__ f4 diff_east(f4 x)
{
    const float c0 = f2lo(x.a), c1 = f2hi(x.a), c2 = f2lo(x.b), c3 = f2hi(x.b);
    return {pk(__fsub_rn(c1, c0), __fsub_rn(c2, c1)),
            pk(__fsub_rn(c3, c2), __fsub_rn(__shfl_down_sync(0xffffffffu, c0, 1), c3))};
}

template <int KL>
struct StreamShape {
    static constexpr int N = KL + 1;                            // steps unrolled
    static constexpr int D = KL == 4 ? 10 : 12;                 // staged rows
    static constexpr int PF = D - KL - 2;                       // rows copied ahead
    static constexpr int SMEM = D * ST_ROW + 2 * 2 * ST_COLS;   // elements of a pair: ring, two handed-over rows of vx, vy
    static_assert(D % N == 0, "slots repeat with the unrolled steps");
};

// 2 KL - ODD sweeps of one strip and segment per pair of warps.  BATCH: of the
// tasks of a table of grids, else of the grid `one`.  SQ: square cells (one coefficient for Txx and Tyy, one scaled shear), as in the pair
// kernel.
template <int KL, bool ODD, bool SQ, bool BATCH>
__global__ void __launch_bounds__(ST_THREADS, 1)
    k_ras_stream(const __grid_constant__ StreamEntry one, const StreamEntry *__restrict__ tab,
                 const StreamTask *__restrict__ tasks, int ntasks, const int *__restrict__ live)
{
    using Sh = StreamShape<KL>;
    constexpr int N = Sh::N, D = Sh::D, PF = Sh::PF;
    extern __shared__ __align__(16) float smem[];
    __shared__ float walls[ST_PAIRS][ST_WALLS]; // vx of column 0 of the last rows taken in, slot = row
    __shared__ StreamEntry held[BATCH ? ST_PAIRS : 1];
    // (the shuffle tells the compiler that the warp number is uniform)
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = (int)threadIdx.x & 31;
    const int pair = warp % ST_PAIRS; // each SM partition holds a front and a back warp
    const bool back = warp >= ST_PAIRS;
    const int id = (int)blockIdx.x * ST_PAIRS + pair;
    if (id >= ntasks) return; // both warps of a pair; pairs never meet
    int piece = id;
    if (BATCH) {
        const StreamTask t = tasks[id];
        if (live && !live[tab[t.entry].inst]) return;
        piece = t.part;
        if (!back) {
            constexpr int W = (int)(sizeof(StreamEntry) / 4);
            static_assert(sizeof(StreamEntry) % 4 == 0, "copied by words");
            for (int w = lane; w < W; w += 32)
                reinterpret_cast<int *>(&held[BATCH ? pair : 0])[w] = reinterpret_cast<const int *>(&tab[t.entry])[w];
        }
        pair_sync(pair);
    }
    const StreamEntry &a = BATCH ? held[BATCH ? pair : 0] : one;
    const int strip = piece % a.strips, seg = piece / a.strips;
    const int nx = a.g.nx, ny = a.g.ny, n = a.sweeps;
    const int c0 = strip * a.own - a.hl + 4 * lane; // first of this lane's columns (a multiple of four, may lie outside)
    const int y0 = seg * a.rows, y1 = min(y0 + a.rows, ny);
    const int jb = y0 - n; // first row loaded
    // Steps: one per row from jb to y1 - 1 + n, rounded up to whole unrolled
    // rounds.  In step s the front warp takes in row jb + s and gives its last
    // sweep's row jb + s - KL to the back warp, whose step s takes that in and
    // gives row jb + s - n.  The back warp starts KL steps late and runs one
    // round less; both meet at rounds * N barriers.
    const int rounds = (y1 - y0 + 2 * n + 1 + N - 1) / N;
    float *const ring = smem + pair * Sh::SMEM + 4 * lane; // this lane's columns of field 0 of slot 0
    float *const hand = ring + D * ST_ROW;                  // handed-over rows: step parity, vx, vy
    const int P = a.g.pitch;

    // bytes of this lane's columns inside a row of nx (cell) or nx + 1 (node) columns
    const int bc = c0 < 0 ? 0 : max(0, min(4, nx - c0)) * 4;
    const int bn = c0 < 0 ? 0 : max(0, min(4, nx + 1 - c0)) * 4;
    const int cc = min(max(c0, 0), P - 4); // columns inside the rows for the copies that read nothing
    const uint32_t ring_addr = smem_addr(ring);
    auto issue = [&](int j, uint32_t to) { // copy row j to the slot at `to`
        const long long at = (long long)min(max(j, 0), ny) * P + cc;
        const bool in0 = (unsigned)j < (unsigned)ny, in1 = (unsigned)j <= (unsigned)ny; // rows of the cells / of the nodes
        const int cr = in0 ? bc : 0, nr = in0 ? bn : 0, cn = in1 ? bc : 0, nn = in1 ? bn : 0;
        const int bytes[ST_FIELDS] = {nr, cn, cr, nn, nr, cn, nr, cn};
#pragma unroll
        for (int f = 0; f < ST_FIELDS; ++f) cp_async16z(to + f * ST_COLS * 4, a.f[f] + at, bytes[f]);
        cp_commit();
    };
    if (!back)
        for (int d = 0; d < PF; ++d) issue(jb + d, ring_addr + d * (ST_ROW * 4));

    const f2 z2 = {0ull};
    const f4 zero = {z2, z2};
    const f2 om = pk(a.omega, a.omega), cx = pk(a.g.ihx2, a.g.ihx2), cy = pk(a.g.ihy2, a.g.ihy2);
    const f2 ihx = pk(a.g.ihx, a.g.ihx), ihy = pk(a.g.ihy, a.g.ihy);
    // Coefficients of the rows taken in, slot = step mod N: the sweeps need the
    // last KL rows, the spare slot makes the period that of the state below.
    // Per sweep: the velocity it starts from at its last row, that row's shear
    // (Sx, Sy) and the Tyy of the row before.  Sweep t's new row of each goes to
    // the slot that sweep t - 1 has just left, so sweep t's state moves one slot
    // down a step and is back after N steps: nothing is ever copied.
    f4 ax[N], ay[SQ ? 1 : N], en[N], bx[N], by[N], wx[N], wy[N];
    f4 vx[N], vy[N], sx[N], sy[SQ ? 1 : N], ty[N];
#pragma unroll
    for (int t = 0; t < N; ++t) {
        ax[t] = en[t] = bx[t] = by[t] = wx[t] = wy[t] = zero;
        vx[t] = vy[t] = sx[t] = ty[t] = zero;
        if (!SQ) ay[SQ ? 0 : t] = sy[SQ ? 0 : t] = zero;
    }
    // columns this lane writes: all four, or `part` at the grid's right end
    const bool mine = 4 * lane >= a.hl && 4 * lane < a.hl + a.own;
    const bool full = mine && c0 + 4 <= nx, west = mine && c0 == 0;
    const int part = mine && !full ? nx - c0 : 0;
    const bool ragged = __any_sync(0xffffffffu, part > 0);
    const uint32_t wring = smem_addr(walls[pair]);
    // (by a branch where that is the faster form: 8192^2 7.11 ms, 7.17 predicated;
    // the general form 425 us and 410 at 4001 x 2999)
    constexpr bool BRANCH = SQ && !BATCH;
    int row = jb - n + (back ? KL : 0);       // row the pass completes in this step, as a back warp
    long long q = (long long)row * P + c0;
    int slot = 0;                             // staged slot of the round's first row
    int par = back ? KL & 1 : 0;              // parity of the round's first step
    uint32_t ahead = ring_addr + PF * (ST_ROW * 4); // slot of the next row to copy
    if (back)
        for (int s = 0; s < KL; ++s) pair_sync(pair);
    for (int rd = back ? 1 : 0; rd < rounds; ++rd) {
        const float *lp = ring + slot * ST_ROW;
#pragma unroll
        for (int u = 0; u < N; ++u) {
            // the row taken in: the snapshot's from the ring, or the front warp's
            if (back) pair_sync(pair);
            else cp_wait<PF - 1>();
            if (!back) {
                issue(jb + rd * N + u + PF, ahead);
                ahead = ahead == ring_addr + (D - 1) * (ST_ROW * 4) ? ring_addr : ahead + ST_ROW * 4;
            }
            const float *const in = back ? hand + ((par + u) & 1) * (2 * ST_COLS) : lp + u * ST_ROW;
            f4 ix = ld4(in), iy = ld4(in + ST_COLS);
            if (BRANCH) {
                if (!back && west) walls[pair][(jb + rd * N + u) & (ST_WALLS - 1)] = f2lo(ix.a);
            } else if (!back) {
                sts_if(wring + ((jb + rd * N + u) & (ST_WALLS - 1)) * 4, f2lo(ix.a), west);
            }
            auto ld = [&](int f) { return ld4(lp + u * ST_ROW + f * ST_COLS); };
            en[u] = SQ ? mul4(ld(3), cx) : ld(3);
            // the row's coefficients replace those of the row KL steps ago
            // (coef_x, coef_y, jacobi_weight and shear_sq of stencil.cuh, lane for lane)
            const f4 ec = ld(2), e2 = ec + ec;
            ax[u] = mul4(e2, cx);
            if (!SQ) ay[SQ ? 0 : u] = mul4(e2, cy);
            bx[u] = ld(4);
            by[u] = ld(5);
            wx[u] = mul4(ld(6), om);
            wy[u] = mul4(ld(7), om);
#pragma unroll
            for (int t = 1; t <= KL; ++t) {
                const int c = (u - t + N) % N, e = (u - t + 1 + N) % N; // slots of the sweep's row and of the row above
                const int v = (t - 1 - u + N) % N, w = (v + N - 1) % N; // slots of the sweep's state: now, next step
                if (ODD && t == KL && back) break;
                const f4 txx = mul4r(ax[c], diff_east(vx[v]));
                const f4 dy = diff_east(SQ ? sx[v] : sy[SQ ? 0 : v]);
                const f4 tyy = mul4r(SQ ? ax[c] : ay[SQ ? 0 : c], iy - vy[v]);
                const f4 my = dy + (tyy - ty[v]);
                const f4 nvy = fma4(by[c] - my, wy[c], vy[v]);
                f4 sxn, syn;
                if (SQ) {
                    sxn = syn = mul4r(en[e], (ix - vx[v]) + diff_west(iy));
                } else {
                    const f4 sh = mul4(en[e], fma4(ix - vx[v], ihy, mul4(diff_west(iy), ihx)));
                    sxn = mul4r(sh, ihy);
                    syn = mul4r(sh, ihx);
                }
                const f4 mx = diff_west(txx) + (sxn - sx[v]);
                const f4 nvx = fma4(bx[c] - mx, wx[c], vx[v]);
                vx[w] = ix;
                vy[w] = iy;
                sx[w] = sxn;
                if (!SQ) sy[SQ ? 0 : w] = syn;
                ty[w] = tyy;
                ix = nvx;
                iy = nvy;
            }
            if (!back) {
                float *const out = hand + ((par + u) & 1) * (2 * ST_COLS);
                *reinterpret_cast<f4 *>(out) = ix;
                *reinterpret_cast<f4 *>(out + ST_COLS) = iy;
            } else if (row >= y0 && row < y1) {
                if (BRANCH) {
                    if (west) ix.a = pk(walls[pair][row & (ST_WALLS - 1)], f2hi(ix.a));
                } else {
                    ix.a = pk(lds_if(wring + (row & (ST_WALLS - 1)) * 4, f2lo(ix.a), west), f2hi(ix.a));
                }
                st4_both(a.ox + q, ix, a.oy + q, iy, full, row);
                if (ragged) {
                    const bool uy = row > 0;
                    const f4 o[2] = {ix, iy};
#pragma unroll
                    for (int w = 0; w < 2; ++w) {
                        float *const p = (w ? a.oy : a.ox) + q;
                        if (part > 0 && (!w || uy)) p[0] = f2lo(o[w].a);
                        if (part > 1 && (!w || uy)) p[1] = f2hi(o[w].a);
                        if (part > 2 && (!w || uy)) p[2] = f2lo(o[w].b);
                    }
                }
            }
            ++row;
            q += P;
            if (!back) {
                pair_sync(pair);
            }
        }
        par ^= N & 1;
        slot += N;
        if (slot == D) slot = 0;
    }
    if (back) pair_sync(pair);
    cp_wait<0>(); // no copy outlives the warp
}

using StreamKernel = void (*)(StreamEntry, const StreamEntry *, const StreamTask *, int, const int *);

template <int KL, bool BATCH>
StreamKernel pick_stream(bool odd, bool square)
{
    if (odd) return square ? k_ras_stream<KL, true, true, BATCH> : k_ras_stream<KL, true, false, BATCH>;
    return square ? k_ras_stream<KL, false, true, BATCH> : k_ras_stream<KL, false, false, BATCH>;
}

template <bool BATCH>
cudaError_t run(int sweeps, bool square, const StreamEntry &one, const StreamEntry *tab, const StreamTask *tasks,
                int ntasks, const int *live, cudaStream_t s)
{
    const int kl = (sweeps + 1) / 2;
    const bool odd = sweeps & 1;
    const StreamKernel kern = kl == 2   ? pick_stream<2, BATCH>(odd, square)
                              : kl == 3 ? pick_stream<3, BATCH>(odd, square)
                                        : pick_stream<4, BATCH>(odd, square);
    const int elems = kl == 2 ? StreamShape<2>::SMEM : kl == 3 ? StreamShape<3>::SMEM : StreamShape<4>::SMEM;
    const size_t smem = (size_t)ST_PAIRS * elems * sizeof(float);
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<(ntasks + ST_PAIRS - 1) / ST_PAIRS, ST_THREADS, smem, s>>>(one, tab, tasks, ntasks, live);
    return cudaGetLastError();
}

int stream_wave()
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return std::max(sms, 1) * ST_PAIRS;
}

} // namespace

int stream_passes(long long cells, int sweeps, const RasRun &run)
{
    if (!run.allow_tma || run.pair_mode != 1 || sweeps < ST_MIN_SWEEPS) return 0;
    // Below this a segment's 2 n extra rows outweigh the tiles' halo: 40 sweeps
    // take 101 us either way at 768^2, 80 (48 x 64 tiles: 70) at 512^2 and 111
    // (132) at 1024^2.  In a batch the instances' strips fill the wave together,
    // half-empty ones too (20 sweeps, against 48 x 64 tiles: 200 grids of 64^2 101
    // us and 180, 3000 of 32^2 551 and 892, 4000 of 16^2 474 and 595; three sweeps
    // of 200 of 64^2 46 and 61).
    if (cells < ST_MIN_CELLS) return 0;
    return (sweeps + ST_MAX_SWEEPS - 1) / ST_MAX_SWEEPS;
}

StreamEntry stream_entry(const GridDesc<float> &g, const Coeffs<float> &c, float omega, int sweeps, const float *vx,
                         const float *vy, float *ox, float *oy)
{
    StreamEntry a{};
    a.g = g;
    a.omega = omega;
    a.ox = ox;
    a.oy = oy;
    a.sweeps = sweeps;
    const float *const f[ST_FIELDS] = {vx, vy, c.eta_c, c.eta_n, c.bx, c.by, c.inv_dx, c.inv_dy};
    for (int q = 0; q < ST_FIELDS; ++q) a.f[q] = f[q];
    // at least `sweeps` columns at either side of the owned ones; strips start
    // on 16-byte boundaries, and owned columns are a multiple of eight
    a.hl = sweeps <= 4 ? 4 : 8;
    a.own = ST_COLS - 2 * a.hl;
    a.strips = (g.nx + a.own - 1) / a.own;
    return a;
}

int stream_split(StreamEntry *e, int n)
{
    // the strips' rows, and the shortest segment that keeps the tasks within
    // one wave (several where a wave's share is long: finer pieces even out
    // grids of different heights, at 2 n + 1 extra rows each)
    long long total = 0;
    int longest = 1;
    for (int q = 0; q < n; ++q) {
        total += (long long)e[q].strips * e[q].g.ny;
        longest = std::max(longest, e[q].g.ny);
    }
    const long long wave = stream_wave(), share = total / wave;
    const long long want = wave * (n == 1 ? 1 : std::max(1LL, std::min(8LL, share / 100)));
    auto tasks = [&](int rows) {
        long long t = 0;
        for (int q = 0; q < n; ++q) t += (long long)e[q].strips * ((e[q].g.ny + rows - 1) / rows);
        return t;
    };
    int lo = 1, hi = longest; // tasks(hi) may exceed `want` (many strips): then one segment each
    while (lo < hi) {
        const int mid = (lo + hi) / 2;
        if (tasks(mid) <= want) hi = mid;
        else lo = mid + 1;
    }
    int t = 0;
    for (int q = 0; q < n; ++q) {
        const int segs = (e[q].g.ny + lo - 1) / lo;
        e[q].rows = (e[q].g.ny + segs - 1) / segs;
        e[q].segs = (e[q].g.ny + e[q].rows - 1) / e[q].rows;
        t += e[q].strips * e[q].segs;
    }
    return t;
}

cudaError_t launch_ras_stream(const GridDesc<float> &g, const Coeffs<float> &c, float omega, int sweeps,
                              const float *vx, const float *vy, float *ox, float *oy, cudaStream_t s)
{
    if (!c.inv_dx || !c.inv_dy || sweeps < ST_MIN_SWEEPS || sweeps > ST_MAX_SWEEPS) return cudaErrorInvalidValue;
    StreamEntry a = stream_entry(g, c, omega, sweeps, vx, vy, ox, oy);
    const int ntasks = stream_split(&a, 1);
    return run<false>(sweeps, g.square != 0, a, nullptr, nullptr, ntasks, nullptr, s);
}

cudaError_t launch_ras_stream_batch(const StreamEntry *tab, const StreamTask *tasks, int ntasks, int sweeps,
                                    bool square, const int *live, cudaStream_t s)
{
    if (sweeps < ST_MIN_SWEEPS || sweeps > ST_MAX_SWEEPS) return cudaErrorInvalidValue;
    if (ntasks <= 0) return cudaSuccess;
    return run<true>(sweeps, square, StreamEntry{}, tab, tasks, ntasks, live, s);
}

} // namespace stokes
