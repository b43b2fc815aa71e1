// FP64 Cholesky A = L L^T in one launch, by 32 x 32 tiles (the FP64 form, the integer-order
// case, the GMRES preconditioner and the allocation-free solve).
//
// GB300 runs FP64 at two multiply-adds per SM and clock, so what bounds this factorisation
// is the FP64 pipe: of one SM along the diagonal chain, of all SMs over the rest.  A
// 64-wide diagonal step is 300,000 FP64 multiply-add slots of one SM (about 150 us); the same
// 64 columns in two 32-wide steps are a quarter of that, because the chain's products
// (update of the diagonal tile, solve of the tile below it) shrink with the cube of the width
// and there are twice as many.  The other SMs do not mind: a 32^3 product is 8 us of one SM's
// FP64 pipe, enough to hide the next tiles' loads and flags.  Narrower (16) tiles would not be.
//
// The first CTA to start runs the diagonal chain: for each block column j it applies the last update
// (k = j - 1) to the diagonal tile, factors and inverts it, solves the tile below it,
// L_{j+1,j} = A_{j+1,j} L_jj^{-T}, and keeps that tile in shared memory for the next
// diagonal update, so the critical path never leaves one SM.  The other CTAs take tasks
// W(i, j) over the lower tiles from an atomic ticket, column by column: W(i, j) subtracts
// L_ik L_jk^T for k < j (for a diagonal tile k < j - 1), each as soon as tiles (i, k) and
// (j, k) are final; the diagonal and sub-diagonal tiles are then stored for the chain
// ("updated" flag U), every other tile is solved with L_jj^{-1} once the chain has published
// it and stored as final (flag F).  Every task depends only on tiles of earlier columns (or,
// for the solve, on the chain's step j), and tickets are taken in column order, so the
// earliest unfinished claimed task always proceeds.  The chain itself waits for tasks, which no CTA
// may have claimed yet when other work holds the rest of the chip: a chain that has waited
// kHelpSpins then takes tickets up to the tile it needs and does them itself.  So every wait is
// for a CTA that is running, and the launch needs no co-residency: one CTA alone finishes it (with
// all SMs but one held by other work, the allocation-free solve of 384 unknowns takes 21 ms, 16 of
// them before the chain first helps; 0.42 ms undisturbed, as without this provision).
// Waits are bounded; one that expires sets the abort word, which every other wait also
// watches, and records ERR_CHOL.
// flags: F [0, ntask), U [ntask, 2 ntask), ticket [2 ntask], abort word [2 ntask + 1], CTAs that
// have started [2 ntask + 2]; all zero at launch.
//
// Work split.  Warp w of 16 owns the 8 x 8 outputs (block row w / 4, block column w % 4) of a
// tile product, two neighbouring columns per lane.  With whole 8 x 8 blocks per warp the
// diagonal update skips the six blocks above the diagonal and a product with the triangular
// L_jj^{-1} stops at the block's last nonzero column: both take 5/8 of a full product's slots
// of the FP64 pipe.
//
// Measured (GB300; before: the 64 x 64 tiles that the FP32 factor keeps): order 1,000 3.08 ->
// 0.91 ms, order 2,744 9.3 -> 6.9 ms (n^3 / 3 multiply-adds at the FP64 rate: 5.5 ms); one chain step
// of 32 columns 28 us (diagonal factor 31,000 clocks, update and sub-solve 10,400 each)
// where one of 64 took 193 us.
//
// Profile.  Given `first` (per block row the first tile column that holds a nonzero of A), the
// tiles left of it are skipped: a Cholesky factor fills only inside the profile of A.  The
// integer-order matrices are banded in the node order (2,744 dofs of the 15^3 cube: 7 of up
// to 86 tile columns; factor 6.9 -> 2.4 ms, the diagonal chain alone).  The fractional ones
// are full, their calls pass none.
//
// Output: A's tiles below the diagonal become L (a diagonal tile keeps its last update), and
// the inverses of the 64 x 64 diagonal blocks that the triangular solves use go to dinv:
// 32 x 32 diagonal halves by the chain, the block below them, -X22 L21 X11, by
// k_join_dinv.
#include <algorithm>

#include "chol_f64.cuh"

namespace fem3 {

namespace {

#include "chol_smem.cuh"

constexpr int kT = kChol64Tile;
constexpr int kLd = kT + 2;            // shared tile row: 272 bytes, 16-byte aligned
constexpr int kThreads = 512;
// more than half an SM's shared memory, so that the chain CTA has its SM to itself
constexpr int kSmemBytes = 120 * 1024;

__device__ __forceinline__ int tile_id(int i, int j) { return i * (i + 1) / 2 + j; }

__device__ __forceinline__ bool wait_tile(const int *f, int *abort_w, int32_t *err) {
    int spins = 0;
    while (ld_acquire_gpu(f) == 0) {
        if (ld_acquire_gpu(abort_w) != 0) return false;
        if (++spins > kSpinLimit) {
            atomicAdd(&err[ERR_CHOL], 1);
            atomicExch(abort_w, 1);
            return false;
        }
        if (spins > 64) __nanosleep(128);   // 150 pollers on one L2 line slow its owner
    }
    return true;
}

// polls of the chain before it helps, and once it had to: 16 ms, above the chain's waits in an
// undisturbed launch up to some 30,000 columns, and some 20 us
constexpr int kHelpSpins = 1 << 15, kHungrySpins = 32;
// the chain's look at a flag: 1 set, 0 another wait gave up, 2 not set after `limit` polls
__device__ __forceinline__ int poll_tile(const int *f, const int *abort_w, int limit) {
    for (int spins = 0; ld_acquire_gpu(f) == 0; spins++) {
        if (ld_acquire_gpu(abort_w) != 0) return 0;
        if (spins >= limit) return 2;
        if (spins > 64) __nanosleep(128);
    }
    return 1;
}

// rows 2w, 2w + 1 of a tile for warp w, lane = column (L2 loads: the tile was written by
// another CTA of the same launch); rows from `rows` on read as zero
__device__ __forceinline__ double2 tile_rows(const double *src, int64_t ld, int64_t rows) {
    const int lane = threadIdx.x & 31, r = (threadIdx.x >> 5) * 2;
    double2 v;
    v.x = r < rows ? __ldcg(src + (int64_t)r * ld + lane) : 0.0;
    v.y = r + 1 < rows ? __ldcg(src + (int64_t)(r + 1) * ld + lane) : 0.0;
    return v;
}
// dst[c][r] = the loaded tile's entry (r, c)
__device__ __forceinline__ void tile_store_T(double2 v, double (*dst)[kLd]) {
    const int lane = threadIdx.x & 31, r = (threadIdx.x >> 5) * 2;
    *reinterpret_cast<double2 *>(&dst[lane][r]) = v;
}

// t = sum over k < kn of bi[k][r] bj[k][c .. c + 1]
__device__ __forceinline__ double2 dot2(const double (*bi)[kLd], const double (*bj)[kLd], int kn,
                                        int r, int c) {
    double2 t = make_double2(0.0, 0.0);
#pragma unroll 8
    for (int k = 0; k < kn; k++) {
        const double u = bi[k][r];
        const double2 v = *reinterpret_cast<const double2 *>(&bj[k][c]);
        t.x = fma(u, v.x, t.x);
        t.y = fma(u, v.y, t.y);
    }
    return t;
}

// entries (r, c), (r, c + 1) of tile (r0, c0) of A (identity past n on a diagonal tile)
__device__ __forceinline__ double2 load_acc(const double *A, int64_t n, int64_t r0, int64_t c0,
                                            bool diag, int r, int c) {
    double2 v = make_double2(diag && r == c ? 1.0 : 0.0, diag && r == c + 1 ? 1.0 : 0.0);
    if (r0 + r < n) {
        const double *p = A + (r0 + r) * n + c0 + c;
        if (c0 + c < n) v.x = __ldcg(p);
        if (c0 + c + 1 < n) v.y = __ldcg(p + 1);
    }
    return v;
}
__device__ __forceinline__ void store_acc(double *A, int64_t n, int64_t r0, int64_t c0, double2 v,
                                          int r, int c) {
    if (r0 + r >= n) return;
    double *p = A + (r0 + r) * n + c0 + c;
    if (c0 + c < n) p[0] = v.x;
    if (c0 + c + 1 < n) p[1] = v.y;
}

// all threads' global stores of a tile are visible before its flag: the barrier orders
// them before thread 0's release, which is cumulative
__device__ __forceinline__ void publish(int *f) {
    __syncthreads();
    if (threadIdx.x == 0) st_release_gpu(f, 1);
}

// where the inverse of diagonal tile j sits in the 64 x 64 inverses (row stride 64)
__device__ __forceinline__ int64_t dinv_at(int j) {
    return (int64_t)(j >> 1) * (64 * 64) + (j & 1) * (kT * 65);
}

// ---------------------------------------------------------------------------------
// The diagonal chain (one CTA).  One FP64 instruction of a warp holds its SM sub-partition's
// FP64 pipe for 64 clocks whatever its lanes do (measured), so the chain is counted in
// those slots.  Warps 0-11 compute; warps 12-15 load the tiles of the coming step and publish
// the finished ones, so no compute warp waits for a flag, a load or a release.
// ---------------------------------------------------------------------------------
constexpr int kMainWarps = 12, kMainThreads = 32 * kMainWarps;
constexpr int kMd = kT + 1;   // row stride of the diagonal step's shared arrays
// named barriers of the chain (0 is __syncthreads)
constexpr int kBarMain = 1, kBarDiag = 2, kBarSub = 3, kBarDone = 4, kBarIo = 5;

struct ChainSmem {
    double xt[2][kT][kLd];   // L_{j+1,j}^T of the last two steps
    double at[kT][kLd];      // A_{j+1,j}^T
    double d[kT][kMd];       // the diagonal tile before the update k = j - 1
    double x[kT][kMd];       // L_jj^{-1}
    // the diagonal factorisation (diag_factor_inv): columns of U = L D and of L for the 32 rows
    // of the tile and the 32 rows of the identity under it
    double u[2 * kT][kMd], f[2 * kT][kMd];
    double piv[kT], rs[kT];
    int ok_diag, ok_sub;   // the waits for the step's two tiles (written by the loading warps)
};
static_assert(sizeof(ChainSmem) <= kSmemBytes, "chain shared memory");

constexpr size_t kTaskAt = (sizeof(ChainSmem) + 15) / 16 * 16;   // shared memory of a task
static_assert(kTaskAt + sizeof(double) * 4 * kT * kLd <= kSmemBytes, "shared memory");

// Task W(i, j), all threads; false if a wait gave up.  Not inlined: the workers and the chain's help
// share one copy, and shared memory is named here so that it is addressed as such.
__device__ __noinline__ bool tile_task(double *A, int64_t n, int nblk, double *dinv,
                                       const int *__restrict__ first_col, int i, int j, int *F, int *U,
                                       int *abort_w, int32_t *err) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double(*b0)[kLd] = reinterpret_cast<double(*)[kLd]>(smem_raw + kTaskAt);   // two pairs of tiles
    __shared__ int s_ok, s_fa, s_fb, s_pa[2], s_pb[2];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rb = warp >> 2, cb = warp & 3;
    const int r = rb * 8 + (lane >> 2), c = cb * 8 + (lane & 3) * 2;
    const int64_t r0 = (int64_t)i * kT, c0 = (int64_t)j * kT;
    const int kmax = i == j ? max(j - 1, 0) : j;   // the chain applies k = j - 1 to (j, j)
    int kmin = 0;
    if (first_col) kmin = max(first_col[i], first_col[j]);
    double2 acc = load_acc(A, n, r0, c0, false, r, c);
    // Updates k = 0 .. kmax-1, pipelined: the tiles L_ik, L_jk of update k + 1 are
    // loaded into registers while update k's product runs (when their flags are
    // already set; otherwise after it, with a blocking wait), and stored into the other
    // pair of shared tiles.  Threads 0 and 32 read the two flags at the same time.
    double2 va, vb;
    bool have = false;   // va / vb hold the tiles of update k
    for (int k = kmin; k < kmax; k++) {
        double(*ta)[kLd] = b0 + (k & 1) * 2 * kT;
        double(*tb)[kLd] = ta + kT;
        if (!have) {
            if (tid == 0) s_fa = wait_tile(&F[tile_id(i, k)], abort_w, err);
            if (tid == 32) s_fb = wait_tile(&F[tile_id(j, k)], abort_w, err);
            __syncthreads();
            if (!(s_fa && s_fb)) return false;
            va = tile_rows(A + r0 * n + (int64_t)k * kT, n, n - r0);
            if (i != j) vb = tile_rows(A + c0 * n + (int64_t)k * kT, n, n - c0);
        }
        tile_store_T(va, ta);
        if (i != j) tile_store_T(vb, tb);
        const int q = (k + 1) & 1;
        if (k + 1 < kmax) {   // a look at update k + 1's flags, without waiting
            if (tid == 0) s_pa[q] = ld_acquire_gpu(&F[tile_id(i, k + 1)]) != 0;
            if (tid == 32) s_pb[q] = ld_acquire_gpu(&F[tile_id(j, k + 1)]) != 0;
        }
        __syncthreads();   // update k's tiles stored (the pair written two updates ago
                           // is no longer read); update k + 1's flags seen
        have = k + 1 < kmax && s_pa[q] && s_pb[q];
        if (have) {
            va = tile_rows(A + r0 * n + (int64_t)(k + 1) * kT, n, n - r0);
            if (i != j) vb = tile_rows(A + c0 * n + (int64_t)(k + 1) * kT, n, n - c0);
        }
        if (i != j || rb >= cb) {
            const double2 s = dot2(ta, i == j ? ta : tb, kT, r, c);
            acc.x -= s.x;
            acc.y -= s.y;
        }
    }
    __syncthreads();   // the last product is done before the shared tiles are reused
    if (i <= j + 1) {
        // diagonal or sub-diagonal tile: the chain finishes it
        store_acc(A, n, r0, c0, acc, r, c);
        publish(&U[tile_id(i, j)]);
        return true;
    }
    // L_ij = A_ij L_jj^{-T}: column c of the product ends at the inverse's row c
    double(*at)[kLd] = b0, (*lt)[kLd] = b0 + kT;   // A_ij^T, (L_jj^{-1})^T
    at[c][r] = acc.x;
    at[c + 1][r] = acc.y;
    if (tid == 0) s_ok = wait_tile(&F[tile_id(j, j)], abort_w, err);
    __syncthreads();
    if (!s_ok) return false;
    tile_store_T(tile_rows(dinv + dinv_at(j), 64, kT), lt);
    __syncthreads();
    const double2 o = dot2(at, lt, 8 * (cb + 1), r, c);
    store_acc(A, n, r0, c0, o, r, c);
    publish(&F[tile_id(i, j)]);
    return true;
}

// first ticket of a column
__device__ __forceinline__ int ticket_of(int nblk, int i, int j) {
    return j * nblk - j * (j - 1) / 2 + (i - j);
}

// The chain's CTA, all threads: one ticket up to `last`, if there is one that nobody has claimed;
// false if not.  Ends with a barrier.
__device__ bool help(double *A, int64_t n, int nblk, double *dinv, const int *__restrict__ first_col,
                     int last, int *F, int *U, int *ticket, int *abort_w, int32_t *err) {
    __shared__ int s_claim;
    if (threadIdx.x == 0) {
        int t = ld_acquire_gpu(ticket);
        while (t <= last) {
            const int seen = atomicCAS(ticket, t, t + 1);
            if (seen == t) break;
            t = seen;
        }
        s_claim = t <= last ? t : -1;
    }
    __syncthreads();
    const int t = s_claim;
    if (t >= 0) {
        int j = 0;
        while (t >= ticket_of(nblk, j + 1, j + 1)) j++;
        const int i = j + (t - ticket_of(nblk, j, j));
        if (!first_col || i <= j + 1 || j >= first_col[i])
            tile_task(A, n, nblk, dinv, first_col, i, j, F, U, abort_w, err);
    }
    __syncthreads();   // also after a task whose wait gave up (the chain's next poll sees that)
    return t >= 0;
}

// Panel p (columns 8p .. 8p + 7) of the augmented rows [A; I] by one warp: lanes 0-7 the
// pivot rows, lanes 8-31 the rows in `row` (-1: none).  Step j: f = x_j / d_j,
// x_k -= f a_kj (k > j), a_kj = x_j of lane k; the columns of U stay unscaled and f are
// those of the unit factor, so no square root is on the path.  Warps that share a panel
// repeat the pivot rows and get the same bits.
__device__ __forceinline__ void panel8(ChainSmem &S, int p, int row, bool first, int nb, int64_t k0,
                                       int32_t *err) {
    const int lane = threadIdx.x & 31, P = 8 * p;
    double x[8], f[8];
#pragma unroll
    for (int k = 0; k < 8; k++) x[k] = row >= 0 ? S.u[row][P + k] : 0.0;
    int bad = -1;
#pragma unroll
    for (int j = 0; j < 8; j++) {
        const double d = __shfl_sync(0xffffffffu, x[j], j);
        const bool pos = pivot_pos(d);
        if (!pos && bad < 0) bad = j;
        f[j] = x[j] * (pos ? recip_t<double>(d) : 1.0);
#pragma unroll
        for (int k = j + 1; k < 8; k++)
            x[k] = fma(-f[j], __shfl_sync(0xffffffffu, x[j], k), x[k]);
    }
    if (first && lane < 8) {
        double d = x[0];
#pragma unroll
        for (int j = 1; j < 8; j++)
            if (lane == j) d = x[j];
        S.piv[P + lane] = pivot_pos(d) ? d : 1.0;
    }
    if (lane >= 8 && row >= 0) {
#pragma unroll
        for (int k = 0; k < 8; k++) {
            S.u[row][P + k] = x[k];
            S.f[row][P + k] = f[k];
        }
    }
    if (first && bad >= 0 && lane == 0 && P + bad < nb)
        atomicCAS(&err[ERR_NOT_SPD], 0, (int32_t)(k0 + P + bad + 1));
}

// u[row][col] -= sum over panel p of f[row][.] u[col][.]
__device__ __forceinline__ void panel_update(ChainSmem &S, int p, int row, int col) {
    double t = 0.0;
#pragma unroll
    for (int k = 0; k < 8; k++) t = fma(S.f[row][8 * p + k], S.u[col][8 * p + k], t);
    S.u[row][col] -= t;
}

// the tile in u (rows 0 .. 31, identity in rows 32 .. 63): x = L^{-1} of its Cholesky factor.
// Eliminating the augmented rows gives U = L D on the tile's rows and L^{-T} (unit) on the
// identity's, in four panels of eight columns; row i of L^{-1} is then scaled by
// 1 / sqrt(d_i).  Of the identity only rows 0 .. 8p + 7 are nonzero up to panel p, so with
// the tile's rows below it a panel always has 32 rows beside its own pivots.
// Slots of one sub-partition on the critical path: 60 per panel and 16 for the update of the
// next panel's columns; the update of later columns runs beside the next panel on the
// sub-partitions (2 and 3) it leaves free.
__device__ __forceinline__ void diag_factor_inv(ChainSmem &S, int nb, int64_t k0, int32_t *err) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int p = 0; p < 4; p++) {
        const int P = 8 * p;
        if (warp < 2 || (warp == 2 && p == 3)) {
            const int q = lane - 8;
            int row = P + lane;   // pivot rows
            if (lane >= 8) {
                if (warp == 0) row = P + 8 + q < kT ? P + 8 + q : -1;
                else if (warp == 1) row = q < P + 8 ? kT + q : -1;
                else row = q < 8 ? kT + 24 + q : -1;
            }
            panel8(S, p, row, warp == 0, nb, k0, err);
            if (warp == 0 && p == 3) {
                __syncwarp();   // the lanes' pivots
                if (lane >= 24) S.rs[lane] = rsqrt(S.piv[lane]);
            }
        } else if (p > 0 && p < 3 && (warp & 2)) {
            // columns from P + 8 on, with panel p - 1: rows of the tile from P + 8 and of the
            // identity up to P - 1
            const int cols = kT - (P + 8), rows = kT - (P + 8) + P;
            const int w6 = (warp >> 2) * 2 + (warp & 1);   // 0 .. 5
            for (int e = w6 * 32 + lane; e < rows * cols; e += 6 * 32) {
                const int i = e / cols, c = P + 8 + (e - i * cols);
                panel_update(S, p - 1, i < P ? kT + i : P + 8 + (i - P), c);
            }
        } else if (p == 3 && warp == 3 && lane < 24) {
            S.rs[lane] = rsqrt(S.piv[lane]);
        }
        bar_sync_n(kBarMain, kMainThreads);
        if (p < 3) {
            // the next panel's columns: tile rows P + 8 .. 31, identity rows 0 .. P + 7
            if (warp < 8) {
                const int e = warp * 32 + lane, i = e >> 3, c = P + 8 + (e & 7);
                panel_update(S, p, i < P + 8 ? kT + i : i, c);
            }
            bar_sync_n(kBarMain, kMainThreads);
        }
    }
    for (int i = warp; i < kT; i += kMainWarps)
        S.x[i][lane] = lane <= i ? S.u[kT + lane][i] * S.rs[i] : 0.0;
    bar_sync_n(kBarMain, kMainThreads);
}

__device__ void chain64(double *A, int64_t n, int nblk, double *dinv,
                        const int *__restrict__ first_col, int *F, int *U, int *ticket, int *abort_w,
                        int32_t *err) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ChainSmem &S = *reinterpret_cast<ChainSmem *>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp >= kMainWarps) {
        // ---- loads and publication (four warps, eight rows of a tile each) ----
        const int iw = warp - kMainWarps;
        const bool lead = tid == kMainThreads;
        int limit = kHelpSpins;
        // `wait`: the flag of tile (i, j) into ok and, once it is set, load(); the chain's other
        // warps stand at barrier `bar`.  While it is not set and its ticket or an earlier one is
        // unclaimed, all of them help.
        const auto wait = [&](int *ok, int i, int j, int bar, auto load) {
            bool claimed = false;   // by a CTA that is running: no more to help with
            for (;;) {
                if (lead) {
                    int got = poll_tile(&U[tile_id(i, j)], abort_w, claimed ? kSpinLimit : limit);
                    if (got == 2 && claimed) {
                        atomicAdd(&err[ERR_CHOL], 1);
                        atomicExch(abort_w, 1);
                        got = 0;
                    }
                    *ok = got;
                }
                bar_sync_n(kBarIo, 128);
                if (*ok == 1) load();
                bar_sync_n(bar, kThreads);
                if (*ok != 2) return *ok == 1;
                claimed = !help(A, n, nblk, dinv, first_col, ticket_of(nblk, i, j), F, U, ticket,
                                abort_w, err);
                limit = kHungrySpins;
            }
        };
        for (int j = 0; j < nblk; j++) {
            const int64_t c0 = (int64_t)j * kT, r0 = c0 + kT;
            const bool next = j + 1 < nblk;
            const auto load_d = [&] {
#pragma unroll
                for (int k = 0; k < 8; k++) {
                    const int64_t i = 8 * iw + k;
                    S.d[i][lane] = c0 + i < n && c0 + lane < n ? __ldcg(A + (c0 + i) * n + c0 + lane)
                                                              : (i == lane ? 1.0 : 0.0);
                }
            };
            if (!wait(&S.ok_diag, j, j, kBarDiag, load_d)) return;
            const auto load_at = [&] {
#pragma unroll
                for (int k = 0; k < 8; k += 2) {
                    const int i = 8 * iw + k;
                    const double *src = A + (r0 + i) * n + c0 + lane;
                    *reinterpret_cast<double2 *>(&S.at[lane][i]) =
                        make_double2(r0 + i < n ? __ldcg(src) : 0.0,
                                     r0 + i + 1 < n ? __ldcg(src + n) : 0.0);
                }
            };
            if (next && !wait(&S.ok_sub, j + 1, j, kBarSub, load_at)) return;
            bar_sync_n(kBarDone, kThreads);
            double *Lj = dinv + dinv_at(j);
            const double(*xt)[kLd] = S.xt[j & 1];
#pragma unroll
            for (int k = 0; k < 8; k++) {
                const int i = 8 * iw + k;
                Lj[i * 64 + lane] = S.x[i][lane];
                if (next && r0 + i < n) A[(r0 + i) * n + c0 + lane] = xt[lane][i];
            }
            bar_sync_n(kBarIo, 128);   // every store is issued before the (cumulative) releases
            if (lead) {
                st_release_gpu(&F[tile_id(j, j)], 1);
                if (next) st_release_gpu(&F[tile_id(j + 1, j)], 1);
            }
        }
        return;
    }
    // ---- compute ----
    const auto wait = [&](const int *ok, int i, int j, int bar) {   // as above
        for (;;) {
            bar_sync_n(bar, kThreads);
            if (*ok != 2) return *ok == 1;
            help(A, n, nblk, dinv, first_col, ticket_of(nblk, i, j), F, U, ticket, abort_w, err);
        }
    };
    for (int j = 0; j < nblk; j++) {
        const bool next = j + 1 < nblk;
        // the update k = j - 1 on and below the diagonal: 20 half blocks of 8 x 4 outputs,
        // five per sub-partition
        const double(*xp)[kLd] = S.xt[(j & 1) ^ 1];
        double t[2] = {0.0, 0.0};
        int tr[2], tc[2];
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int hb = warp + kMainWarps * h;
            int rb = 0, b = hb >> 1;   // block b of the lower triangle, row by row
            while (b > rb) b -= ++rb;
            tr[h] = rb * 8 + (lane >> 2);
            tc[h] = b * 8 + (hb & 1) * 4 + (lane & 3);
            if (j > 0 && hb < 20) {
#pragma unroll 8
                for (int k = 0; k < kT; k++) t[h] = fma(xp[k][tr[h]], xp[k][tc[h]], t[h]);
            }
        }
        if (!wait(&S.ok_diag, j, j, kBarDiag)) return;
#pragma unroll
        for (int h = 0; h < 2; h++)
            if (warp + kMainWarps * h < 20) S.u[tr[h]][tc[h]] = S.d[tr[h]][tc[h]] - t[h];
        for (int i = warp; i < kT; i += kMainWarps) S.u[kT + i][lane] = i == lane ? 1.0 : 0.0;
        bar_sync_n(kBarMain, kMainThreads);
        diag_factor_inv(S, (int)min((int64_t)kT, n - (int64_t)j * kT), (int64_t)j * kT, err);
        if (next) {
            if (!wait(&S.ok_sub, j + 1, j, kBarSub)) return;
            // xt = L_jj^{-1} A_{j+1,j}^T: row r of the inverse ends at column r
            double(*xt)[kLd] = S.xt[j & 1];
            const int cb = warp & 3;
            for (int rb = 3 - (warp >> 2); rb >= 0; rb -= rb == 1 ? 1 : 4) {
                const int r = rb * 8 + (lane >> 2), c = cb * 8 + (lane & 3) * 2;
                double2 o = make_double2(0.0, 0.0);
#pragma unroll 8
                for (int k = 0; k < 8 * (rb + 1); k++) {
                    const double u = S.x[r][k];
                    const double2 v = *reinterpret_cast<const double2 *>(&S.at[k][c]);
                    o.x = fma(u, v.x, o.x);
                    o.y = fma(u, v.y, o.y);
                }
                *reinterpret_cast<double2 *>(&xt[r][c]) = o;
            }
        }
        bar_sync_n(kBarDone, kThreads);
    }
}

__global__ void __launch_bounds__(kThreads, 1) k_chol_f64(double *A, int64_t n, int nblk,
                                                          double *dinv,
                                                          const int *__restrict__ first_col,
                                                          int *flags, int32_t *err) {
    __shared__ int s_task;
    const int ntask = nblk * (nblk + 1) / 2;
    int *F = flags, *U = flags + ntask, *ticket = flags + 2 * ntask, *abort_w = ticket + 1;
    const int tid = threadIdx.x;
    if (tid == 0) s_task = atomicAdd(ticket + 2, 1);
    __syncthreads();
    if (s_task == 0) {
        chain64(A, n, nblk, dinv, first_col, F, U, ticket, abort_w, err);
        return;
    }
    __syncthreads();   // s_task is read before the first ticket is stored in it
    int j = 0, first = 0;   // column of the last ticket and the first ticket of that column
    const auto row_of = [&](int t) {   // (t in column j from here on)
        while (t - first >= nblk - j) first += nblk - j++;
        return j + (t - first);
    };
    for (;;) {
        // Thread 0 draws until it holds a task inside the profile (the others are zero and never
        // read) and stores that one: every task then passes a barrier between the reads of
        // s_task and the next store to it.
        if (tid == 0) {
            int t = atomicAdd(ticket, 1);
            while (first_col && t < ntask) {
                const int i = row_of(t);
                if (i <= j + 1 || j >= first_col[i]) break;
                t = atomicAdd(ticket, 1);
            }
            s_task = t;
        }
        __syncthreads();
        const int t = s_task;
        if (t >= ntask) return;
        const int i = row_of(t);
        if (!tile_task(A, n, nblk, dinv, first_col, i, j, F, U, abort_w, err)) return;
    }
}

// the rest of the 64 x 64 diagonal inverses: block b's lower left quarter -X22 L21 X11, zero
// above it, and the identity in the second half of a last block of at most 32 columns
__global__ void __launch_bounds__(256) k_join_dinv(const double *__restrict__ A, int64_t n,
                                                   int nblk, double *dinv) {
    __shared__ double x1[kT][kT + 1], x2[kT][kT + 1], l[kT][kT + 1], t[kT][kT + 1];
    const int b = blockIdx.x;
    const bool half = 2 * b + 1 >= nblk;   // no second tile
    double *D = dinv + (int64_t)b * 64 * 64;
    const int64_t r0 = (int64_t)b * 64 + kT, c0 = (int64_t)b * 64;
    for (int e = threadIdx.x; e < kT * kT; e += 256) {
        const int i = e >> 5, q = e & 31;
        x1[i][q] = D[i * 64 + q];
        x2[i][q] = half ? (i == q ? 1.0 : 0.0) : D[(kT + i) * 64 + kT + q];
        l[i][q] = r0 + i < n ? A[(r0 + i) * n + c0 + q] : 0.0;
        D[i * 64 + kT + q] = 0.0;
        if (half) D[(kT + i) * 64 + kT + q] = i == q ? 1.0 : 0.0;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < kT * kT; e += 256) {
        const int i = e >> 5, q = e & 31;
        double s = 0.0;
        for (int k = q; k < kT; k++) s = fma(l[i][k], x1[k][q], s);   // X11 lower triangular
        t[i][q] = s;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < kT * kT; e += 256) {
        const int i = e >> 5, q = e & 31;
        double s = 0.0;
        for (int k = 0; k <= i; k++) s = fma(x2[i][k], t[k][q], s);
        D[(kT + i) * 64 + q] = -s;
    }
}

}  // namespace

int chol_f64(double *A, int64_t n, double *dinv, const int *first_col, int *flags, int32_t *err,
             cudaStream_t s, int *launches) {
    if (n <= 0) return FEM3_OK;
    int sms = 0;
    FEM3_CUDA(device_sms(&sms));
    FEM3_CUDA(device_smem((const void *)k_chol_f64, kSmemBytes));
    const int nblk = (int)((n + kT - 1) / kT);
    const int ntask = nblk * (nblk + 1) / 2;
    FEM3_CUDA(cudaMemsetAsync(flags, 0, sizeof(int) * chol_f64_flags(n), s));
    // one CTA per SM: the chain CTA gets an SM of its own
    k_chol_f64<<<std::min(ntask + 1, std::max(sms, 2)), kThreads, kSmemBytes, s>>>(
        A, n, nblk, dinv, first_col, flags, err);
    k_join_dinv<<<(unsigned)((nblk + 1) / 2), 256, 0, s>>>(A, n, nblk, dinv);
    *launches += 2;
    FEM3_CUDA(cudaGetLastError());
    return FEM3_OK;
}

}  // namespace fem3
