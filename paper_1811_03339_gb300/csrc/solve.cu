// Load vector, dense SPD solve and iterative refinement.
//
//  - b = M f with the P1 mass matrix (|T|/20 (1 + delta_ab) per tet), the weak
//    right-hand side (f, v) of Section 3.
//  - Cholesky A = L L^T: by tile tasks (FP32 here, FP64 in chol_f64.cu) or blocked on the
//    tensor cores (chol_tc.cu); row-major storage: the tiles below the diagonal in A's
//    lower triangle, each 64 x 64 diagonal block as its inverse L_jj^{-1} (all the solves
//    use).
//  - Triangular solves: trisolve.cu.
//  - Refinement for the mixed forms: r = b - A u with A u applied at FP64 accuracy
//    (operator.cu), the correction solved with the FP32 factor.
#include <math.h>

#include <algorithm>
#include <vector>

#include "chol_f64.cuh"
#include "fem3_impl.cuh"

namespace fem3 {

namespace {

__global__ void k_load(const int32_t *__restrict__ tets, const double *__restrict__ vol,
                       const int32_t *__restrict__ dof, int64_t n_tets, int64_t n_nodes,
                       int64_t n_dof, const double *__restrict__ f, int nrhs, double *b) {
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= n_tets) return;
    int32_t v[4];
    for (int k = 0; k < 4; k++) v[k] = tets[4 * t + k];
    double c = vol[t] / 20.0;
    for (int r = 0; r < nrhs; r++) {
        const double *fr = f + (int64_t)r * n_nodes;
        double fv[4], fs = 0;
        for (int k = 0; k < 4; k++) { fv[k] = fr[v[k]]; fs += fv[k]; }
        for (int k = 0; k < 4; k++) {
            int32_t j = dof[v[k]];
            if (j >= 0) atomicAdd(&b[(int64_t)r * n_dof + j], c * (fs + fv[k]));
        }
    }
}

__global__ void k_load_T(const int32_t *__restrict__ tets, const double *__restrict__ vol,
                         const int32_t *__restrict__ dof, int64_t n_tets,
                         const double *__restrict__ lam, double *out) {
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= n_tets) return;
    int32_t v[4];
    double lv[4], ls = 0;
    for (int k = 0; k < 4; k++) {
        v[k] = tets[4 * t + k];
        int32_t j = dof[v[k]];
        lv[k] = j >= 0 ? lam[j] : 0.0;
        ls += lv[k];
    }
    double c = vol[t] / 20.0;
    for (int k = 0; k < 4; k++) atomicAdd(&out[v[k]], c * (ls + lv[k]));
}

#include "chol_smem.cuh"

// ---------------------------------------------------------------------------------
// Tile-task Cholesky of the FP32 factor in one launch, 64 x 64 tiles (the FP64 form has its
// own, chol_f64.cu).  CTA 0 runs the diagonal chain: for each block
// column j it applies the last update (k = j - 1) to the diagonal tile, factors it
// (L_jj and L_jj^{-1}), solves the tile below it, L_{j+1,j} = A_{j+1,j} L_jj^{-T}, and
// keeps that tile in shared memory for the next diagonal update, so the critical path
// never leaves one SM.  The other CTAs take tasks W(i, j) over the lower 64 x 64 tiles
// from an atomic ticket, column by column: W(i, j) subtracts L_ik L_jk^T for k < j (for a
// diagonal tile k < j - 1), each as soon as tiles (i, k) and (j, k) are final; the
// diagonal and sub-diagonal tiles are then stored for the chain ("updated" flag U),
// every other tile is solved with L_jj^{-1} once the chain has published it and stored
// as final (flag F).  Every task depends only on tiles of earlier columns (or, for the
// solve, on the chain's step j), and tickets are taken in column order, so the earliest
// unfinished claimed task always proceeds and the launch needs no co-residency.  Waits
// are bounded; a wait that expires sets the abort word, which every other wait also
// watches, and records ERR_CHOL.
// flags: F [0, ntask), U [ntask, 2 ntask), ticket [2 ntask], abort word [2 ntask + 1];
// all zero at launch.
// ---------------------------------------------------------------------------------
constexpr int kTileLd = NB + 4;
constexpr int kCholTilesSmem = 4 * NB * kTileLd;   // elements of dynamic shared memory

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

// Tile loads, 512 threads: warp w reads rows 4w .. 4w + 3, lanes over the columns (each
// load instruction covers 32 consecutive entries of one row), element e = 2k + h of a
// thread is (row 4w + k, column lane + 32h).  L2 loads: the tile was written by another CTA
// of the same launch.
__device__ __forceinline__ void tile_regs(const float *src, int64_t ld, int64_t rows, float v[8]) {
    const int lane = threadIdx.x & 31, r0 = (threadIdx.x >> 5) * 4;
#pragma unroll
    for (int k = 0; k < 4; k++)
#pragma unroll
        for (int h = 0; h < 2; h++)
            v[2 * k + h] = r0 + k < rows ? __ldcg(src + (int64_t)(r0 + k) * ld + lane + 32 * h)
                                         : 0.f;
}
// dst[c][r] = the loaded tile's entry (r, c)
__device__ __forceinline__ void tile_store_T(const float v[8], float (*dst)[kTileLd]) {
    const int lane = threadIdx.x & 31, r0 = (threadIdx.x >> 5) * 4;
#pragma unroll
    for (int k = 0; k < 4; k++)
#pragma unroll
        for (int h = 0; h < 2; h++) dst[lane + 32 * h][r0 + k] = v[2 * k + h];
}
// dst[c][r] = src[r * ld + c] (r < rows, else 0), c < 64
__device__ __forceinline__ void load_tile_T(const float *src, int64_t ld, int64_t rows,
                                            float (*dst)[kTileLd]) {
    float v[8];
    tile_regs(src, ld, rows, v);
    tile_store_T(v, dst);
}

// acc[p][q] += sgn * sum_c bi[c][ty*2+p] bj[c][tx*4+q] (operands in transposed layout).
// The 64-term product is summed from zero and added to acc once: summing into acc
// directly would round every term at the magnitude of the (much larger) tile entry,
// which made the FP32 factor several times less accurate.
template <bool SUB>
__device__ __forceinline__ void tile_gemm_T(float acc[2][4], const float (*bi)[kTileLd],
                                            const float (*bj)[kTileLd], int tx, int ty) {
    float t[2][4];
#pragma unroll
    for (int p = 0; p < 2; p++)
#pragma unroll
        for (int q = 0; q < 4; q++) t[p][q] = 0.f;
#pragma unroll 8
    for (int c = 0; c < NB; c++) {
        float u[2], v[4];
        lds2(&bi[c][ty * 2], u);
        lds4(&bj[c][tx * 4], v);
#pragma unroll
        for (int p = 0; p < 2; p++)
#pragma unroll
            for (int q = 0; q < 4; q++) t[p][q] = fma(u[p], v[q], t[p][q]);
    }
#pragma unroll
    for (int p = 0; p < 2; p++)
#pragma unroll
        for (int q = 0; q < 4; q++) acc[p][q] = SUB ? acc[p][q] - t[p][q] : acc[p][q] + t[p][q];
}

// load tile (r0, c0) of A into acc (rows/columns beyond n: identity on the diagonal tile)
__device__ __forceinline__ void load_acc(const float *A, int64_t n, int64_t r0, int64_t c0,
                                         bool diag, float acc[2][4], int tx, int ty) {
#pragma unroll
    for (int p = 0; p < 2; p++)
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const int r = ty * 2 + p, c = tx * 4 + q;
            acc[p][q] = (r0 + r < n && c0 + c < n) ? __ldcg(&A[(r0 + r) * n + c0 + c])
                                                   : ((diag && r == c) ? 1.f : 0.f);
        }
}

__device__ __forceinline__ void store_acc(float *A, int64_t n, int64_t r0, int64_t c0,
                                          const float acc[2][4], int tx, int ty) {
#pragma unroll
    for (int p = 0; p < 2; p++) {
        const int r = ty * 2 + p;
        if (r0 + r >= n) continue;
#pragma unroll
        for (int q = 0; q < 4; q++)
            if (c0 + tx * 4 + q < n) A[(r0 + r) * n + c0 + tx * 4 + q] = acc[p][q];
    }
}

// all threads' global stores of a tile are visible before its flag: the barrier orders
// them before thread 0's release, which is cumulative
__device__ __forceinline__ void publish(int *f) {
    __syncthreads();
    if (threadIdx.x == 0) st_release_gpu(f, 1);
}

__device__ void chol_chain(float *A, int64_t n, int nblk, float *dinv, int *F, int *U, int *abort_w,
                           int32_t *err, unsigned char *smem_raw) {
    float (*b0)[kTileLd] = reinterpret_cast<float (*)[kTileLd]>(smem_raw);
    float (*b1)[kTileLd] = b0 + NB;
    float (*xt)[kTileLd] = b1 + NB;   // L_{j+1,j}^T (from the sub-solve, for the next update)
    float (*at)[kTileLd] = xt + NB;   // A_{j+1,j}^T as the sub-solve reads it
    float (*a_s)[NB + 1] = reinterpret_cast<float (*)[NB + 1]>(&b0[0][0]);
    float (*x_s)[NB + 1] = reinterpret_cast<float (*)[NB + 1]>(&b1[0][0]);
    __shared__ int s_ok, s_pre;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    float acc[2][4];   // the diagonal tile A~_jj of the coming step (loaded one step ahead)
    if (tid == 0) s_ok = wait_tile(&U[tile_id(0, 0)], abort_w, err);
    __syncthreads();
    if (!s_ok) return;
    load_acc(A, n, 0, 0, true, acc, tx, ty);
    for (int j = 0; j < nblk; j++) {
        const int64_t c0 = (int64_t)j * NB, r0 = c0 + NB;
        const bool next = j + 1 < nblk;
        if (j > 0) tile_gemm_T<true>(acc, xt, xt, tx, ty);   // the update k = j - 1
#pragma unroll
        for (int p = 0; p < 2; p++)
#pragma unroll
            for (int q = 0; q < 4; q++) a_s[ty * 2 + p][tx * 4 + q] = acc[p][q];
        __syncthreads();
        potrf_inv_smem(a_s, x_s, (int)min((int64_t)NB, n - c0), c0, err);
        if (next) {
            // L_{j+1,j} = A~_{j+1,j} L_jj^{-T}, computed transposed: xt = L_jj^{-1} A~_{j+1,j}^T
            // the next diagonal tile's flag is looked at now, beside this wait, and once more
            // after the sub-solve if it was not set yet
            if (tid == 0) s_ok = wait_tile(&U[tile_id(j + 1, j)], abort_w, err);
            if (tid == 32) s_pre = ld_acquire_gpu(&U[tile_id(j + 1, j + 1)]) != 0;
            __syncthreads();
            if (!s_ok) return;
            load_tile_T(A + r0 * n + c0, n, n - r0, at);   // at[k][r] = A_{j+1,j}[r][k]
            __syncthreads();
            float o[2][4];
#pragma unroll
            for (int p = 0; p < 2; p++)
#pragma unroll
                for (int q = 0; q < 4; q++) o[p][q] = 0.f;
#pragma unroll 8
            for (int k = 0; k < NB; k++) {
                float v[4];
                lds4(&at[k][tx * 4], v);
                const float u0 = x_s[ty * 2][k], u1 = x_s[ty * 2 + 1][k];
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    o[0][q] = fma(u0, v[q], o[0][q]);
                    o[1][q] = fma(u1, v[q], o[1][q]);
                }
            }
            // o[p][q] = L_{j+1,j}[tx*4+q][ty*2+p]; xt was last read by this step's update
#pragma unroll
            for (int p = 0; p < 2; p++) {
                float *dst = &xt[ty * 2 + p][tx * 4];
                *reinterpret_cast<float4 *>(dst) = make_float4(o[p][0], o[p][1], o[p][2], o[p][3]);
            }
            // the next diagonal tile goes into registers now if it is ready.  It is not
            // waited for here: its task may be queued behind tasks of this column that
            // wait for F(j, j), so the wait comes after the publication below.
            if (tid == 0 && !s_pre) s_pre = ld_acquire_gpu(&U[tile_id(j + 1, j + 1)]) != 0;
        }
        __syncthreads();   // xt complete; the next diagonal tile's flag seen
        const bool pre = next && s_pre;
        if (pre) load_acc(A, n, r0, r0, true, acc, tx, ty);
        // L_jj^{-1} into dinv, L_{j+1,j} into A: rows of 64, coalesced.  L_jj itself is not
        // stored: every solve with the factor applies L_jj^{-1}, so A's diagonal tiles keep
        // their last update.
        float *Lj = dinv + (int64_t)j * NB * NB;
        for (int e = tid; e < NB * NB; e += blockDim.x) {
            const int i = e >> 6, c = e & 63;
            Lj[e] = x_s[i][c];
            if (next && r0 + i < n) A[(r0 + i) * n + c0 + c] = xt[c][i];
        }
        __syncthreads();   // every store is issued before the (cumulative) releases
        if (tid == 0) {
            st_release_gpu(&F[tile_id(j, j)], 1);
            if (next) st_release_gpu(&F[tile_id(j + 1, j)], 1);
        }
        if (next && !pre) {
            if (tid == 0) s_ok = wait_tile(&U[tile_id(j + 1, j + 1)], abort_w, err);
            __syncthreads();
            if (!s_ok) return;
            load_acc(A, n, r0, r0, true, acc, tx, ty);
        }
    }
}

__global__ void __launch_bounds__(512, 1) k_chol_tiles(float *A, int64_t n, int nblk, float *dinv,
                                                       int *flags, int32_t *err) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float (*b0)[kTileLd] = reinterpret_cast<float (*)[kTileLd]>(smem_raw);
    float (*b1)[kTileLd] = b0 + NB;
    __shared__ int s_task, s_ok, s_fa, s_fb, s_pa[2], s_pb[2];
    const int ntask = nblk * (nblk + 1) / 2;
    int *F = flags, *U = flags + ntask, *ticket = flags + 2 * ntask, *abort_w = ticket + 1;
    if (blockIdx.x == 0) {
        chol_chain(A, n, nblk, dinv, F, U, abort_w, err, smem_raw);
        return;
    }
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;   // rows ty*2+{0,1}, cols tx*4+{0..3}
    for (;;) {
        if (tid == 0) s_task = atomicAdd(ticket, 1);
        __syncthreads();
        const int t = s_task;
        if (t >= ntask) return;
        int j = 0, rem = t;
        while (rem >= nblk - j) { rem -= nblk - j; j++; }
        const int i = j + rem;
        const int64_t r0 = (int64_t)i * NB, c0 = (int64_t)j * NB;
        const int64_t rows_i = n - r0;
        const int kmax = i == j ? max(j - 1, 0) : j;   // the chain applies k = j - 1 to (j, j)
        float acc[2][4];
        load_acc(A, n, r0, c0, false, acc, tx, ty);
        // Updates k = 0 .. kmax-1, pipelined: the tiles L_ik, L_jk of update k + 1 are
        // loaded into registers while update k's product runs (when their flags are
        // already set; otherwise after it, with a blocking wait), and stored into the other
        // pair of shared tiles.  Threads 0 and 32 read the two flags at the same time.
        float va[8], vb[8];
        bool have = false;   // va / vb hold the tiles of update k
        for (int k = 0; k < kmax; k++) {
            float (*ta)[kTileLd] = b0 + (k & 1) * 2 * NB;
            float (*tb)[kTileLd] = ta + NB;
            if (!have) {
                if (tid == 0) s_fa = wait_tile(&F[tile_id(i, k)], abort_w, err);
                if (tid == 32) s_fb = wait_tile(&F[tile_id(j, k)], abort_w, err);
                __syncthreads();
                if (!(s_fa && s_fb)) return;
                tile_regs(A + r0 * n + (int64_t)k * NB, n, rows_i, va);
                if (i != j) tile_regs(A + c0 * n + (int64_t)k * NB, n, n - c0, vb);
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
                tile_regs(A + r0 * n + (int64_t)(k + 1) * NB, n, rows_i, va);
                if (i != j) tile_regs(A + c0 * n + (int64_t)(k + 1) * NB, n, n - c0, vb);
            }
            tile_gemm_T<true>(acc, ta, i == j ? ta : tb, tx, ty);
        }
        __syncthreads();   // the last product is done before the shared tiles are reused
        if (i <= j + 1) {
            // diagonal or sub-diagonal tile: the chain finishes it
            store_acc(A, n, r0, c0, acc, tx, ty);
            publish(&U[tile_id(i, j)]);
            continue;
        }
        // L_ij = A_ij L_jj^{-T}: o[p][q] = sum_c acc[ty*2+p][c] Linv[tx*4+q][c]
        float (*a)[NB + 1] = reinterpret_cast<float (*)[NB + 1]>(smem_raw);   // overlays b0 only
#pragma unroll
        for (int p = 0; p < 2; p++)
#pragma unroll
            for (int q = 0; q < 4; q++) a[ty * 2 + p][tx * 4 + q] = acc[p][q];
        if (tid == 0) s_ok = wait_tile(&F[tile_id(j, j)], abort_w, err);
        __syncthreads();
        if (!s_ok) return;
        load_tile_T(dinv + (int64_t)j * NB * NB, NB, NB, b1);   // b1[c][q] = Linv[q][c]
        __syncthreads();
        float o[2][4];
#pragma unroll
        for (int p = 0; p < 2; p++)
#pragma unroll
            for (int q = 0; q < 4; q++) o[p][q] = 0.f;
#pragma unroll 8
        for (int c = 0; c < NB; c++) {
            float v[4];
            lds4(&b1[c][tx * 4], v);
            const float u0 = a[ty * 2][c], u1 = a[ty * 2 + 1][c];
#pragma unroll
            for (int q = 0; q < 4; q++) {
                o[0][q] = fma(u0, v[q], o[0][q]);
                o[1][q] = fma(u1, v[q], o[1][q]);
            }
        }
        store_acc(A, n, r0, c0, o, tx, ty);
        publish(&F[tile_id(i, j)]);
    }
}

int chol_tiles(float *A, int64_t n, cudaStream_t s, Mesh *m) {
    if (n <= 0) return FEM3_OK;
    const int nblk = (int)((n + NB - 1) / NB);
    const int ntask = nblk * (nblk + 1) / 2;
    int sms = 0;
    FEM3_CUDA(device_sms(&sms));
    FEM3_CUDA(cudaMemsetAsync(m->chol_flags, 0, sizeof(int32_t) * (2 * ntask + 2), s));
    // one CTA per SM: the chain CTA gets an SM of its own
    const int grid = std::min(ntask + 1, std::max(sms, 2));
    FEM3_CUDA(device_smem((const void *)k_chol_tiles, kCholTilesSmem * sizeof(float)));
    kc_begin(m, KC_FACTOR);
    k_chol_tiles<<<grid, 512, kCholTilesSmem * sizeof(float), s>>>(
        A, n, nblk, reinterpret_cast<float *>(m->dinv), m->chol_flags, m->err);
    kc_end(m, KC_FACTOR);
    note_launch(m);
    FEM3_CUDA(cudaGetLastError());
    return FEM3_OK;
}

// Per-axis forms sum_g w_g ((L lam)(R u) + (R lam)(L u)) (adjoint), one CTA per bin: the bin's u
// and lam in shared memory, thread = (Gauss point, slice of the template rows), all sums and
// products in FP64 whatever the form, so that dK scales with u and lam over the FP64 range.
// Bound: the FP64 pipe, which holds a warp's instruction for 16 clocks of the SM.  A nonzero
// table entry takes three (the pair's sum, two multiply-adds): the pair is converted by its bits,
// as f32 -> f64 conversions run at the FP64 rate, and entries that are zero for a warp's 32
// points (sorted along the axis) are skipped.  Measured, GB300: the three axes of the 16^3 cube
// 0.95 ms with conversion instructions and nothing skipped; the 16^3 gradient 4.82 ms so, 4.85 ms with
// double-float FP32 sums, which keep 2^-48 a term and not the range (nothing below 2^-126 or from
// 2^128 on, 24 bits below 2^-74).
constexpr int kFormSlices = 4, kFormPoints = 64, kFormRows = 4;   // rows of a slice in flight
__global__ void __launch_bounds__(kFormSlices *kFormPoints) k_axis_form(
    const float2 *__restrict__ tabL, const float2 *__restrict__ tabR,
    const int32_t *__restrict__ gp_off, const int32_t *__restrict__ dof_off,
    const int32_t *__restrict__ dof_idx, const int64_t *__restrict__ tab_off,
    const int32_t *__restrict__ tab_ld, const double *__restrict__ w_slot,
    const double *__restrict__ u, const double *__restrict__ lam, double *out) {
    extern __shared__ __align__(16) double2 sm_form[];   // (u, lam) per row
    __shared__ double part[kFormSlices][4][kFormPoints];
    __shared__ double red[kFormPoints / 32];
    const int bin = blockIdx.x;
    const int D = dof_off[bin + 1] - dof_off[bin];
    const int g0 = gp_off[bin], G = gp_off[bin + 1] - g0;
    if (D == 0 || G == 0) return;
    const int ld = tab_ld[bin];
    const float2 *L = tabL + tab_off[bin], *R = tabR + tab_off[bin];
    const int32_t *dofs = dof_idx + dof_off[bin];
    for (int c = threadIdx.x; c < D; c += blockDim.x)
        sm_form[c] = make_double2(u[dofs[c]], lam[dofs[c]]);
    __syncthreads();
    const int p = threadIdx.x % kFormPoints, q = threadIdx.x / kFormPoints;
    double acc = 0;
    for (int r0 = 0; r0 < G; r0 += kFormPoints) {
        const int r = r0 + p;
        double t[4] = {0.0, 0.0, 0.0, 0.0};   // Lu, Ru, Llam, Rlam
        if (r < G) {
            for (int c0 = q; c0 < D; c0 += kFormSlices * kFormRows) {
                float2 a[kFormRows], b[kFormRows];
#pragma unroll
                for (int k = 0; k < kFormRows; k++) {
                    const int c = c0 + kFormSlices * k;
                    a[k] = b[k] = make_float2(0.f, 0.f);
                    if (c < D) {
                        a[k] = __ldg(L + (int64_t)c * ld + r);
                        b[k] = __ldg(R + (int64_t)c * ld + r);
                    }
                }
#pragma unroll
                for (int k = 0; k < kFormRows; k++) {
                    const int c = c0 + kFormSlices * k;
                    if (a[k].x != 0.f || a[k].y != 0.f) {
                        const double2 v = sm_form[c];
                        const double e = f32_to_f64_exact(a[k].x) + f32_to_f64_exact(a[k].y);
                        t[0] = fma(e, v.x, t[0]);
                        t[2] = fma(e, v.y, t[2]);
                    }
                    if (b[k].x != 0.f || b[k].y != 0.f) {
                        const double2 v = sm_form[c];
                        const double e = f32_to_f64_exact(b[k].x) + f32_to_f64_exact(b[k].y);
                        t[1] = fma(e, v.x, t[1]);
                        t[3] = fma(e, v.y, t[3]);
                    }
                }
            }
        }
#pragma unroll
        for (int k = 0; k < 4; k++) part[q][k][p] = t[k];
        __syncthreads();
        if (q == 0 && r < G) {
#pragma unroll
            for (int k = 0; k < 4; k++)
                t[k] = (part[0][k][p] + part[1][k][p]) + (part[2][k][p] + part[3][k][p]);
            acc = fma(w_slot[g0 + r], fma(t[2], t[1], t[3] * t[0]), acc);
        }
        __syncthreads();
    }
    if (q == 0) {
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if ((p & 31) == 0) red[p >> 5] = acc;
    }
    __syncthreads();
    if (threadIdx.x == 0) atomicAdd(out, red[0] + red[1]);
}

// (r may be Au)
__global__ void k_residual_cols(const double *__restrict__ b, const double *Au, int64_t n,
                                double *r, double *norms) {
    const int c = blockIdx.y;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double rr = 0, bb = 0;
    if (i < n) {
        const int64_t k = (int64_t)c * n + i;
        const double v = b[k] - Au[k];
        r[k] = v;
        rr = v * v;
        bb = b[k] * b[k];
    }
    for (int o = 16; o > 0; o >>= 1) {
        rr += __shfl_down_sync(0xffffffffu, rr, o);
        bb += __shfl_down_sync(0xffffffffu, bb, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&norms[2 * c], rr);
        atomicAdd(&norms[2 * c + 1], bb);
    }
}

// r -= Ad (where given) with the norms of r and b per column; where Ac, A times the carries, is
// given, the norms of r + Ac in norms[kTrueSlot + c]
constexpr int kTrueSlot = 64;   // of Mesh::norms
constexpr double kCarryScale = 0x1p48;   // carries are stored times this
__global__ void k_residual_update_cols(const double *__restrict__ b, const double *__restrict__ Ad,
                                       const double *__restrict__ Ac, int64_t n, double *r,
                                       double *norms) {
    const int c = blockIdx.y;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double rr = 0, bb = 0, tt = 0;
    if (i < n) {
        const int64_t k = (int64_t)c * n + i;
        double v = r[k];
        if (Ad) r[k] = v = v - Ad[k];
        rr = v * v;
        bb = b[k] * b[k];
        if (Ac) {
            const double t = fma(Ac[k], 1.0 / kCarryScale, v);
            tt = t * t;
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        rr += __shfl_down_sync(0xffffffffu, rr, o);
        bb += __shfl_down_sync(0xffffffffu, bb, o);
        tt += __shfl_down_sync(0xffffffffu, tt, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&norms[2 * c], rr);
        atomicAdd(&norms[2 * c + 1], bb);
        if (Ac) atomicAdd(&norms[kTrueSlot + c], tt);
    }
}

__global__ void k_to_f32(const double *__restrict__ a, float *b, int64_t n) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = (float)a[i];
}
// u + c += d: u takes the rounded sum, c what it lost (TwoSum: u + y = s + e exactly), or nothing
// if the residual is formed from u anew (keep = false)
__global__ void k_add_correction(const float *__restrict__ d, double *u, float *c, int64_t n, bool keep) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double y = (double)d[i] + (double)c[i] * (1.0 / kCarryScale), u0 = u[i];
    const double s = u0 + y, z = s - u0;
    u[i] = s;
    c[i] = keep ? (float)(((u0 - (s - z)) + (y - z)) * kCarryScale) : 0.f;
}
__global__ void k_f32_to_f64(const float *__restrict__ a, double *b, int64_t n) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = (double)a[i];
}

__global__ void k_sub(const double *__restrict__ a, const double *__restrict__ b, double *c,
                      int64_t n) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) c[i] = a[i] - b[i];
}

inline unsigned g256(int64_t n) { return (unsigned)(n > 0 ? (n + 255) / 256 : 1); }

}  // namespace

// upper triangle := transpose of the lower triangle (n x n row-major); a CTA copies one
// 32 x 32 tile of the lower triangle through shared memory (both sides along rows)
__global__ void __launch_bounds__(256) k_sym_from_lower(double *A, int64_t n) {
    __shared__ double t[32][33];
    if (blockIdx.x > blockIdx.y) return;
    const int64_t r0 = 32 * (int64_t)blockIdx.y, c0 = 32 * (int64_t)blockIdx.x;
    const int x = threadIdx.x & 31;
    for (int y = threadIdx.x >> 5; y < 32; y += 8)
        if (r0 + y < n && c0 + x < n) t[y][x] = A[(r0 + y) * n + c0 + x];
    __syncthreads();
    for (int y = threadIdx.x >> 5; y < 32; y += 8)
        if (c0 + y < n && r0 + x < n && r0 + x > c0 + y) A[(c0 + y) * n + r0 + x] = t[x][y];
}

int sym_from_lower(double *A, int64_t n, cudaStream_t s) {
    if (n <= 0) return FEM3_OK;
    const unsigned g = (unsigned)((n + 31) / 32);
    k_sym_from_lower<<<dim3(g, g), 256, 0, s>>>(A, n);
    FEM3_CUDA(cudaGetLastError());
    return FEM3_OK;
}

int f32_to_f64(const float *a, double *b, int64_t n, cudaStream_t s) {
    k_f32_to_f64<<<g256(n), 256, 0, s>>>(a, b, n);
    FEM3_CUDA(cudaGetLastError());
    return FEM3_OK;
}

int sub_vec(const double *a, const double *b, double *c, int64_t n, cudaStream_t s) {
    k_sub<<<g256(n), 256, 0, s>>>(a, b, c, n);
    FEM3_CUDA(cudaGetLastError());
    return FEM3_OK;
}

int load_vector(Mesh *m, const double *f_d, int nrhs, double *b_d) {
    cudaStream_t s = m->stream;
    FEM3_CUDA(cudaMemsetAsync(b_d, 0, sizeof(double) * m->n_dof * nrhs, s));
    k_load<<<g256(m->n_tets), 256, 0, s>>>(m->tets, m->vol, m->dof, m->n_tets, m->n_nodes, m->n_dof,
                                            f_d, nrhs, b_d);
    note_launch(m);
    FEM3_CUDA(cudaGetLastError());
    return FEM3_OK;
}

int load_vector_T(Mesh *m, const double *lam_d, double *out_d) {
    cudaStream_t s = m->stream;
    FEM3_CUDA(cudaMemsetAsync(out_d, 0, sizeof(double) * m->n_nodes, s));
    k_load_T<<<g256(m->n_tets), 256, 0, s>>>(m->tets, m->vol, m->dof, m->n_tets, lam_d, out_d);
    note_launch(m);
    FEM3_CUDA(cudaGetLastError());
    return FEM3_OK;
}

// FP32 factorisations of at least this order take the blocked factorisation with
// tensor-core trailing updates (chol_tc.cu); smaller ones the one-launch tile-task
// factorisation, whose diagonal chain is the shorter critical path there.
constexpr int64_t kCholTcMinN = 4096;

bool factor_on_tc(const Mesh *m) {
    return m->chol_tc_opt > 0 || (m->chol_tc_opt == 0 && m->n_dof >= kCholTcMinN);
}

// The refinement's operator (a contraction that fills the chip) is built beside the tile-task
// factorisation (a serial chain that leaves most of it idle): a TF32 x 3 step after against
// before, 658 -> 646 us at n = 27, 1,012 -> 993 at 343, 2,559 -> 2,308 at 1,728.  Not beside the blocked factorisation: its trailing updates take an SM's whole shared memory
// each, so the critical chain waited for the operator's CTAs to drain (24^3 step 30.6 ms
// with, 30.3 ms without).  A profiled mesh times its launches one at a time.
static bool op_beside_factor(const Mesh *m) {
    return !m->profile && !factor_on_tc(m);
}

// the FP32 factor; on return m->stream waits for everything enqueued on cx's streams
static int factor_mixed(Mesh *m, SideCtx *cx) {
    cudaStream_t s = m->stream;
    const bool tc = factor_on_tc(m);
    const bool beside = op_beside_factor(m) && !m->op_ready;
    if (beside) {
        FEM3_TRY(op_prepare(m, true));
        FEM3_CUDA(cudaEventRecord(cx->op_done, s));
        FEM3_CUDA(cudaStreamWaitEvent(cx->op, cx->op_done, 0));
    }
    int st;
    if (tc) {
        st = chol_tc(m, cx, m->A32, m->n_dof);
        m->chol_tc_used = st == FEM3_OK;
    } else {
        st = chol_tiles(m->A32, m->n_dof, s, m);
    }
    if (beside) {   // enqueued after the factorisation, whose CTAs are to be placed first
        m->stream = cx->op;
        const int so = op_build(m);
        m->stream = s;
        if (st == FEM3_OK) st = so;
    }
    if (st == FEM3_OK) st = tri_prepare<float>(m, m->A32, m->n_dof);
    if (beside) {
        cudaError_t e = cudaEventRecord(cx->op_done, cx->op);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(s, cx->op_done, 0);
        if (e != cudaSuccess && st == FEM3_OK) st = cuda_error(e, "operator join");
    }
    return st;
}

int factor(Mesh *m) {
    m->chol_tc_used = false;
    if (m->precision == FEM3_FP64) {
        // the residual's operator, before the factor takes the matrix's place
        if (!m->integer_order && !m->nonsym) FEM3_TRY(op_from_dense(m, m->A64));
        int launches = 0;
        kc_begin(m, KC_FACTOR);
        FEM3_TRY(chol_f64(m->A64, m->n_dof, reinterpret_cast<double *>(m->dinv),
                          m->integer_order ? m->p1_first : nullptr, m->chol_flags, m->err,
                          m->stream, &launches));
        kc_end(m, KC_FACTOR);
        m->launches += launches;
        return tri_prepare<double>(m, m->A64, m->n_dof);
    }
    SideCtx *cx = m->lent;
    if (!cx) FEM3_TRY(side_acquire(&cx));
    const int st = factor_mixed(m, cx);
    if (!m->lent) side_release(cx);
    return st;
}

int axis_forms(Mesh *m, const double *u_d, const double *lam_d, double out[3]) {
    cudaStream_t s = m->stream;
    FEM3_CUDA(device_smem((const void *)k_axis_form, sizeof(double2) * kMaxBinItems));
    FEM3_CUDA(cudaMemsetAsync(m->norms, 0, sizeof(double) * 3, s));
    for (int axis = 0; axis < 3; axis++) {
        AxisBins &B = m->bins[axis];
        const size_t sh = sizeof(double2) * std::max(1, B.max_dof);
        k_axis_form<<<B.n_bins, kFormSlices * kFormPoints, sh, s>>>(
            m->tabL[axis], m->tabR[axis], B.gp_off, B.dof_off, B.dof_idx, B.tab_off, B.tab_ld,
            B.w_slot, u_d, lam_d, m->norms + axis);
        note_launch(m);
    }
    FEM3_CUDA(cudaMemcpyAsync(m->h_norms, m->norms, sizeof(double) * 3, cudaMemcpyDeviceToHost, s));
    FEM3_CUDA(cudaStreamSynchronize(s));
    for (int a = 0; a < 3; a++) out[a] = m->s[a] * m->h_norms[a];
    return FEM3_OK;
}

int solve_direct(Mesh *m, const double *b_d, int nrhs, double *u_d) {
    cudaStream_t s = m->stream;
    const int64_t n = m->n_dof;
    FEM3_CUDA(cudaMemcpyAsync(u_d, b_d, sizeof(double) * n * nrhs, cudaMemcpyDeviceToDevice, s));
    return tri_solve<double>(m, m->A64, n, u_d, nrhs);
}

// Refinement for all right-hand sides together: u = 0, r = b; repeat
//   d = A32^{-1} r (FP32 factor, trisolve.cu), u += d,
//   r = b - A u in FP64, or r -= A d,
// until every column has ||r|| <= tol ||b|| or max_iter sweeps.  The first sweep's residual is
// formed from u in FP64.  Once the residual is below kUpdateBelow the correction is as small
// against u, and r -= A d in double-float arithmetic (2^-46 of |A| |d|) loses less than the
// rounding of u to FP64 (2^-53 of |A| |u|) does; below kLateFactor * tol plain FP32 does: its error is
// 2^-24 or so of |A| |d|, that is 6e-8 kLateFactor tol = 6e-4 tol times the ratio of |A| |d| to
// the residual A d before the sweep (tens on these operators).
//
// u's own rounding: what u += d rounds off is kept (c, FP32, exact to 2^-24 of itself) and the next
// sum takes it in, so r -= A d follows b - A (u + c), and the residual of u itself is r + A c.
// The first sweep's residual tells whether A c matters: its u holds FP32 numbers, whose rounding is
// 2^29 times FP64's, so A c is 2^-29 of that residual or less (2^-32 was measured).  A tolerance
// of at least kRoundingFactor times it (and 2^-53) leaves A c below tol / 16.  For a smaller one
// r + A c is formed, in plain FP32, once r has reached it, and decides: a tolerance that r reaches and u
// cannot does not pass for reached.  Where late sweeps are allowed, r + A c <= kLateFactor tol is
// enough (the level at which b - A u has been formed before them), else r + A c <= tol.
constexpr double kUpdateBelow = 1e-3;
constexpr double kLateFactor = 1e4;
constexpr double kRoundingFactor = 0x1p-25;

int refine_start(const RefineVecs &v, int64_t n, int nrhs, cudaStream_t s) {
    const int64_t nn = n * nrhs;
    FEM3_CUDA(cudaMemsetAsync(v.u, 0, sizeof(double) * nn, s));
    FEM3_CUDA(cudaMemsetAsync(v.dc + nn, 0, sizeof(float) * nn, s));
    FEM3_CUDA(cudaMemcpyAsync(v.r, v.b, sizeof(double) * nn, cudaMemcpyDeviceToDevice, s));
    return FEM3_OK;
}

// one sweep, enqueued on m->stream; the norms arrive in m->h_norms (2 nrhs values, from kTrueSlot
// on nrhs more)
int refine_sweep(Mesh *m, const RefineVecs &v, int nrhs, RefineMode mode) {
    cudaStream_t s = m->stream;
    const int64_t n = m->n_dof, nn = n * nrhs;
    if (mode != kRefineCheck) {
        k_to_f32<<<g256(nn), 256, 0, s>>>(v.r, v.dc, nn);
        note_launch(m);
        FEM3_TRY(tri_solve<float>(m, m->A32, n, v.dc, nrhs));
        k_add_correction<<<g256(nn), 256, 0, s>>>(v.dc, v.u, v.dc + nn, nn, mode != kRefineFull);
        note_launch(m);
    }
    const size_t bytes = sizeof(double) * (mode == kRefineCheck ? kTrueSlot + nrhs : 2 * nrhs);
    FEM3_CUDA(cudaMemsetAsync(m->norms, 0, bytes, s));
    const dim3 grid(g256(n), nrhs);
    if (mode == kRefineFull) {
        FEM3_TRY(apply_multi(m, v.u, nrhs, v.Au));
        k_residual_cols<<<grid, 256, 0, s>>>(v.b, v.Au, n, v.r, m->norms);
    } else if (mode == kRefineCheck) {
        FEM3_TRY(apply_correction(m, v.dc + nn, nrhs, v.Au, true));
        k_residual_update_cols<<<grid, 256, 0, s>>>(v.b, nullptr, v.Au, n, v.r, m->norms);
    } else {
        FEM3_TRY(apply_correction(m, v.dc, nrhs, v.Au, mode == kRefineLate));
        k_residual_update_cols<<<grid, 256, 0, s>>>(v.b, v.Au, nullptr, n, v.r, m->norms);
    }
    note_launch(m);
    FEM3_CUDA(cudaMemcpyAsync(m->h_norms, m->norms, bytes, cudaMemcpyDeviceToHost, s));
    return FEM3_OK;
}

// largest relative residual over the columns from the norms that have arrived, of r or (of_u) of
// u; infinity for NaN
static double worst_norm(const Mesh *m, int nrhs, bool of_u) {
    double worst = 0;
    for (int c = 0; c < nrhs; c++) {
        const double b = m->h_norms[2 * c + 1], r = m->h_norms[of_u ? kTrueSlot + c : 2 * c];
        const double rel = b > 0 ? sqrt(r / b) : 0.0;
        worst = (rel == rel) ? std::max(worst, rel) : INFINITY;
    }
    return worst;
}

// After the sweep q->mode, whose norms have arrived: whether the columns have converged, and what
// the next sweep is (late: plain FP32 updates are allowed).  False once there is none.
bool refine_next(const Mesh *m, int nrhs, double tol, int max_iter, bool late, RefineState *q) {
    const RefineMode was = q->mode;
    const double r = worst_norm(m, nrhs, false);
    q->worst = was == kRefineCheck ? worst_norm(m, nrhs, true) : r;
    if (was != kRefineCheck && ++q->sweeps == 1) q->check = tol < kRoundingFactor * std::max(r, 0x1p-28);
    if (was == kRefineCheck)
        q->converged = q->worst <= (late ? kLateFactor : 1.0) * tol;
    else
        q->converged = r <= tol && (was == kRefineFull || !q->check);
    if (r <= tol && q->check && was != kRefineCheck)
        q->mode = kRefineCheck;
    else
        q->mode = late && r <= kLateFactor * tol ? kRefineLate
                                                 : (r <= kUpdateBelow ? kRefineUpdate : kRefineFull);
    return !q->converged && q->worst < INFINITY && (q->sweeps < max_iter || q->mode == kRefineCheck);
}

// largest ||b - A u|| / ||b|| over the columns (synchronises)
int residual_worst(Mesh *m, const double *b, const double *u, int nrhs, double *worst) {
    cudaStream_t s = m->stream;
    const int64_t n = m->n_dof;
    const int group = std::min(nrhs, 24);   // norms: 2 values a column
    double *Au = nullptr;   // A u, then the residual
    FEM3_CUDA(cudaMallocAsync((void **)&Au, sizeof(double) * n * group, s));
    int st = FEM3_OK;
    *worst = 0.0;
    for (int c0 = 0; c0 < nrhs && st == FEM3_OK; c0 += group) {
        const int cnt = std::min(group, nrhs - c0);
        if (m->integer_order) {
            for (int c = 0; c < cnt && st == FEM3_OK; c++)
                st = apply_integer(m, u + (int64_t)(c0 + c) * n, Au + (int64_t)c * n);
        } else {
            st = apply_multi(m, u + (int64_t)c0 * n, cnt, Au);
        }
        if (st != FEM3_OK) break;
        cudaMemsetAsync(m->norms, 0, sizeof(double) * 2 * cnt, s);
        k_residual_cols<<<dim3(g256(n), cnt), 256, 0, s>>>(b + (int64_t)c0 * n, Au, n, Au, m->norms);
        note_launch(m);
        cudaError_t e = cudaMemcpyAsync(m->h_norms, m->norms, sizeof(double) * 2 * cnt,
                                        cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) st = cuda_error(e, "residual norms");
        else *worst = std::max(*worst, worst_norm(m, cnt, false));
    }
    cudaFreeAsync(Au, s);
    return st;
}

int solve_refined(Mesh *m, const double *b_d, int nrhs, double tol, int max_iter, double *u_d,
                  int *iters, double *resid) {
    cudaStream_t s = m->stream;
    const int64_t n = m->n_dof;
    const int64_t nn = n * nrhs;
    if (nrhs > 32) return set_error(FEM3_E_ARG, "at most 32 right-hand sides per solve");
    RefineVecs v{b_d, u_d, nullptr, nullptr, nullptr};
    FEM3_CUDA(cudaMallocAsync((void **)&v.Au, sizeof(double) * nn, s));
    FEM3_CUDA(cudaMallocAsync((void **)&v.r, sizeof(double) * nn, s));
    FEM3_CUDA(cudaMallocAsync((void **)&v.dc, sizeof(float) * 2 * nn, s));
    RefineState q;
    int st = refine_start(v, n, nrhs, s);
    do {
        if (st != FEM3_OK || (st = refine_sweep(m, v, nrhs, q.mode)) != FEM3_OK) break;
        FEM3_CUDA(cudaStreamSynchronize(s));
    } while (refine_next(m, nrhs, tol, max_iter, true, &q));
    cudaFreeAsync(v.Au, s);
    cudaFreeAsync(v.r, s);
    cudaFreeAsync(v.dc, s);
    if (iters) *iters = q.sweeps;
    if (resid) *resid = q.worst;
    if (st != FEM3_OK) return st;
    if (!q.converged)
        return set_error(FEM3_E_NO_CONVERGE, "iterative refinement did not reach the tolerance");
    return FEM3_OK;
}

}  // namespace fem3
