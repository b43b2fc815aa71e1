// fem3_spd_solve_static: a dense SPD solve that allocates no device memory.
//
// Some callers cannot allocate device memory at the point where they need a solve:
// latency-critical loops that must never enter the allocator, and host applications or
// plugin hosts that own every device allocation themselves and hand the library only the
// buffers of the problem.  This entry point serves them: its working memory (the
// Cholesky factor, the inverses of its 64 x 64 diagonal blocks, flags and error words) is
// one file-scope static device array, so the caller passes only the matrix, the
// right-hand side and the output.  Each call ends by reading the error words back and
// synchronising its stream.
//
// Three steps: copy A, scaled (the factorisation works in place), the FP64 tile factorisation of
// chol_f64.cu, and one launch for both substitutions (k_na_solve).  What bounds it is the
// factorisation's diagonal chain (12 steps of 28 us at n = 384) and, for the substitutions,
// a hand-over between SMs per 64-row block.  Measured at n = 384 (GB300): 2.58 ms as one
// launch per 64-column step and phase, with a column-by-column 64 x 64 factor and one-warp
// substitutions; 0.42 ms now.
#include <math.h>

#include <mutex>

#include "chol_f64.cuh"
#include "fem3_impl.cuh"

namespace fem3 {

namespace {

constexpr int kNaMaxN = 512;   // largest system this entry point accepts
constexpr int NBS = 64;

// factor [kNaMaxN^2] | diagonal-block inverses [8][64 * 64] | y, then z | flags of the
// factorisation, then of the substitutions (2 kNaBlocks, a ticket, an abort word) | ERR_COUNT error
// words | exponents of the rows' scales
constexpr int kNaBlocks = kNaMaxN / NBS;
constexpr size_t kNaFactor = (size_t)kNaMaxN * kNaMaxN;
constexpr size_t kNaInv = (size_t)kNaBlocks * NBS * NBS;
constexpr int kNaCholTiles = kNaMaxN / kChol64Tile;
constexpr size_t kNaCholFlags = (size_t)kNaCholTiles * (kNaCholTiles + 1) + 3;
constexpr size_t kNaSolveFlags = 2 * kNaBlocks + 2;
constexpr size_t kNaElems =
    kNaFactor + kNaInv + kNaMaxN + (kNaCholFlags + kNaSolveFlags + ERR_COUNT + kNaMaxN + 1) / 2;
static __device__ __align__(256) double g_na_scratch[kNaElems];

#include "chol_smem.cuh"

std::mutex g_na_mutex;
void *g_na_ptr[256];   // per device: device address of g_na_scratch (host-side table)

// e with d 2^(2 e) in [1, 4) for a positive finite d, else 0
__device__ __forceinline__ int scale_exponent(double d) {
    if (!(d > 0.0) || isinf(d)) return 0;
    const int x = ilogb(d);
    return -((x - (x & 1)) / 2);
}

// F = S A S (the lower triangle, row-major n x n), S = diag(2^e) so that F's diagonal lies in [1, 4):
// an exact step, F's factor is A's with its rows scaled alike, but the factorisation's
// reciprocals of pivots stay finite where a pivot of A is subnormal.  Flags and error words cleared.
__global__ void __launch_bounds__(256) k_na_copy(const double *__restrict__ A, int n, double *F,
                                                 int *scale, int *flags, int n_flags) {
    const int i = blockIdx.x;
    const int ei = scale_exponent(A[(int64_t)i * n + i]);
    for (int c = threadIdx.x; c <= i; c += blockDim.x)
        F[(int64_t)i * n + c] =
            scalbn(A[(int64_t)i * n + c], ei + scale_exponent(A[(int64_t)c * n + c]));
    if (threadIdx.x == 0) scale[i] = ei;
    if (i == 0)
        for (int q = threadIdx.x; q < n_flags; q += blockDim.x) flags[q] = 0;
}

// part[16 columns 16 q ..] of row r of a 64 x 64 block times v: thread (r, q)
__device__ __forceinline__ double dot16(const double m[16], const double *v, int q) {
    double s = 0.0;
#pragma unroll
    for (int e = 0; e < 16; e++) s = fma(m[e], v[16 * q + e], s);
    return s;
}

// Both substitutions in one launch: L y = S b, then L^T z = y (z in y's place) and x = S z, in
// blocks of 64 rows.  A CTA takes roles from a ticket: role s < nb is the forward step of block s, role nb + s the backward
// step of block nb - 1 - s.  A step reads the tiles of its block row (column) into registers
// one ahead, adds each solved block as its flag appears, multiplies by the diagonal inverse
// and publishes the block.  A role waits only for earlier tickets, so the launch needs no
// co-residency; the waits are bounded (ERR_SOLVE, abort word).
// 256 threads, thread (row r = t & 63, quarter q = t >> 6 of the columns).
__global__ void __launch_bounds__(256) k_na_solve(const double *__restrict__ F,
                                                  const double *__restrict__ dinv, int n, int nb,
                                                  const double *__restrict__ b,
                                                  const int *__restrict__ scale, double *y,
                                                  double *x, int *flags, int *err) {
    __shared__ double v[NBS], red[4][NBS];
    __shared__ int s_role, s_ok;
    int *done = flags, *ticket = flags + 2 * nb, *abort_w = ticket + 1;
    const int t = threadIdx.x, r = t & 63, q = t >> 6;
    for (;;) {
        if (t == 0) s_role = atomicAdd(ticket, 1);
        __syncthreads();
        const int role = s_role;
        if (role >= 2 * nb) return;
        const bool bw = role >= nb;
        const int blk = bw ? 2 * nb - 1 - role : role;   // this step's block
        const int nd = bw ? role - nb : role;            // blocks it depends on
        const int row = blk * NBS + r;
        // the tile between this block and dependency d as applied (transposed when backward)
        auto tile = [&](int d, double m[16]) {
            const int jd = bw ? nb - 1 - d : d;
#pragma unroll
            for (int e = 0; e < 16; e++) {
                const int o = jd * NBS + 16 * q + e;     // row of the other block
                m[e] = (row < n && o < n) ? (bw ? __ldcg(F + (int64_t)o * n + row)
                                                : __ldcg(F + (int64_t)row * n + o))
                                          : 0.0;
            }
        };
        double mt[16], mn[16], acc = 0.0;
        if (nd > 0) tile(0, mt);
        for (int d = 0; d < nd; d++) {
            const int jd = bw ? nb - 1 - d : d;
            if (t == 0) {
                s_ok = 1;
                for (int spins = 0; ld_acquire_gpu(&done[bw ? nb + d : d]) == 0; spins++) {
                    if (ld_acquire_gpu(abort_w) != 0 || spins > kSpinLimit) {
                        if (spins > kSpinLimit) atomicAdd(&err[ERR_SOLVE], 1);
                        atomicExch(abort_w, 1);
                        s_ok = 0;
                        break;
                    }
                }
            }
            __syncthreads();
            if (!s_ok) return;
            if (t < NBS) v[t] = jd * NBS + t < n ? __ldcg(y + jd * NBS + t) : 0.0;
            if (d + 1 < nd) tile(d + 1, mn);
            __syncthreads();
            acc += dot16(mt, v, q);
#pragma unroll
            for (int e = 0; e < 16; e++) mt[e] = mn[e];
        }
        // the diagonal inverse as applied: X or X^T (loaded before the reduction's barriers)
#pragma unroll
        for (int e = 0; e < 16; e++) {
            const int c = 16 * q + e;
            mt[e] = __ldcg(dinv + (int64_t)blk * NBS * NBS + (bw ? c * NBS + r : r * NBS + c));
        }
        red[q][r] = acc;
        if (bw && nd == 0) {   // y of the last block comes from its forward role
            if (t == 0) {
                s_ok = 1;
                for (int spins = 0; ld_acquire_gpu(&done[nb - 1]) == 0; spins++) {
                    if (ld_acquire_gpu(abort_w) != 0 || spins > kSpinLimit) {
                        if (spins > kSpinLimit) atomicAdd(&err[ERR_SOLVE], 1);
                        atomicExch(abort_w, 1);
                        s_ok = 0;
                        break;
                    }
                }
            }
        } else if (t == 0) {
            s_ok = 1;
        }
        __syncthreads();
        if (!s_ok) return;
        if (t < NBS) {
            const int i = blk * NBS + t;
            const double rhs = i < n ? (bw ? __ldcg(y + i) : scalbn(b[i], scale[i])) : 0.0;
            v[t] = rhs - ((red[0][t] + red[1][t]) + (red[2][t] + red[3][t]));
        }
        __syncthreads();
        red[q][r] = dot16(mt, v, q);
        __syncthreads();
        if (t < NBS && blk * NBS + t < n) {
            const int i = blk * NBS + t;
            const double z = (red[0][t] + red[1][t]) + (red[2][t] + red[3][t]);
            y[i] = z;   // (only this step reads this block of y)
            if (bw) x[i] = scalbn(z, scale[i]);
        }
        __syncthreads();   // the block's stores are issued before the (cumulative) release
        if (t == 0) st_release_gpu(&done[role], 1);
    }
}

// device address of the static scratch for the current device (set up once per device)
int na_scratch(double **out) {
    int dev = 0;
    FEM3_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 256) return set_error(FEM3_E_ARG, "device ordinal out of range");
    std::lock_guard<std::mutex> lock(g_na_mutex);
    if (!g_na_ptr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_na_scratch);
        if (e != cudaSuccess) return cuda_error(e, "cudaGetSymbolAddress(static scratch)");
        g_na_ptr[dev] = p;
    }
    *out = static_cast<double *>(g_na_ptr[dev]);
    return FEM3_OK;
}

// true if p is device (or managed) memory that the current device can use directly
bool on_current_device(const void *p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (a.type == cudaMemoryTypeManaged) return true;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice && a.device == dev;
}

}  // namespace

}  // namespace fem3

using namespace fem3;

extern "C" int fem3_spd_solve_static(const double *A, int64_t n, const double *b, double *x,
                                     void *stream) {
    if (!A || !b || !x) return set_error(FEM3_E_ARG, "null argument");
    if (n < 1 || n > kNaMaxN)
        return set_error(FEM3_E_ARG, "fem3_spd_solve_static accepts 1 <= n <= 512 (its static "
                                     "working memory holds one 512 x 512 factor)");
    // the kernels read A and b and write x directly: all three must be device memory of
    // the current device (a host or foreign-device pointer is rejected, never dereferenced)
    if (!on_current_device(A) || !on_current_device(b) || !on_current_device(x))
        return set_error(FEM3_E_ARG, "fem3_spd_solve_static: A, b and x must be device memory "
                                     "of the current device");
    double *scratch = nullptr;
    FEM3_TRY(na_scratch(&scratch));
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int nn = (int)n, nb = (nn + NBS - 1) / NBS;
    double *F = scratch, *dinv = F + kNaFactor, *y = dinv + kNaInv;
    int *chol_flags = reinterpret_cast<int *>(y + kNaMaxN);
    int *flags = chol_flags + kNaCholFlags;
    int *err = flags + kNaSolveFlags;   // cleared with the substitutions' flags
    int *scale = err + ERR_COUNT;
    int launches = 0;
    k_na_copy<<<(unsigned)nn, 256, 0, s>>>(A, nn, F, scale, flags,
                                                 (int)(kNaSolveFlags + ERR_COUNT));
    FEM3_TRY(chol_f64(F, n, dinv, nullptr, chol_flags, err, s, &launches));
    k_na_solve<<<(unsigned)nb, 256, 0, s>>>(F, dinv, nn, nb, b, scale, y, x, flags, err);
    FEM3_CUDA(cudaGetLastError());
    int h_err[ERR_COUNT];
    FEM3_CUDA(cudaMemcpyAsync(h_err, err, sizeof(h_err), cudaMemcpyDeviceToHost, s));
    FEM3_CUDA(cudaStreamSynchronize(s));
    if (h_err[ERR_NOT_SPD])
        return set_error(FEM3_E_NOT_SPD, "non-positive pivot in Cholesky at column " +
                                             std::to_string(h_err[ERR_NOT_SPD] - 1));
    if (h_err[ERR_CHOL] || h_err[ERR_SOLVE])
        return set_error(FEM3_E_CUDA, "a factorisation or solve wait gave up (bounded wait expired)");
    return FEM3_OK;
}
