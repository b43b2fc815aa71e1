// The assembled operator in FP64, block-sparse: what the refinement's residual b - A u
// applies (Section 2.1 element sum of the Section 2.3 tables).
//
// A couples two dofs only when a line parallel to an axis meets both element patches, so on a
// mesh of n cells per side a row has about 75 n nonzeros of n^3 columns.  The nonzero 32 x 32
// blocks (by the bins' template sets) are kept column-major, both triangles, so a block row's
// sums belong to one CTA and need no atomics.
//   once per mesh: k_op_mark, scans, k_op_rows - the block pattern;
//   once per assembly: the contraction adds the lower blocks in FP64 (k_contract_rows, from
//     double-float row sums) and k_op_mirror transposes them; the FP64 form copies its dense
//     matrix instead, before the factorisation overwrites it (k_op_from_dense);
//   per apply: k_op_apply, in one of three arithmetics:
//     kOpFull    FP64: the residual of a whole solution, b - A u, whose terms cancel (a double-
//                float sum there leaves ten times the error in u: its 2^-48 per term is amplified
//                by the solve);
//     kOpUpdate  double-float FP32 (11 instructions per multiply-add against 64 clocks of the
//                FP64 pipe): the update r -= A d of a correction d, 1e-3 of u or less;
//     kOpLate    FP32: the update of the single-mesh solve's last sweeps, and A times the carries
//                (about 1e-6 relative).
//
// Bound: the FP64 pipe in kOpFull with many vectors, FP32 issue in the others, HBM for one
// vector (8 bytes per entry of a nonzero block, a tenth to a half of n^2).  Applying the
// tables' nonzeros instead, L^T W (R u) and R^T W (L u) in double-float arithmetic, took two
// multiply-adds for each of 144 entries per Gauss point on the 24^3 mesh with two passes that
// wait on each other.  Measured at the 24^3
// parallelepiped, 17 vectors (GB300): 3.48 ms (1.81 ms in plain FP32) so; 1.94, 0.49 and 0.13 ms in
// the three arithmetics here.  Eight vectors at 20^3: 0.95 (0.84) ms; 0.39, 0.11, 0.04 ms.
#include <algorithm>
#include <type_traits>

#include "fem3_impl.cuh"

namespace fem3 {

namespace {

constexpr int kOB = kOpBlock;
constexpr int kOpThreads = 256, kOpWarps = kOpThreads / 32;
constexpr int kOpSplitMax = 8;
// up to this many block rows (1,024 dofs) the pattern is every block: three quarters of them
// or more are nonzero there, and finding them costs twelve launches and a wait
constexpr int kOpAllMax = 32;
constexpr int kOpCountSlot = 124;   // of h_norms: the two block counts
enum OpMode { kOpFull = 0, kOpUpdate = 1, kOpLate = 2 };

__host__ __device__ inline int64_t tri_id(int64_t i, int64_t j) { return i * (i + 1) / 2 + j; }

struct MarkAxis {
    const int32_t *dof_off, *dof_idx;
    int n_bins;
};
struct MarkAxes {
    MarkAxis a[3];
};

// flag[tri(i, j)] = 1 for the block pairs (i >= j) of every two template rows of a bin (the
// stores of one value race harmlessly).  One CTA per bin: the rows' blocks as a bit set in
// shared memory, listed in order, then every pair of the list.
__global__ void __launch_bounds__(256) k_op_mark(const __grid_constant__ MarkAxes P, int nb,
                                                 int32_t *flag) {
    extern __shared__ uint32_t sm_mark[];
    int b = blockIdx.x, axis = 0;
    while (axis < 2 && b >= P.a[axis].n_bins) b -= P.a[axis++].n_bins;
    const int d0 = P.a[axis].dof_off[b], D = P.a[axis].dof_off[b + 1] - d0;
    const int32_t *dofs = P.a[axis].dof_idx + d0;
    const int nw = (nb + 31) / 32;
    uint32_t *bits = sm_mark;                              // [nw]
    uint16_t *list = reinterpret_cast<uint16_t *>(bits + nw);   // [min(nb, max_dof)]
    __shared__ int s_n;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int w = threadIdx.x; w < nw; w += 256) bits[w] = 0;
    __syncthreads();
    for (int c = threadIdx.x; c < D; c += 256) {
        const int i = __ldg(dofs + c) / kOB;
        atomicOr(&bits[i >> 5], 1u << (i & 31));
    }
    __syncthreads();
    if (warp == 0) {
        int n = 0;
        for (int w0 = 0; w0 < nw; w0 += 32) {
            uint32_t x = w0 + lane < nw ? bits[w0 + lane] : 0u;
            const int c = __popc(x);
            int pre = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, pre, o);
                if (lane >= o) pre += y;
            }
            for (int k = n + pre - c; x; x &= x - 1)
                list[k++] = (uint16_t)(32 * (w0 + lane) + __ffs(x) - 1);
            n += __shfl_sync(0xffffffffu, pre, 31);
        }
        if (lane == 0) s_n = n;
    }
    __syncthreads();
    for (int p = warp; p < s_n; p += 8) {
        const int i = list[p];
        for (int q = lane; q <= p; q += 32) flag[tri_id(i, list[q])] = 1;
    }
}

// map[p] = id of lower block p (from the scan of the flags) or -1
__global__ void k_op_map(const int32_t *__restrict__ flag, const int32_t *__restrict__ off,
                         int64_t n, int32_t *map) {
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p < n) map[p] = flag[p] ? off[p] : -1;
}

// one warp per block row: the columns of its blocks in order.  FILL = false: their number
// into cnt; true: column and source (2 * lower block id + 1 if read transposed) at row_off[i]
template <bool FILL>
__global__ void __launch_bounds__(256) k_op_rows(const int32_t *__restrict__ map, int nb,
                                                 int32_t *cnt, const int32_t *row_off, int32_t *col,
                                                 int32_t *src) {
    const int i = (int)(blockIdx.x * (int64_t)(blockDim.x >> 5)) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (i >= nb) return;
    int n = 0;
    const int base = FILL ? row_off[i] : 0;
    for (int j0 = 0; j0 < nb; j0 += 32) {
        const int j = j0 + lane;
        const int id = j < nb ? map[j <= i ? tri_id(i, j) : tri_id(j, i)] : -1;
        const unsigned m = __ballot_sync(0xffffffffu, id >= 0);
        if (FILL && id >= 0) {
            const int k = base + n + __popc(m & ((1u << lane) - 1u));
            col[k] = j;
            src[k] = 2 * id + (j > i ? 1 : 0);
        }
        n += __popc(m);
    }
    if (!FILL && lane == 0) cnt[i] = n;
}

// block k of the full pattern, column-major, from its lower block.  A lower block is
// row-major; the diagonal ones hold their lower triangle.
__global__ void __launch_bounds__(256) k_op_mirror(const double *__restrict__ low,
                                                   const int32_t *__restrict__ src,
                                                   const int32_t *__restrict__ row_of,
                                                   const int32_t *__restrict__ col, double *full) {
    __shared__ double t[kOB][kOB + 1];
    const int64_t k = blockIdx.x;
    const int s = src[k];
    const double *L = low + (int64_t)(s >> 1) * (kOB * kOB);
    for (int e = threadIdx.x; e < kOB * kOB; e += 256) t[e / kOB][e % kOB] = L[e];
    __syncthreads();
    const bool diag = row_of[k] == col[k], tr = s & 1;
    double *F = full + k * (kOB * kOB);
    for (int e = threadIdx.x; e < kOB * kOB; e += 256) {
        const int c = e / kOB, r = e % kOB;   // column-major output
        const bool swap = diag ? c > r : tr;
        F[e] = swap ? t[c][r] : t[r][c];
    }
}

// the same from a dense lower triangle (row-major n x n)
__global__ void __launch_bounds__(256) k_op_from_dense(const double *__restrict__ A, int64_t n,
                                                       const int32_t *__restrict__ row_of,
                                                       const int32_t *__restrict__ col,
                                                       double *full) {
    __shared__ double t[kOB][kOB + 1];
    const int64_t k = blockIdx.x;
    const int i = row_of[k], j = col[k];
    const bool tr = j > i;
    const int64_t r0 = (int64_t)(tr ? j : i) * kOB, c0 = (int64_t)(tr ? i : j) * kOB;
    for (int e = threadIdx.x; e < kOB * kOB; e += 256) {
        const int r = e / kOB, c = e % kOB;
        t[r][c] = r0 + r < n && c0 + c < n ? A[(r0 + r) * n + c0 + c] : 0.0;
    }
    __syncthreads();
    double *F = full + k * (kOB * kOB);
    for (int e = threadIdx.x; e < kOB * kOB; e += 256) {
        const int c = e / kOB, r = e % kOB;
        const bool swap = i == j ? c > r : tr;
        F[e] = swap ? t[c][r] : t[r][c];
    }
}

// row of every block of the full pattern
__global__ void k_op_row_of(const int32_t *__restrict__ row_off, int nb, int32_t *row_of) {
    const int i = blockIdx.x;
    for (int k = row_off[i] + threadIdx.x; k < row_off[i + 1]; k += blockDim.x) row_of[k] = i;
}

// the pattern with every block: lower blocks in triangle order (grid: block rows)
__global__ void k_op_all(int nb, int32_t *map, int32_t *row_off, int32_t *col, int32_t *src,
                         int32_t *row_of) {
    const int i = blockIdx.x;
    if (threadIdx.x == 0) {
        row_off[i] = i * nb;
        if (i == 0) row_off[nb] = nb * nb;
    }
    for (int j = threadIdx.x; j < nb; j += blockDim.x) {
        const int p = (int)(j <= i ? tri_id(i, j) : tri_id(j, i)), k = i * nb + j;
        if (j <= i) map[p] = p;
        col[k] = j;
        src[k] = 2 * p + (j > i ? 1 : 0);
        row_of[k] = i;
    }
}

// vectors interleaved, [rows padded to whole blocks][XS]: FP64 solutions or FP32 corrections,
// XS a multiple of 16 bytes so that the apply reads them 16 bytes at a time
template <int NR, int MODE> struct OpCfg {
    using X = float;
    static constexpr int XS = NR == 1 ? 1 : (NR + 3) / 4 * 4;
};
template <int NR> struct OpCfg<NR, kOpFull> {
    using X = double;
    static constexpr int XS = NR == 1 ? 1 : (NR + 1) / 2 * 2;
};

template <class T, int XS>
__global__ void k_op_gather(const T *__restrict__ u, int64_t n, int64_t rows, int nv, T *x) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= XS * rows) return;
    const int64_t i = e / XS;
    const int v = (int)(e - i * XS);
    x[e] = v < nv && i < n ? u[(int64_t)v * n + i] : T(0);
}

// (sh, sl) += (ah + al) x
__device__ __forceinline__ void df_fma_f(float ah, float al, float x, float &sh, float &sl) {
    const float p = ah * x;
    const float e = fmaf(al, x, fmaf(ah, x, -p));
    const float t = sh + p;
    const float z = t - sh;
    const float err = (sh - (t - z)) + (p - z);
    sh = t;
    sl += err + e;
}

// Part blockIdx.y of S of block row blockIdx.x: the sums over its share of the row's blocks
// for NR vectors.  Warp w takes blocks w, w + 8, ... of the share (lane = row): the block's
// 32 entries of x go to the warp's shared memory (read back as broadcasts), the block's
// columns come straight from global memory, 256 bytes per column, U columns in flight; the
// eight warps' sums are added in a fixed order.
template <int NR, int MODE>
__global__ void __launch_bounds__(kOpThreads, NR > 8 ? 2 : 3)
    k_op_apply(const int32_t *__restrict__ row_off, const int32_t *__restrict__ col,
               const double *__restrict__ full, const typename OpCfg<NR, MODE>::X *__restrict__ x,
               double *part, int nb) {
    using X = typename OpCfg<NR, MODE>::X;
    constexpr int XS = OpCfg<NR, MODE>::XS;
    constexpr int U = NR == 1 ? 16 : 8;   // columns in flight
    extern __shared__ __align__(16) unsigned char sm_op[];   // x of the warps, then their sums
    const int i = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int k0 = row_off[i], nk = row_off[i + 1] - k0;
    const int S = gridDim.y, s = blockIdx.y;
    const int ka = k0 + (int)((int64_t)nk * s / S), kb = k0 + (int)((int64_t)nk * (s + 1) / S);
    X *xs = reinterpret_cast<X *>(sm_op) + warp * (kOB * XS);
    // sums: FP64, or hi and lo parts
    using Acc = typename std::conditional<MODE == kOpFull, double, float>::type;
    Acc h[NR];
    float l[NR];
#pragma unroll
    for (int v = 0; v < NR; v++) { h[v] = Acc(0); l[v] = 0.f; }
    for (int k = ka + warp; k < kb; k += kOpWarps) {
        const X *xb = x + (int64_t)col[k] * (kOB * XS);
#pragma unroll
        for (int e = 0; e < XS; e++) xs[lane + 32 * e] = __ldg(xb + lane + 32 * e);
        __syncwarp();
        const double *B = full + (int64_t)k * (kOB * kOB) + lane;
        for (int c0 = 0; c0 < kOB; c0 += U) {
            double a[U];
#pragma unroll
            for (int j = 0; j < U; j++) a[j] = __ldcs(B + (c0 + j) * kOB);
#pragma unroll
            for (int j = 0; j < U; j++) {
                const X *xc = xs + (c0 + j) * XS;
                float ah = 0.f, al = 0.f;
                if constexpr (MODE != kOpFull) f64_split(a[j], ah, al);
                auto add = [&](int v, X xv) {
                    if constexpr (MODE == kOpFull) h[v] = fma(a[j], xv, h[v]);
                    else if constexpr (MODE == kOpUpdate) df_fma_f(ah, al, xv, h[v], l[v]);
                    else h[v] = fmaf(ah, xv, h[v]);
                };
                if constexpr (NR == 1) {
                    add(0, xc[0]);
                } else if constexpr (MODE == kOpFull) {
#pragma unroll
                    for (int v = 0; v < NR; v += 2) {
                        const double2 q = *reinterpret_cast<const double2 *>(xc + v);
                        add(v, q.x);
                        if (v + 1 < NR) add(v + 1, q.y);
                    }
                } else {
#pragma unroll
                    for (int v = 0; v < NR; v += 4) {
                        const float4 q = *reinterpret_cast<const float4 *>(xc + v);
                        add(v, q.x);
                        if (v + 1 < NR) add(v + 1, q.y);
                        if (v + 2 < NR) add(v + 2, q.z);
                        if (v + 3 < NR) add(v + 3, q.w);
                    }
                }
            }
        }
        __syncwarp();
    }
    __syncthreads();
    double *sums = reinterpret_cast<double *>(sm_op);   // [warps][NR][32]
#pragma unroll
    for (int v = 0; v < NR; v++) {
        double y;
        if constexpr (MODE == kOpFull) y = h[v];
        else if constexpr (MODE == kOpUpdate) y = f32_to_f64_exact(h[v]) + f32_to_f64_exact(l[v]);
        else y = f32_to_f64_exact(h[v]);
        sums[(warp * NR + v) * 32 + lane] = y;
    }
    __syncthreads();
    double *out = part + ((int64_t)s * nb + i) * (NR * kOB);
    for (int e = threadIdx.x; e < NR * kOB; e += kOpThreads) {
        double y = sums[e];
#pragma unroll
        for (int w = 1; w < kOpWarps; w++) y += sums[w * NR * 32 + e];
        out[e] = y;
    }
}

// Au[v][row] = scale times the parts' sum, added in order (grid: block rows; thread: vector, row)
__global__ void __launch_bounds__(256) k_op_sum(const double *__restrict__ part, int nb, int S,
                                                int nr, int64_t n, int nv, double scale, double *Au) {
    const int64_t i = blockIdx.x;
    for (int e = threadIdx.x; e < nv * kOB; e += 256) {
        const int64_t row = i * kOB + (e & 31);
        if (row >= n) continue;
        double y = part[i * (nr * kOB) + e];
        for (int s = 1; s < S; s++) y += part[((int64_t)s * nb + i) * (nr * kOB) + e];
        Au[(int64_t)(e >> 5) * n + row] = y * scale;
    }
}

inline unsigned g256(int64_t n) { return (unsigned)(n > 0 ? (n + 255) / 256 : 1); }

template <int NR, int MODE>
int apply_group(Mesh *m, const typename OpCfg<NR, MODE>::X *u, int nv, double *Au, double *ws) {
    using X = typename OpCfg<NR, MODE>::X;
    constexpr int XS = OpCfg<NR, MODE>::XS;
    cudaStream_t s = m->stream;
    const OpBlocks &O = m->op;
    const int64_t rows = (int64_t)O.nb * kOB;
    X *x = reinterpret_cast<X *>(ws);
    double *part = ws + (int64_t)kOpVecs * rows;
    // parts of a block row: CTAs for about four rounds of the SMs, a warp-round of blocks each
    const int64_t per_row = std::max<int64_t>(1, O.n_full / O.nb);
    const int S = (int)std::max<int64_t>(
        1, std::min<int64_t>(std::min<int64_t>(kOpSplitMax, (1216 + O.nb - 1) / O.nb),
                             (per_row + kOpWarps - 1) / kOpWarps));
    k_op_gather<X, XS><<<g256(XS * rows), 256, 0, s>>>(u, m->n_dof, rows, nv, x);
    note_launch(m);
    const size_t sh = std::max(sizeof(X) * kOpWarps * kOB * XS, sizeof(double) * kOpWarps * kOB * NR);
    kc_begin(m, KC_APPLY);
    k_op_apply<NR, MODE><<<dim3(O.nb, S), kOpThreads, sh, s>>>(O.row_off, O.col, O.full, x, part, O.nb);
    kc_end(m, KC_APPLY);
    note_launch(m);
    k_op_sum<<<O.nb, 256, 0, s>>>(part, O.nb, S, NR, m->n_dof, nv, O.scale, Au);
    note_launch(m);
    FEM3_CUDA(cudaGetLastError());
    return FEM3_OK;
}

// Au = A u for nv vectors (column-major, leading dimension n_dof), in groups: up to 17 per
// pass while at least 13 are left, then up to eight, and a last group of one or up to four
// vectors takes the narrower form of the kernel
template <int MODE>
int apply_groups(Mesh *m, const typename OpCfg<1, MODE>::X *u_d, int nv, double *Au_d) {
    const int64_t n = m->n_dof;
    if (n == 0 || nv < 1) return FEM3_OK;
    FEM3_TRY(op_build(m));
    double *ws = nullptr;
    const int64_t rows = (int64_t)m->op.nb * kOB;
    FEM3_CUDA(cudaMallocAsync((void **)&ws,
                              sizeof(double) * rows * (kOpVecs + (int64_t)kOpVecs * kOpSplitMax),
                              m->stream));
    int st = FEM3_OK;
    for (int v0 = 0, cnt = 0; v0 < nv && st == FEM3_OK; v0 += cnt) {
        const int left = nv - v0;
        const auto *u = u_d + (int64_t)v0 * n;
        double *out = Au_d + (int64_t)v0 * n;
        cnt = left >= 13 ? std::min(17, left) : (left >= 5 ? std::min(8, left) : std::min(4, left));
        if (left >= 13) st = apply_group<17, MODE>(m, u, cnt, out, ws);
        else if (left >= 5) st = apply_group<8, MODE>(m, u, cnt, out, ws);
        else if (left >= 2) st = apply_group<4, MODE>(m, u, cnt, out, ws);
        else st = apply_group<1, MODE>(m, u, cnt, out, ws);
    }
    cudaFreeAsync(ws, m->stream);
    return st;
}

}  // namespace

// Finds the nonzero blocks and sends their numbers to the host (once per mesh; nothing to do
// for the small patterns with every block).  Enqueued before the walk of an assembly, so that
// op_prepare, called once the factorisation's turn has come, finds the numbers there.
int op_count(Mesh *m) {
    OpBlocks &O = m->op;
    if (O.counted || m->n_dof == 0) return FEM3_OK;
    const int nb = (int)((m->n_dof + kOB - 1) / kOB);
    if (nb <= kOpAllMax) return FEM3_OK;
    cudaStream_t s = m->stream;
    cudaStreamCaptureStatus cap;   // in a caller's capture: left to the solve
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return FEM3_OK;
    }
    const int64_t np = tri_id(nb, 0);
    int32_t *flag, *off, *cnt;
    if (!O.ev) FEM3_CUDA(cudaEventCreateWithFlags(&O.ev, cudaEventDisableTiming));
    FEM3_TRY(dev_alloc_t(m, &O.map, np));
    FEM3_TRY(dev_alloc_t(m, &O.row_off, nb + 1));
    FEM3_TRY(dev_alloc_t(m, &flag, np));
    FEM3_TRY(dev_alloc_t(m, &off, np + 1));
    FEM3_TRY(dev_alloc_t(m, &cnt, nb));
    FEM3_CUDA(cudaMemsetAsync(flag, 0, sizeof(int32_t) * np, s));
    MarkAxes P;
    int64_t bins = 0;
    int max_dof = 0;
    for (int a = 0; a < 3; a++) {
        max_dof = std::max(max_dof, m->bins[a].max_dof);
        P.a[a] = MarkAxis{m->bins[a].dof_off, m->bins[a].dof_idx, m->bins[a].n_bins};
        bins += m->bins[a].n_bins;
    }
    const size_t sh = sizeof(uint32_t) * ((nb + 31) / 32) +
                      sizeof(uint16_t) * (size_t)std::min(nb, std::max(1, max_dof));
    k_op_mark<<<(unsigned)bins, 256, sh, s>>>(P, nb, flag);
    FEM3_TRY(scan_i32(flag, off, np, s, m));
    k_op_map<<<g256(np), 256, 0, s>>>(flag, off, np, O.map);
    k_op_rows<false><<<(nb + 7) / 8, 256, 0, s>>>(O.map, nb, cnt, nullptr, nullptr, nullptr);
    FEM3_TRY(scan_i32(cnt, O.row_off, nb, s, m));
    int32_t *h = reinterpret_cast<int32_t *>(m->h_norms + kOpCountSlot);
    FEM3_CUDA(cudaMemcpyAsync(h, off + np, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    FEM3_CUDA(cudaMemcpyAsync(h + 1, O.row_off + nb, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    FEM3_CUDA(cudaEventRecord(O.ev, s));
    m->launches += 3;
    FEM3_CUDA(cudaGetLastError());
    O.counted = true;
    return FEM3_OK;
}

// the block pattern of the mesh and the storage of its blocks (once)
static int op_pattern(Mesh *m) {
    OpBlocks &O = m->op;
    if (O.full) return FEM3_OK;
    cudaStream_t s = m->stream;
    const int nb = (int)((m->n_dof + kOB - 1) / kOB);
    const bool all = nb <= kOpAllMax;
    if (all) {
        const int64_t np = tri_id(nb, 0);
        if (!O.map) FEM3_TRY(dev_alloc_t(m, &O.map, np));
        if (!O.row_off) FEM3_TRY(dev_alloc_t(m, &O.row_off, nb + 1));
        O.n_low = np;
        O.n_full = (int64_t)nb * nb;
    } else {
        FEM3_TRY(op_count(m));
        if (!O.counted) return set_error(FEM3_E_STATE, "the solve cannot be captured");
        FEM3_CUDA(cudaEventSynchronize(O.ev));
        const int32_t *h = reinterpret_cast<const int32_t *>(m->h_norms + kOpCountSlot);
        O.n_low = h[0];
        O.n_full = h[1];
    }
    O.nb = nb;
    const int64_t nf = std::max<int64_t>(1, O.n_full);
    FEM3_TRY(dev_alloc_t(m, &O.col, nf));
    FEM3_TRY(dev_alloc_t(m, &O.src, nf));
    FEM3_TRY(dev_alloc_t(m, &O.row_of, nf));
    double *full = nullptr;
    FEM3_TRY(dev_alloc(m, (void **)&full, sizeof(double) * kOB * kOB * nf));
    if (all) {
        k_op_all<<<nb, 64, 0, s>>>(nb, O.map, O.row_off, O.col, O.src, O.row_of);
    } else {
        k_op_rows<true><<<(nb + 7) / 8, 256, 0, s>>>(O.map, nb, nullptr, O.row_off, O.col, O.src);
        k_op_row_of<<<nb, 128, 0, s>>>(O.row_off, nb, O.row_of);
        note_launch(m);
    }
    note_launch(m);
    FEM3_CUDA(cudaGetLastError());
    O.full = full;
    return FEM3_OK;
}

int op_prepare(Mesh *m, bool low) {
    FEM3_TRY(op_pattern(m));
    OpBlocks &O = m->op;
    if (low && !O.low)
        FEM3_TRY(dev_alloc(m, (void **)&O.low,
                           sizeof(double) * kOB * kOB * (size_t)std::max<int64_t>(1, O.n_low)));
    return FEM3_OK;
}

// the operator of the current tables (nothing to do if it is ready)
int op_build(Mesh *m) {
    if (m->op_ready || m->n_dof == 0) return FEM3_OK;
    FEM3_TRY(op_prepare(m, true));
    OpBlocks &O = m->op;
    FEM3_CUDA(cudaMemsetAsync(O.low, 0, sizeof(double) * kOB * kOB * (size_t)std::max<int64_t>(1, O.n_low),
                              m->stream));
    FEM3_TRY(contract_blocks(m, O));
    if (O.n_full > 0) {
        kc_begin(m, KC_OPERATOR);
        k_op_mirror<<<(unsigned)O.n_full, 256, 0, m->stream>>>(O.low, O.src, O.row_of, O.col, O.full);
        kc_end(m, KC_OPERATOR);
        note_launch(m);
    }
    FEM3_CUDA(cudaGetLastError());
    m->op_ready = true;
    return FEM3_OK;
}

// the operator of the FP64 form: its matrix itself, before the factorisation
int op_from_dense(Mesh *m, const double *A) {
    if (m->op_ready || m->n_dof == 0) return FEM3_OK;
    FEM3_TRY(op_pattern(m));
    OpBlocks &O = m->op;
    if (O.n_full > 0) {
        k_op_from_dense<<<(unsigned)O.n_full, 256, 0, m->stream>>>(A, m->n_dof, O.row_of, O.col,
                                                                    O.full);
        note_launch(m);
    }
    FEM3_CUDA(cudaGetLastError());
    O.scale = 1.0;
    m->op_ready = true;
    return FEM3_OK;
}

int apply_multi(Mesh *m, const double *u_d, int nv, double *Au_d) {
    return apply_groups<kOpFull>(m, u_d, nv, Au_d);
}

int apply_correction(Mesh *m, const float *d, int nv, double *Ad, bool late) {
    return late ? apply_groups<kOpLate>(m, d, nv, Ad) : apply_groups<kOpUpdate>(m, d, nv, Ad);
}

int apply_A64(Mesh *m, const double *u_d, double *Au_d) { return apply_multi(m, u_d, 1, Au_d); }

}  // namespace fem3
