// Contraction A = sum_i s_i K_i (L_i^T W R_i + R_i^T W L_i) on CUDA cores, bin by bin
// (Section 2.1 element sum, Section 2.3 template: only dofs of a bin's template set can
// meet the bin's Gauss points, so each bin contributes to a D_b x D_b block), from the
// nonzeros of the bin's table blocks (about a fifth of their entries: k_contract_rows).
#include <math.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "fem3_impl.cuh"

namespace fem3 {

namespace {

constexpr int kRowsThreads = 256, kRowsWarps = kRowsThreads / 32;
// bins of at most this many rows take one point per half warp (a point's entries are about a
// fifth of the rows).  Measured for the three axes' double-float contraction, half against
// whole warps: 16^3 cube (115 rows on average) 0.67 against 0.83 ms, 24^3 parallelepiped (150) 5.1
// against 4.6 ms.
constexpr int kRowsHalfMax = 176;
constexpr int kRowsFlush = 4;   // elements of a finished row whose addresses are formed together
constexpr int kRowsEntryBytes = 48 * 1024;   // compacted entries in shared memory, at most
// the largest launch: entries, accumulator rows, weights, offsets and cursors of the points,
// dofs
constexpr size_t kRowsSmemMax =
    kRowsEntryBytes + sizeof(double) * (2 * kRowsWarps * kRowsWindow + kMaxBinItems) +
    sizeof(int) * (3 * kMaxBinItems + 1) + 64;
static_assert(kRowsWindow < (1 << 12) && kRowsEntryBytes / 6 < (1 << 19), "packed spans");

// Arithmetic of the contraction: double (FP64 form), float (FP32 form), or float2, a hi + lo
// FP32 pair (the refinement's operator: FP64 accuracy on the FP32 pipes).
// value(v): a table entry; weight(w): a Gauss weight; weigh(v, w): their product;
// add(acc, t, v): acc += t v; sum(a, b): a + b as the matrix's type
template <class TA> struct Arith;
template <> struct Arith<double> {
    using Out = double;
    // from the pair's bits (f32 -> f64 conversions run at the FP64 rate) and one add
    __device__ static double value(float2 v) { return f32_to_f64_exact(v.x) + f32_to_f64_exact(v.y); }
    __device__ static double weight(double w) { return w; }
    __device__ static double weigh(float2 v, double w) { return value(v) * w; }
    __device__ static double shfl(double t, int l) { return __shfl_sync(0xffffffffu, t, l); }
    __device__ static void add(double &acc, double t, double v) { acc = fma(t, v, acc); }
    __device__ static bool zero(double a) { return a == 0.0; }
    __device__ static double sum(double a, double b) { return a + b; }
};
template <> struct Arith<float> {
    using Out = float;
    __device__ static float value(float2 v) { return v.x + v.y; }
    __device__ static float weight(double w) { return (float)w; }
    __device__ static float weigh(float2 v, float w) { return value(v) * w; }
    __device__ static float shfl(float t, int l) { return __shfl_sync(0xffffffffu, t, l); }
    __device__ static void add(float &acc, float t, float v) { acc = fma(t, v, acc); }
    __device__ static bool zero(float a) { return a == 0.f; }
    __device__ static float sum(float a, float b) { return a + b; }
};
template <> struct Arith<float2> {
    using Out = double;
    __device__ static float2 value(float2 v) { return v; }
    __device__ static float2 weight(double w) {
        float h, l;
        f64_split(w, h, l);
        return make_float2(h, l);
    }
    __device__ static float2 weigh(float2 v, float2 w) {
        float h, l;
        df_mul(v.x, v.y, w.x, w.y, h, l);
        return make_float2(h, l);
    }
    __device__ static float2 shfl(float2 t, int l) {
        return make_float2(__shfl_sync(0xffffffffu, t.x, l), __shfl_sync(0xffffffffu, t.y, l));
    }
    __device__ static void add(float2 &acc, float2 t, float2 v) {
        df_fma(t.x, t.y, v.x, v.y, acc.x, acc.y);
    }
    __device__ static bool zero(float2 a) { return a.x == 0.f && a.y == 0.f; }
    __device__ static double sum(float2 a, float2 b) {
        df_add(b.x, b.y, a.x, a.y);
        return f32_to_f64_exact(a.x) + f32_to_f64_exact(a.y);
    }
};
template <class TA> __device__ __forceinline__ TA arith_zero() { return TA{}; }

// where an element goes: the lower triangle of a dense matrix (the fold A = s K (X + X^T):
// X(c1, c2) and X(c2, c1) land on the same element, the diagonal gets 2 X), a whole dense
// matrix (general form), or the lower triangle in 32 x 32 blocks
enum RowsOut { kLower = 0, kDense = 1, kBlocks = 2 };
// element index of (j1, j2) in A
template <int OUT>
__device__ __forceinline__ int64_t rows_index(int64_t n, const int32_t *__restrict__ map,
                                              int32_t j1, int32_t j2) {
    if constexpr (OUT == kDense) return j1 * n + j2;
    const int32_t i = max(j1, j2), j = min(j1, j2);
    if constexpr (OUT == kLower) return i * n + j;
    const uint32_t bi = (uint32_t)i / kOpBlock, bj = (uint32_t)j / kOpBlock;   // bi < 2^16
    const int64_t id = __ldg(map + bi * (bi + 1) / 2 + bj);
    return id * (kOpBlock * kOpBlock) + (i % kOpBlock * kOpBlock + j % kOpBlock);
}

// one axis of the product X = T^T diag(w) S over its bins
struct RowsAxis {
    const float2 *__restrict__ T, *__restrict__ S;   // tables of the rows and of the columns
    const int4 *__restrict__ work;                   // (bin, first column of the window, 0, 0)
    const int32_t *__restrict__ gp_off, *__restrict__ dof_off, *__restrict__ dof_idx,
        *__restrict__ tab_ld;
    const int64_t *__restrict__ tab_off;
    const double *__restrict__ w;                    // weights per slot, or per Gauss point
    const int32_t *__restrict__ w_idx;               // slot -> Gauss point (null: w per slot)
    double scale;
    int n_work;
};
struct RowsAxes {
    RowsAxis a[3];
};

// X(c1, c2) = sum_r w_r T[c1][r] S[c2][r] of one bin, row by row over the nonzeros (the
// order of Gustavson's sparse product): one CTA per (bin, window of <= win columns c2).
//   1. the window's nonzeros of S, compacted per Gauss point into shared memory (value and
//      column; counts, a scan, then the entries in any order: a point's columns differ, so
//      the sums do not depend on it);
//   2. warp = row c1: for every Gauss point with T[c1][r] != 0 a warp (HALF: half of one) takes
//      the point's entries, acc[c2] += (s K w T) S, in shared memory (the halves into rows of
//      their own: two points may share a column);
//   3. the row's nonzeros go to A (rows_index).
// Points go in groups whose entries fit `cap` (>= win, so a group holds at least one point);
// usually one group.
//
// Bound: shared-memory latency and the FP64 pipe (1/64 of the FP32 rate).  A dense 64 x 64
// tile product over the same blocks does 15 to 30 times the sum over points of
// nnz(T) nnz(S); here a point's entries are about one warp-wide pass (1.5 n on a mesh of n
// cells per side, both sides together 3 n).  Measured against that tile product, GB300: FP64
// assemble + solve of the 11^3 parallelepiped 9.57 -> 5.03 ms (contraction 4.76 -> 0.21 ms),
// one FP64 general-form term at the 13^3 cube 2.32 -> 0.51 ms (1.98 -> 0.19 ms without the
// walk), FP32 step at the 13^3 cube 3.37 -> 3.13 ms (three axes 0.48 -> 0.25 ms).
template <class TA, int OUT, bool HALF>
__global__ void __launch_bounds__(kRowsThreads) k_contract_rows(
    const __grid_constant__ RowsAxes P, int cap, int win, int max_gp, int max_dof,
    typename Arith<TA>::Out *A, int64_t n_dof, const int32_t *__restrict__ map) {
    using Ar = Arith<TA>;
    constexpr int NACC = HALF ? 2 : 1, LANES = 32 / NACC;   // accumulator rows, lanes per point
    extern __shared__ __align__(16) unsigned char sm_rows[];
    int b = blockIdx.x, axis = 0;
    while (axis < 2 && b >= P.a[axis].n_work) b -= P.a[axis++].n_work;
    const RowsAxis &X = P.a[axis];
    const int4 wk = X.work[b];
    const int bin = wk.x, col0 = wk.y;
    const int d0 = X.dof_off[bin], D = X.dof_off[bin + 1] - d0;
    const int g0 = X.gp_off[bin], G = X.gp_off[bin + 1] - g0;
    const int ld = X.tab_ld[bin];
    const int ncol = min(win, D - col0);
    const float2 *T = X.T + X.tab_off[bin];
    const float2 *S = X.S + X.tab_off[bin] + (int64_t)col0 * ld;
    TA *vals = reinterpret_cast<TA *>(sm_rows);               // [cap]
    TA *accs = vals + cap;                                    // [warps][NACC][win]
    TA *wts = accs + NACC * kRowsWarps * win;                    // [max_gp] s K w
    int *first = reinterpret_cast<int *>(wts + max_gp);       // [max_gp + 1]
    int *cur = first + max_gp + 1;                            // [max_gp]
    int *dofs = cur + max_gp;                                 // [max_dof]
    uint16_t *cols = reinterpret_cast<uint16_t *>(dofs + max_dof);   // [cap]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nchunk = (G + 31) >> 5;
    for (int g = tid; g < G; g += kRowsThreads) {
        cur[g] = 0;
        wts[g] = Ar::weight(X.scale * X.w[X.w_idx ? X.w_idx[g0 + g] : g0 + g]);
    }
    for (int c = tid; c < D; c += kRowsThreads) dofs[c] = X.dof_idx[d0 + c];
    __syncthreads();
    // (chunk of 32 points, one of kRowsWarps row slices) per warp and pass, lane = point
    for (int it = warp; it < nchunk * kRowsWarps; it += kRowsWarps) {
        const int g = 32 * (it / kRowsWarps) + lane;
        if (g >= G) continue;
        int c = 0;
#pragma unroll 8
        for (int r = it % kRowsWarps; r < ncol; r += kRowsWarps) {
            const float2 v = __ldg(S + (int64_t)r * ld + g);
            c += v.x != 0.f || v.y != 0.f;
        }
        if (c) atomicAdd(&cur[g], c);
    }
    __syncthreads();
    if (warp == 0) {   // exclusive scan of the counts
        int carry = 0;
        for (int q = 0; q < G; q += 32) {
            const int c = q + lane < G ? cur[q + lane] : 0;
            int x = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (q + lane < G) first[q + lane] = carry + x - c;
            carry += __shfl_sync(0xffffffffu, x, 31);
        }
        if (lane == 0) first[G] = carry;
    }
    __syncthreads();
    // the warp's accumulator rows, zero between rows, and this lane's
    TA *acc0 = accs + NACC * warp * win;
    for (int c = lane; c < NACC * win; c += 32) acc0[c] = arith_zero<TA>();
    const bool lead = lane < LANES;
    TA *acc = lead ? acc0 : acc0 + win;
    for (int ga = 0; ga < G;) {
        // the group [ga, gb): as many points as fit (all threads find the same gb)
        const int base = first[ga];
        int gb = G;
        if (first[G] - base > cap) {
            int lo = ga + 1, hi = G;   // first[lo] - base <= win <= cap
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (first[mid] - base <= cap) lo = mid;
                else hi = mid;
            }
            gb = lo;
        }
        for (int g = ga + tid; g < gb; g += kRowsThreads) cur[g] = first[g] - base;
        __syncthreads();
        const int ca = ga >> 5, cn = ((gb + 31) >> 5) - ca;
        for (int it = warp; it < cn * kRowsWarps; it += kRowsWarps) {
            const int g = 32 * (ca + it / kRowsWarps) + lane;
            if (g < ga || g >= gb) continue;
#pragma unroll 4
            for (int r = it % kRowsWarps; r < ncol; r += kRowsWarps) {
                const float2 v = __ldg(S + (int64_t)r * ld + g);
                if (v.x != 0.f || v.y != 0.f) {
                    const int k = atomicAdd(&cur[g], 1);
                    vals[k] = Ar::value(v);
                    cols[k] = (uint16_t)r;
                }
            }
        }
        __syncthreads();
        // the rows, each chunk of 32 points' entries of T loaded one chunk ahead
        const int qa = ga & ~31;
        auto load_t = [&](int c1, int q) {
            const int g = q + lane;
            return c1 < D && g >= ga && g < gb ? __ldg(T + (int64_t)c1 * ld + g)
                                               : make_float2(0.f, 0.f);
        };
        float2 tv = load_t(warp, qa);
        for (int c1 = warp; c1 < D; c1 += kRowsWarps) {
            bool any = false;
            for (int q = qa; q < gb; q += 32) {
                const bool more = q + 32 < gb;
                const float2 tn = load_t(more ? c1 : c1 + kRowsWarps, more ? q + 32 : qa);
                const bool nz = tv.x != 0.f || tv.y != 0.f;
                unsigned m = __ballot_sync(0xffffffffu, nz);
                if (m) {
                    any = true;
                    TA t = arith_zero<TA>();
                    int span = 0;   // this lane's point: its first entry and their number
                    if (nz) {
                        const int k0 = first[q + lane];
                        span = (k0 - base) << 12 | (first[q + lane + 1] - k0);
                        t = Ar::weigh(tv, wts[q + lane]);
                    }
                    do {
                        int l = __ffs(m) - 1;
                        m &= m - 1;
                        bool mine = true;
                        if constexpr (HALF) {   // the second half takes the next point
                            mine = lead || m != 0;
                            if (!lead && m != 0) l = __ffs(m) - 1;
                            m &= m - 1;   // (zero stays zero)
                        }
                        const TA tc = Ar::shfl(t, l);
                        const int sp = __shfl_sync(0xffffffffu, span, l);
                        const int k0 = sp >> 12, len = mine ? sp & 0xFFF : 0;
                        for (int o = lane & (LANES - 1); o < len; o += LANES) {
                            const int c = cols[k0 + o];
                            TA x = acc[c];
                            Ar::add(x, tc, vals[k0 + o]);
                            acc[c] = x;
                        }
                        __syncwarp();
                    } while (m);
                }
                tv = tn;
            }
            if (!any) continue;
            const int32_t j1 = dofs[c1];
            for (int cb = lane; cb < ncol; cb += 32 * kRowsFlush) {
                typename Ar::Out v[kRowsFlush];
                int64_t at[kRowsFlush];
#pragma unroll
                for (int u = 0; u < kRowsFlush; u++) {
                    const int c = cb + 32 * u;
                    v[u] = 0;
                    at[u] = -1;
                    if (c < ncol) {
                        const TA a0 = acc0[c], a1 = HALF ? acc0[win + c] : arith_zero<TA>();
                        if (!Ar::zero(a0) || !Ar::zero(a1)) {
                            acc0[c] = arith_zero<TA>();
                            if (HALF) acc0[win + c] = arith_zero<TA>();
                            const int32_t j2 = dofs[col0 + c];
                            at[u] = rows_index<OUT>(n_dof, map, j1, j2);
                            v[u] = Ar::sum(a0, a1);
                            if (OUT != kDense && j1 == j2) v[u] += v[u];   // X(c, c) twice
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < kRowsFlush; u++)
                    if (at[u] >= 0) atomicAdd(&A[at[u]], v[u]);
            }
            __syncwarp();
        }
        ga = gb;
        if (ga < G) __syncthreads();   // the entries are read before the next group's
    }
}

// Algorithmic work of the contraction (the sparse outer products the element sum needs):
// per bin (one CTA) and Gauss point column k, the nonzeros of L[.][k] and R[.][k] over the
// bin's template rows; adds 2 * 2 nnz(L) nnz(R) (two products, one multiply-add each) per
// Gauss point to *flops.
__global__ void __launch_bounds__(128) k_contract_work(
    const float2 *__restrict__ tabL, const float2 *__restrict__ tabR,
    const int32_t *__restrict__ gp_off, const int32_t *__restrict__ dof_off,
    const int64_t *__restrict__ tab_off, const int32_t *__restrict__ tab_ld, double *flops,
    unsigned long long *nnz) {
    const int b = blockIdx.x;
    const int D = dof_off[b + 1] - dof_off[b];
    const int G = gp_off[b + 1] - gp_off[b];
    const int ld = tab_ld[b];
    const float2 *L = tabL + tab_off[b], *R = tabR + tab_off[b];
    double acc = 0.0;
    unsigned long long cnt = 0;
    for (int k = threadIdx.x; k < G; k += blockDim.x) {
        int nl = 0, nr = 0;
        for (int c = 0; c < D; c++) {
            const float2 a = L[(int64_t)c * ld + k], r = R[(int64_t)c * ld + k];
            nl += (a.x != 0.f || a.y != 0.f);
            nr += (r.x != 0.f || r.y != 0.f);
        }
        acc += 4.0 * (double)nl * (double)nr;
        cnt += (unsigned long long)(nl + nr);
    }
    for (int o = 16; o > 0; o >>= 1) {
        acc += __shfl_down_sync(0xffffffffu, acc, o);
        cnt += __shfl_down_sync(0xffffffffu, cnt, o);
    }
    if ((threadIdx.x & 31) == 0 && acc != 0.0) atomicAdd(flops, acc);
    if ((threadIdx.x & 31) == 0 && cnt != 0) atomicAdd(nnz, cnt);
}

// wc[g] = w[g] c[g] (c NULL: w)
__global__ void k_weight_coef(const double *__restrict__ w, const double *__restrict__ c,
                              int64_t n, double *wc) {
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g < n) wc[g] = c ? w[g] * c[g] : w[g];
}

}  // namespace

int weight_coef(Mesh *m, const double *c_gp, double *wc_gp) {
    k_weight_coef<<<(unsigned)((m->n_gp + 255) / 256), 256, 0, m->stream>>>(m->gw, c_gp, m->n_gp,
                                                                             wc_gp);
    note_launch(m);
    FEM3_CUDA(cudaGetLastError());
    return FEM3_OK;
}

// one launch of k_contract_rows over the axes of P (an axis without work has n_work = 0)
template <class TA, int OUT>
static int launch_rows(Mesh *m, const RowsAxes &P, typename Arith<TA>::Out *A,
                       const int32_t *map = nullptr) {
    int64_t nw = 0;
    int max_dof = 1, max_gp = 1;
    for (int axis = 0; axis < 3; axis++) {
        if (!P.a[axis].n_work) continue;
        nw += P.a[axis].n_work;
        max_dof = std::max(max_dof, m->bins[axis].max_dof);
        max_gp = std::max(max_gp, m->bins[axis].max_gp);
    }
    if (nw == 0) return FEM3_OK;
    // room for a third of the largest block's entries (a fifth are nonzero on the
    // configured meshes), 48 KB at most: three CTAs or more per SM
    const int win = std::min(max_dof, kRowsWindow);
    const bool half = max_dof <= kRowsHalfMax;
    const int64_t entry = sizeof(TA) + sizeof(uint16_t);
    const int cap = (int)std::max<int64_t>(
        win, std::min<int64_t>((int64_t)win * max_gp / 3 + 64, kRowsEntryBytes / entry));
    const size_t sh = (sizeof(TA) * (cap + (size_t)(half ? 2 : 1) * kRowsWarps * win + max_gp) +
                       sizeof(int) * (2 * (size_t)max_gp + 1 + max_dof) +
                       sizeof(uint16_t) * cap + 15) &
                      ~size_t(15);
    FEM3_CUDA(device_smem(half ? (const void *)k_contract_rows<TA, OUT, true>
                               : (const void *)k_contract_rows<TA, OUT, false>,
                          kRowsSmemMax));
    const int kc = OUT == kBlocks ? KC_OPERATOR : KC_CONTRACT;
    kc_begin(m, kc);
    if (half)
        k_contract_rows<TA, OUT, true><<<(unsigned)nw, kRowsThreads, sh, m->stream>>>(
            P, cap, win, max_gp, max_dof, A, m->n_dof, map);
    else
        k_contract_rows<TA, OUT, false><<<(unsigned)nw, kRowsThreads, sh, m->stream>>>(
            P, cap, win, max_gp, max_dof, A, m->n_dof, map);
    kc_end(m, kc);
    note_launch(m);
    FEM3_CUDA(cudaGetLastError());
    return FEM3_OK;
}

static int clear_matrix(Mesh *m, int precision) {
    const int64_t n = m->n_dof;
    if (precision == FEM3_FP64)
        FEM3_CUDA(cudaMemsetAsync(m->A64, 0, sizeof(double) * n * n, m->stream));
    else
        FEM3_CUDA(cudaMemsetAsync(m->A32, 0, sizeof(float) * n * n, m->stream));
    return FEM3_OK;
}

// K = T^T diag(wc) S over one axis's bins on CUDA cores (FP64 into A64 or FP32 into A32),
// T the test side's table (R if test_right), S the trial side's
int contract_form(Mesh *m, int axis, bool test_right, const double *wc_gp, int precision) {
    AxisBins &B = m->bins[axis];
    FEM3_TRY(clear_matrix(m, precision));
    RowsAxes P{};
    P.a[axis] = RowsAxis{test_right ? m->tabR[axis] : m->tabL[axis],
                         test_right ? m->tabL[axis] : m->tabR[axis], B.work, B.gp_off,
                         B.dof_off, B.dof_idx, B.tab_ld, B.tab_off, wc_gp, B.gp_idx, 1.0,
                         B.n_work};
    return precision == FEM3_FP64 ? launch_rows<double, kDense>(m, P, m->A64)
                                  : launch_rows<float, kDense>(m, P, m->A32);
}

int contract_work(Mesh *m, double *flops_out, int64_t *nnz_out) {
    cudaStream_t s = m->stream;
    double *d = m->norms + 121;
    unsigned long long *c = reinterpret_cast<unsigned long long *>(m->norms + 122);
    FEM3_CUDA(cudaMemsetAsync(d, 0, 2 * sizeof(double), s));
    for (int axis = 0; axis < 3; axis++) {
        AxisBins &B = m->bins[axis];
        if (B.n_bins == 0 || B.n_tmpl == 0) continue;
        k_contract_work<<<B.n_bins, 128, 0, s>>>(m->tabL[axis], m->tabR[axis], B.gp_off,
                                                  B.dof_off, B.tab_off, B.tab_ld, d, c);
        note_launch(m);
    }
    FEM3_CUDA(cudaGetLastError());
    FEM3_CUDA(cudaMemcpyAsync(m->h_norms + 121, d, 2 * sizeof(double), cudaMemcpyDeviceToHost, s));
    FEM3_CUDA(cudaStreamSynchronize(s));
    if (flops_out) *flops_out = m->h_norms[121];
    if (nnz_out) {
        unsigned long long v;
        memcpy(&v, m->h_norms + 122, sizeof(v));
        *nnz_out = (int64_t)v;
    }
    return FEM3_OK;
}

// Power of two next to the largest |s_i K_i|.  s K w is formed before the products, so as a pair (24 bits
// below 2^-74, nothing below 2^-126) it has to be of the weights' order for the coefficients'
// scale not to cost digits; the factor stays with the blocks, whose entries are split likewise.
static int coef_exponent(const Mesh *m) {
    int e;
    frexp(std::max({fabs(m->sK[0]), fabs(m->sK[1]), fabs(m->sK[2])}), &e);
    return std::min(std::max(e, -126), 126);
}

// the work items of this part's bins of every axis (the lists are in bin order), the
// coefficients times 2^-e
static RowsAxes riesz_axes(Mesh *m, int e) {
    RowsAxes P{};
    for (int axis = 0; axis < 3; axis++) {
        AxisBins &B = m->bins[axis];
        int b0, b1;
        part_bins(m, axis, b0, b1);
        const auto lb = [&](int b) {
            return (int)(std::lower_bound(B.h_work.begin(), B.h_work.end(), b,
                                          [](const int4 &x, int v) { return x.x < v; }) -
                         B.h_work.begin());
        };
        const int w0 = lb(b0), nw = std::max(0, lb(b1) - w0);
        P.a[axis] = RowsAxis{m->tabL[axis], m->tabR[axis], B.work + w0, B.gp_off, B.dof_off,
                             B.dof_idx, B.tab_ld, B.tab_off, B.w_slot, nullptr, ldexp(m->sK[axis], -e), nw};
    }
    return P;
}

// the lower triangle of A (all that the factorisation reads)
int contract(Mesh *m, int precision) {
    double flops = 0;
    FEM3_TRY(clear_matrix(m, precision));
    for (int axis = 0; axis < 3; axis++) {
        const AxisBins &B = m->bins[axis];
        for (int b = 0; b < B.n_bins; b++) {
            double D = B.h_dof_off[b + 1] - B.h_dof_off[b];
            double G = B.h_gp_off[b + 1] - B.h_gp_off[b];
            flops += 2.0 * D * D * G;
        }
    }
    const RowsAxes P = riesz_axes(m, 0);
    m->contract_flops = flops;
    return precision == FEM3_FP64 ? launch_rows<double, kLower>(m, P, m->A64)
                                  : launch_rows<float, kLower>(m, P, m->A32);
}

// the lower blocks of the operator over O.scale, added in FP64 from double-float row sums
int contract_blocks(Mesh *m, OpBlocks &O) {
    const int e = coef_exponent(m);
    O.scale = ldexp(1.0, e);
    return launch_rows<float2, kBlocks>(m, riesz_axes(m, e), O.low, O.map);
}

}  // namespace fem3
