// Contraction A = sum_i s_i K_i (L_i^T W R_i + R_i^T W L_i) on CUDA cores, bin by bin
// (Section 2.1 element sum, Section 2.3 template: only dofs of a bin's template set can
// meet the bin's Gauss points, so each bin contributes to a D_b x D_b block), from the
// nonzeros of the bin's table blocks (about a fifth of their entries: k_contract_rows).
#include <algorithm>
#include <cstring>
#include <vector>

#include "fem3_impl.cuh"

namespace fem3 {

namespace {

constexpr int kRowsThreads = 256, kRowsWarps = kRowsThreads / 32;
constexpr int kRowsEntryBytes = 48 * 1024;   // compacted entries in shared memory, at most
// the largest launch: entries, FP64 accumulator rows, offsets and cursors of the points
constexpr size_t kRowsSmemMax = kRowsEntryBytes + sizeof(double) * kRowsWarps * kRowsWindow +
                                sizeof(int) * (2 * kMaxBinItems + 1) + 64;

// table entry (hi + lo pair) in the arithmetic type of the contraction; the FP64 value is
// assembled from the pair's bits (f32 -> f64 conversions run at the FP64 rate) and one add
template <class TA>
__device__ __forceinline__ TA pair_value(float2 v) {
    if constexpr (sizeof(TA) == 8) return f32_to_f64_exact(v.x) + f32_to_f64_exact(v.y);
    else return v.x + v.y;
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
//   2. warp = row c1: its accumulator row lives in shared memory; for every Gauss point
//      with T[c1][r] != 0 the lanes take the point's entries, acc[c2] += (w T) S;
//   3. the row's nonzeros go to A: with FULL to A[dof c1][dof c2] (general form), else to the
//      lower triangle only, where X(c1, c2) and X(c2, c1) land on the same element (the fold
//      A = s K (X + X^T); the diagonal gets 2 X).
// Points go in groups whose entries fit `cap` (>= win, so a group holds at least one point);
// usually one group.  TA is the arithmetic type: double (FP64 form) or float (FP32 form).
//
// Bound: shared-memory latency and the FP64 pipe (1/64 of the FP32 rate).  A dense 64 x 64
// tile product over the same blocks does 15 to 30 times the sum over points of
// nnz(T) nnz(S); here a point's entries are about one warp-wide pass (1.5 n on a mesh of n
// cells per side, both sides together 3 n).  Measured against that tile product, GB300: FP64
// assemble + solve of the 11^3 parallelepiped 9.57 -> 5.03 ms (contraction 4.76 -> 0.21 ms),
// one FP64 general-form term at the 13^3 cube 2.32 -> 0.51 ms (1.98 -> 0.19 ms without the
// walk), FP32 step at the 13^3 cube 3.37 -> 3.13 ms (three axes 0.48 -> 0.25 ms).
template <class TA, bool FULL>
__global__ void __launch_bounds__(kRowsThreads) k_contract_rows(
    const __grid_constant__ RowsAxes P, int cap, int win, int max_gp, TA *A, int64_t n_dof) {
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
    TA *accs = vals + cap;                                    // [warps][win]
    int *first = reinterpret_cast<int *>(accs + kRowsWarps * win);   // [max_gp + 1]
    int *cur = first + max_gp + 1;                            // [max_gp]
    uint16_t *cols = reinterpret_cast<uint16_t *>(cur + max_gp);     // [cap]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nchunk = (G + 31) >> 5;
    for (int g = tid; g < G; g += kRowsThreads) cur[g] = 0;
    __syncthreads();
    // (chunk of 32 points, one of kRowsWarps row slices) per warp and pass, lane = point
    for (int it = warp; it < nchunk * kRowsWarps; it += kRowsWarps) {
        const int g = 32 * (it / kRowsWarps) + lane;
        if (g >= G) continue;
        int c = 0;
#pragma unroll 4
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
    TA *acc = accs + warp * win;
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
                    vals[k] = pair_value<TA>(v);
                    cols[k] = (uint16_t)r;
                }
            }
        }
        __syncthreads();
        for (int c1 = warp; c1 < D; c1 += kRowsWarps) {
            for (int c = lane; c < ncol; c += 32) acc[c] = TA(0);
            __syncwarp();
            bool any = false;
            for (int q = ga & ~31; q < gb; q += 32) {
                const int g = q + lane;
                float2 tv = make_float2(0.f, 0.f);
                if (g >= ga && g < gb) tv = __ldg(T + (int64_t)c1 * ld + g);
                const bool nz = tv.x != 0.f || tv.y != 0.f;
                unsigned m = __ballot_sync(0xffffffffu, nz);
                if (!m) continue;
                any = true;
                TA t = TA(0);
                if (nz) t = pair_value<TA>(tv) * (TA)X.w[X.w_idx ? X.w_idx[g0 + g] : g0 + g];
                while (m) {
                    const int l = __ffs(m) - 1;
                    m &= m - 1;
                    const TA tc = __shfl_sync(0xffffffffu, t, l);
                    const int k1 = first[q + l + 1] - base;
                    for (int k = first[q + l] - base + lane; k < k1; k += 32) {
                        const int c = cols[k];
                        acc[c] = fma(tc, vals[k], acc[c]);
                    }
                    __syncwarp();
                }
            }
            if (any) {
                const int64_t j1 = X.dof_idx[d0 + c1];
                const TA sc = (TA)X.scale;
                for (int c = lane; c < ncol; c += 32) {
                    const TA v = acc[c];
                    if (v == TA(0)) continue;
                    const int64_t j2 = X.dof_idx[d0 + col0 + c];
                    if constexpr (FULL)
                        atomicAdd(&A[j1 * n_dof + j2], sc * v);
                    else
                        atomicAdd(&A[(j1 > j2 ? j1 : j2) * n_dof + (j1 > j2 ? j2 : j1)],
                                  (j1 == j2 ? TA(2) : TA(1)) * sc * v);
                }
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
template <class TA, bool FULL>
static int launch_rows(Mesh *m, const RowsAxes &P, TA *A) {
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
    const int64_t entry = sizeof(TA) + sizeof(uint16_t);
    const int cap = (int)std::max<int64_t>(
        win, std::min<int64_t>((int64_t)win * max_gp / 3 + 64, kRowsEntryBytes / entry));
    const size_t sh = (sizeof(TA) * (cap + (size_t)kRowsWarps * win) +
                       sizeof(int) * (2 * (size_t)max_gp + 1) + sizeof(uint16_t) * cap + 15) &
                      ~size_t(15);
    static bool attr = false;
    if (!attr) {
        FEM3_CUDA(cudaFuncSetAttribute(k_contract_rows<TA, FULL>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kRowsSmemMax));
        attr = true;
    }
    kc_begin(m, KC_CONTRACT);
    k_contract_rows<TA, FULL><<<(unsigned)nw, kRowsThreads, sh, m->stream>>>(P, cap, win, max_gp,
                                                                            A, m->n_dof);
    kc_end(m, KC_CONTRACT);
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
    return precision == FEM3_FP64 ? launch_rows<double, true>(m, P, m->A64)
                                  : launch_rows<float, true>(m, P, m->A32);
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

// the lower triangle of A (all that the factorisation reads)
int contract(Mesh *m, int precision) {
    double flops = 0;
    FEM3_TRY(clear_matrix(m, precision));
    RowsAxes P{};
    for (int axis = 0; axis < 3; axis++) {
        AxisBins &B = m->bins[axis];
        for (int b = 0; b < B.n_bins; b++) {
            double D = B.h_dof_off[b + 1] - B.h_dof_off[b];
            double G = B.h_gp_off[b + 1] - B.h_gp_off[b];
            flops += 2.0 * D * D * G;
        }
        // the work items of this part's bins (the list is in bin order)
        int b0, b1;
        part_bins(m, axis, b0, b1);
        const auto lb = [&](int b) {
            return (int)(std::lower_bound(B.h_work.begin(), B.h_work.end(), b,
                                          [](const int4 &x, int v) { return x.x < v; }) -
                         B.h_work.begin());
        };
        const int w0 = lb(b0), nw = std::max(0, lb(b1) - w0);
        P.a[axis] = RowsAxis{m->tabL[axis], m->tabR[axis], B.work + w0, B.gp_off, B.dof_off,
                             B.dof_idx, B.tab_ld, B.tab_off, B.w_slot, nullptr, m->sK[axis], nw};
    }
    m->contract_flops = flops;
    return precision == FEM3_FP64 ? launch_rows<double, false>(m, P, m->A64)
                                  : launch_rows<float, false>(m, P, m->A32);
}

}  // namespace fem3
