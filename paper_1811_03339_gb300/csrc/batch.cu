// Batched assembly and solve of many meshes of uneven size (not in the paper: the paper
// assembles one mesh at a time).  One launch walks every Gauss-point line of every mesh;
// contraction, load vector, factorisation and refinement sweeps of each mesh run on internal
// streams so that meshes overlap (a sweep's triangular solves are a chain of launches per
// mesh, latency-bound, so the meshes' chains run side by side); all residuals are checked
// with one host wait per sweep, and none is formed in less than double-float arithmetic.  12 meshes of
// 6 to 20 cells per side, 16 columns: 49.3 ms a run with block-step solves over the whole batch (1,100
// launches, 13.3 ms), 21.3 ms now that each internal stream has factorisation streams of its own (one
// set for all made the large meshes' blocked factorisations follow each other: 26.8 ms).  Last sweeps
// in plain FP32, as the single-mesh solve has them, would take 20.8 ms, but a run's residuals have always
// been FP64-accurate (those sweeps leave them off by up to 3e-14 of b).
//
// The assembly and factorisation of the whole batch (walk, contractions, factorisations) is captured as one CUDA
// graph the second time a run has the same orders, coefficients and precision, and replayed
// as one graph launch from then on (the first run goes eagerly: it makes the allocations, the
// tile tuner's timings and the factorisation's side streams that a capture must not make).
// The load vectors are formed beside the graph, so new right-hand sides need no new capture.
// The refinement sweeps stay host-driven: each one
// checks the residuals before the next.
#include <math.h>

#include <algorithm>
#include <string>
#include <utility>
#include <vector>

#include "fem3_impl.cuh"

namespace fem3 {

struct Batch {
    std::vector<Mesh *> ms;
    std::vector<cudaStream_t> streams;
    std::vector<cudaEvent_t> done;   // one per internal stream
    std::vector<SideCtx *> side;     // factorisation streams, likewise
    cudaEvent_t fork = nullptr;
    BatchWalkScratch ws;
    // per-mesh run buffers, kept across runs: load vector b and the refinement's vectors
    std::vector<double *> bv;
    std::vector<RefineVecs> rv;
    int nrhs_cap = 0;
    // the captured assembly + factorisation and what it was captured for
    cudaGraphExec_t exec = nullptr;
    // the capture runs on a private stream (the caller's may be the legacy stream, which
    // cannot be captured); it starts after the work enqueued so far on the caller's stream
    cudaStream_t cap = nullptr;
    cudaEvent_t cap_in = nullptr;
    std::vector<double> key_ak;          // alpha, K
    // per mesh, what the captured work leaves: whether it builds the operator, and its scale
    std::vector<std::pair<bool, double>> key_op;
    int key_prec = -1;
    int runs = 0;                        // eager runs so far
    int graph_launches = 0;              // replays so far
};

static void free_run_buffers(Batch *b) {
    for (double *p : b->bv) cudaFree(p);
    for (const RefineVecs &v : b->rv) {
        cudaFree(v.r);
        cudaFree(v.Au);
        cudaFree(v.dc);
    }
    b->bv.clear();
    b->rv.clear();
    b->nrhs_cap = 0;
}

static void batch_destroy(Batch *b) {
    if (!b) return;
    for (cudaStream_t s : b->streams) cudaStreamSynchronize(s);
    if (b->exec) cudaGraphExecDestroy(b->exec);
    free_run_buffers(b);
    for (Mesh *m : b->ms) fem3_mesh_free(reinterpret_cast<fem3_mesh>(m));
    for (cudaEvent_t e : b->done) cudaEventDestroy(e);
    for (SideCtx *c : b->side) side_destroy(c);
    for (cudaStream_t s : b->streams) cudaStreamDestroy(s);
    if (b->fork) cudaEventDestroy(b->fork);
    if (b->cap) cudaStreamDestroy(b->cap);
    if (b->cap_in) cudaEventDestroy(b->cap_in);
    cudaFree(b->ws.d_desc);
    cudaFreeHost(b->ws.h_desc);
    delete b;
}

// every internal stream waits for the work enqueued so far on `s`
static int fork_to(Batch *b, cudaStream_t s) {
    FEM3_CUDA(cudaEventRecord(b->fork, s));
    for (cudaStream_t t : b->streams) FEM3_CUDA(cudaStreamWaitEvent(t, b->fork, 0));
    return FEM3_OK;
}
// `s` waits for the work enqueued so far on every internal stream
static int join_to(Batch *b, cudaStream_t s) {
    for (size_t k = 0; k < b->streams.size(); k++) {
        FEM3_CUDA(cudaEventRecord(b->done[k], b->streams[k]));
        FEM3_CUDA(cudaStreamWaitEvent(s, b->done[k], 0));
    }
    return FEM3_OK;
}

static int check_mesh(Mesh *m, int i) {
    int32_t e[ERR_COUNT];
    FEM3_TRY(read_errors(m, e));
    const std::string who = "mesh " + std::to_string(i) + ": ";
    if (e[ERR_WALK]) return set_error(FEM3_E_WALK, who + "a path walk exceeded its step cap");
    if (e[ERR_TEMPLATE]) return set_error(FEM3_E_TEMPLATE, who + "table update outside the template");
    if (e[ERR_NOT_SPD]) {
        cudaMemsetAsync(m->err + ERR_NOT_SPD, 0, sizeof(int32_t), m->stream);
        return set_error(FEM3_E_NOT_SPD, who + "non-positive pivot at column " +
                                             std::to_string(e[ERR_NOT_SPD] - 1));
    }
    if (e[ERR_TC] || e[ERR_SOLVE] || e[ERR_CHOL]) return set_error(FEM3_E_CUDA, who + "a bounded wait expired");
    return FEM3_OK;
}

}  // namespace fem3

using namespace fem3;

extern "C" {

int fem3_batch_create(int n_meshes, const double *const *verts, const int64_t *n_nodes,
                      const int32_t *const *tets, const int64_t *n_tets, const fem3_options *opt,
                      void *stream, fem3_batch *out) {
    if (!out || n_meshes < 1 || !verts || !n_nodes || !tets || !n_tets)
        return set_error(FEM3_E_ARG, "bad argument");
    *out = nullptr;
    Batch *b = new Batch();
    for (int i = 0; i < n_meshes; i++) {
        fem3_mesh h = nullptr;
        int st = fem3_mesh_upload(verts[i], n_nodes[i], tets[i], n_tets[i], opt, stream, &h);
        if (st != FEM3_OK) {
            batch_destroy(b);
            return st;
        }
        b->ms.push_back(reinterpret_cast<Mesh *>(h));
    }
    const int ns = std::min(n_meshes, 8);
    for (int k = 0; k < ns; k++) {
        cudaStream_t s;
        cudaEvent_t e;
        if (cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) != cudaSuccess ||
            cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) {
            batch_destroy(b);
            return cuda_error(cudaGetLastError(), "stream/event creation");
        }
        b->streams.push_back(s);
        b->done.push_back(e);
        SideCtx *c = nullptr;
        if (int st = side_make(&c)) {
            batch_destroy(b);
            return st;
        }
        b->side.push_back(c);
    }
    if (cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&b->cap_in, cudaEventDisableTiming) != cudaSuccess ||
        cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking) != cudaSuccess) {
        batch_destroy(b);
        return cuda_error(cudaGetLastError(), "batch allocation");
    }
    *out = reinterpret_cast<fem3_batch>(b);
    return FEM3_OK;
}

int fem3_batch_mesh(fem3_batch hb, int i, fem3_mesh *out) {
    Batch *b = reinterpret_cast<Batch *>(hb);
    if (!b || !out || i < 0 || i >= (int)b->ms.size()) return set_error(FEM3_E_ARG, "bad argument");
    *out = reinterpret_cast<fem3_mesh>(b->ms[i]);
    return FEM3_OK;
}

int fem3_batch_run(fem3_batch hb, const double *alpha, const double *K, int precision,
                   const double *const *f, int nrhs, double tol, int max_iter, double *const *u,
                   int *iters, double *resid, void *stream) {
    Batch *b = reinterpret_cast<Batch *>(hb);
    if (!b || !alpha || !K || !f || !u || nrhs < 1 || nrhs > 16)
        return set_error(FEM3_E_ARG, "bad argument (1 <= nrhs <= 16)");
    if (precision != FEM3_FP64 && precision != FEM3_TF32X3 && precision != FEM3_FP32 &&
        precision != FEM3_BF16X3)
        return set_error(FEM3_E_ARG, "unknown precision");
    const int n = (int)b->ms.size();
    cudaStream_t cs = reinterpret_cast<cudaStream_t>(stream);
    for (int i = 0; i < n; i++)
        for (int a = 0; a < 3; a++) {
            if (!(alpha[3 * i + a] > 1.0 && alpha[3 * i + a] <= 2.0))
                return set_error(FEM3_E_ARG, "alpha must lie in (1, 2]");
            if (!(K[3 * i + a] > 0.0)) return set_error(FEM3_E_ARG, "K must be positive");
        }
    if (max_iter <= 0) max_iter = 50;
    const bool fp64 = precision == FEM3_FP64;

    // host-side state of every mesh for this run (the refinement reads it)
    for (int i = 0; i < n; i++) {
        Mesh *m = b->ms[i];
        m->stream = cs;
        const int64_t nd = m->n_dof;
        if (fp64 && !m->A64) FEM3_TRY(dev_alloc_t(m, &m->A64, std::max<int64_t>(1, nd * nd)));
        if (!fp64 && !m->A32) FEM3_TRY(dev_alloc_t(m, &m->A32, std::max<int64_t>(1, nd * nd)));
        for (int a = 0; a < 3; a++) {
            m->alpha[a] = alpha[3 * i + a];
            m->K[a] = K[3 * i + a];
            m->s[a] = 1.0 / (2.0 * cos(M_PI * m->alpha[a] / 2.0));
            m->sK[a] = m->s[a] * m->K[a];
        }
        m->precision = precision;
        m->factored = false;
        m->op_ready = false;
        m->integer_order = false;   // of an earlier assembly through the mesh's handle
        m->nonsym = false;
    }
    // the operators' block patterns and storage (the first run's; one wait for all of them)
    for (Mesh *m : b->ms)
        if (m->n_dof > 0) FEM3_TRY(op_count(m));
    for (Mesh *m : b->ms)
        if (m->n_dof > 0) FEM3_TRY(op_prepare(m, !fp64));
    // run buffers for nrhs columns (kept across runs)
    if (b->nrhs_cap < nrhs) {
        for (cudaStream_t t : b->streams) FEM3_CUDA(cudaStreamSynchronize(t));
        FEM3_CUDA(cudaStreamSynchronize(cs));
        free_run_buffers(b);
        b->bv.assign(n, nullptr);
        b->rv.assign(n, RefineVecs{});
        for (int i = 0; i < n; i++) {
            const size_t nn = (size_t)std::max<int64_t>(1, b->ms[i]->n_dof * nrhs);
            RefineVecs &v = b->rv[i];
            if (cudaMalloc((void **)&b->bv[i], sizeof(double) * nn) != cudaSuccess ||
                cudaMalloc((void **)&v.r, sizeof(double) * nn) != cudaSuccess ||
                cudaMalloc((void **)&v.Au, sizeof(double) * nn) != cudaSuccess ||
                cudaMalloc((void **)&v.dc, sizeof(float) * 2 * nn) != cudaSuccess)
                return cuda_error(cudaGetLastError(), "cudaMalloc (batch run buffers)");
        }
        b->nrhs_cap = nrhs;
    }

    // 1 + 2: walk of every line of every mesh (one launch on the caller's stream), then per
    // mesh on the internal streams contraction and factorisation; replayed from
    // the captured graph when the run matches the one it was captured for
    std::vector<double> ak(alpha, alpha + 3 * n);
    ak.insert(ak.end(), K, K + 3 * n);
    const bool same = b->exec && b->key_prec == precision && b->key_ak == ak;
    auto enqueue_assembly = [&](cudaStream_t os) -> int {
        FEM3_TRY(walk_tables_batch(b->ms.data(), n, alpha, os, &b->ws));
        FEM3_TRY(fork_to(b, os));
        for (int i = 0; i < n; i++) {
            Mesh *m = b->ms[i];
            m->stream = b->streams[i % b->streams.size()];
            if (m->n_dof == 0) continue;
            if (precision == FEM3_TF32X3 || precision == FEM3_BF16X3)
                FEM3_TRY(contract_tc(m, precision == FEM3_BF16X3));
            else
                FEM3_TRY(contract(m, precision));
            m->lent = b->side[i % b->streams.size()];
            const int fst = factor(m);
            m->lent = nullptr;
            FEM3_TRY(fst);
        }
        FEM3_TRY(join_to(b, os));
        return FEM3_OK;
    };
    int st = FEM3_OK;
    if (same) {
        FEM3_CUDA(cudaGraphLaunch(b->exec, cs));
        b->graph_launches++;
        // the replay has built (FP64: copied) the operators that the captured run did
        for (int i = 0; i < n; i++) {
            b->ms[i]->op_ready = b->key_op[i].first;
            b->ms[i]->op.scale = b->key_op[i].second;
        }
    } else if (b->runs >= 1) {
        // capture the assembly + factorisation; on any failure discard it and run eagerly
        if (b->exec) {
            FEM3_CUDA(cudaStreamSynchronize(cs));
            cudaGraphExecDestroy(b->exec);
            b->exec = nullptr;
        }
        cudaGraph_t g = nullptr;
        bool captured = false;
        FEM3_CUDA(cudaEventRecord(b->cap_in, cs));
        FEM3_CUDA(cudaStreamWaitEvent(b->cap, b->cap_in, 0));
        if (cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
            const int cst = enqueue_assembly(b->cap);
            const cudaError_t ce = cudaStreamEndCapture(b->cap, &g);
            if (cst == FEM3_OK && ce == cudaSuccess && g &&
                cudaGraphInstantiate(&b->exec, g, 0) == cudaSuccess) {
                captured = true;
                b->key_prec = precision;
                b->key_ak = ak;
                b->key_op.clear();
                for (const Mesh *m : b->ms) b->key_op.emplace_back(m->op_ready, m->op.scale);
            }
            if (g) cudaGraphDestroy(g);
        }
        cudaGetLastError();
        if (captured) {
            FEM3_CUDA(cudaGraphLaunch(b->exec, cs));
            b->graph_launches++;
        } else {
            b->exec = nullptr;
            for (Mesh *m : b->ms) m->op_ready = false;   // the capture built none
            st = enqueue_assembly(cs);
        }
    } else {
        st = enqueue_assembly(cs);
        b->runs++;
    }
    // 3. per mesh on its stream: load vector, then refinement from u = 0 (FP64: a direct solve)
    if (st == FEM3_OK) st = fork_to(b, cs);
    std::vector<char> active(n, 0);
    std::vector<RefineState> q(n);
    int n_active = 0;
    for (int i = 0; i < n && st == FEM3_OK; i++) {
        Mesh *m = b->ms[i];
        m->stream = b->streams[i % b->streams.size()];
        if (m->n_dof == 0) continue;
        m->factored = true;
        if ((st = load_vector(m, f[i], nrhs, b->bv[i])) != FEM3_OK) break;
        if (fp64) {
            st = solve_direct(m, b->bv[i], nrhs, u[i]);
            continue;
        }
        b->rv[i].b = b->bv[i];
        b->rv[i].u = u[i];
        st = refine_start(b->rv[i], m->n_dof, nrhs, m->stream);
        active[i] = 1;
        n_active++;
    }
    while (n_active > 0 && st == FEM3_OK) {
        for (int i = 0; i < n && st == FEM3_OK; i++)
            if (active[i]) st = refine_sweep(b->ms[i], b->rv[i], nrhs, q[i].mode);
        for (cudaStream_t t : b->streams) FEM3_CUDA(cudaStreamSynchronize(t));
        for (int i = 0; i < n && st == FEM3_OK; i++) {
            if (!active[i] || refine_next(b->ms[i], nrhs, tol, max_iter, false, &q[i])) continue;
            active[i] = 0;
            n_active--;
        }
    }

    // 4. join into the caller's stream, report
    FEM3_TRY(join_to(b, cs));
    if (st != FEM3_OK) return st;
    int bad = FEM3_OK;
    for (int i = 0; i < n; i++) {
        Mesh *m = b->ms[i];
        m->stream = cs;
        if (iters) iters[i] = q[i].sweeps;
        if (resid) resid[i] = fp64 || m->n_dof == 0 ? 0.0 : q[i].worst;
        int e = check_mesh(m, i);
        if (e != FEM3_OK && bad == FEM3_OK) bad = e;
        if (!fp64 && m->n_dof > 0 && !q[i].converged && bad == FEM3_OK)
            bad = set_error(FEM3_E_NO_CONVERGE, "mesh " + std::to_string(i) +
                                                    ": iterative refinement did not converge");
    }
    return bad;
}

int fem3_batch_graph_launches(fem3_batch hb, int64_t *n) {
    Batch *b = reinterpret_cast<Batch *>(hb);
    if (!b || !n) return set_error(FEM3_E_ARG, "bad argument");
    *n = b->graph_launches;
    return FEM3_OK;
}

void fem3_batch_free(fem3_batch hb) { batch_destroy(reinterpret_cast<Batch *>(hb)); }

}  // extern "C"
