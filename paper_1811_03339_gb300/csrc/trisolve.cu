// Triangular solves L y = b, L^T x = y with a dense Cholesky factor and many right-hand sides.
//
// A substitution is latency-bound: a step per block of rows, each waiting for the last.  So the
// steps are few and wide.  Once per factorisation the inverses of the B x B diagonal blocks of L
// are built from the factorisation's 64 x 64 ones by doubling (tri_prepare); a solve is then,
// per block J and direction, two launches over the whole chip: y_J = L_JJ^{-1} t_J, and
// t_I -= L_IJ y_J for every later block I (k_tri_rows forward, k_tri_cols, the transposes, on
// the way back).  What bounds a launch is the read of its matrix block (HBM for the updates of
// large factors) and the launch itself, about 2.5 us, of which the chaining hides a part.
//
// B: doubling to B costs n B^2 / 3 multiply-adds, a step less saves two launches per
// direction and solve.  FP32: 1024 above n = 4,096 (n = 12,167: 0.29 ms once, 12 steps per
// direction; at n = 3,375 the last doubling cost more than it gave: 0.33 against 0.10 ms), else 512.  FP64,
// where 1/64 of the FP32 rate makes the doubling dear: 256, or one block of 512 for n <= 512.
//
// Measured (GB300), both directions, against one CTA walking 64-row blocks with worker CTAs
// feeding it partial sums through flags: 17 columns at n = 12,167 1.40 -> 0.99 ms, eight at n = 6,859
// 0.49 -> 0.32 ms, FP64 four columns at n = 1,000 0.31 -> 0.16 ms, one at n = 343 47 -> 14 us.
// Chaining the launches (launch_chained) then took the eight-column refined solve at n = 6,859 from
// 1.77 to 1.62 ms and the 16^3 TF32 x 3 step from 4.31 to 4.16 ms (24^3: 28.1 ms either way, the
// updates take about eight rounds of loads and products one after another there, on 350 CTAs or
// fewer: 0.8 TB/s, an eighth of HBM's rate); without the fetches into L2 the former is 1.70 ms.
#include <algorithm>

#include "fem3_impl.cuh"

namespace fem3 {

namespace {

constexpr int kTriThreads = 256, kTriWarps = kTriThreads / 32;   // k_tri_rows
constexpr int kColThreads = 512, kColWarps = kColThreads / 32;   // k_tri_cols

// The launches of a solve are chained (programmatic dependent launch): a kernel starts while
// the one before it finishes, fetches its share of the matrix (which no launch of the solve
// writes) into L2, and only then waits for the vectors.  Every wait is for the whole launch
// before, which itself waited for its own, so the order of reads and writes is the stream's.
__device__ __forceinline__ void chain_next() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void chain_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void fetch_l2(const void *p) {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

template <class... KP, class... Args>
int launch_chained(bool first, void (*kernel)(KP...), int64_t grid, int threads, size_t sh,
                   cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = sh;
    cfg.stream = s;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = first ? 0 : 1;   // the first waits for whatever wrote the matrix
    FEM3_CUDA(cudaLaunchKernelEx(&cfg, kernel, static_cast<KP>(args)...));
    return FEM3_OK;
}

// diagonal 64 x 64 inverses into the B x B blocks
template <class TF>
__global__ void __launch_bounds__(256) k_tri_seed(const TF *__restrict__ dinv, int B, TF *inv) {
    const int per = B / 64, b = blockIdx.x / per, o = blockIdx.x % per * 64;
    const TF *D = dinv + (int64_t)blockIdx.x * 64 * 64;
    TF *I = inv + (int64_t)b * B * B;
    for (int e = threadIdx.x; e < 64 * 64; e += 256)
        I[(int64_t)(o + (e >> 6)) * B + o + (e & 63)] = D[e];
}

// One doubling step, block width m -> 2 m: [X11 0; X21 X22] with X21 = -X22 (L21 X11), for
// every pair blockIdx.y.  phase 0: T = L21 X11 into the unused block above X22; phase 1: X21.
// Blocks of X11 and X22 above their diagonal hold earlier T: the sums run over the triangular
// parts only (to a multiple of TILE; within a 64 x 64 diagonal inverse the rest is zero).
// TILE x TILE outputs per CTA, Q x Q per thread.
template <class TF, int TILE, int Q>
__global__ void __launch_bounds__(256) k_tri_double(const TF *__restrict__ L, int64_t n, int B, int m,
                                                    int phase, TF *inv) {
    constexpr int KC = 16, TX = TILE / Q;
    static_assert(TX * TX == 256, "256 threads");
    __shared__ TF as[KC][TILE + 4], bs[KC][TILE + 4];   // a: [k][row], b: [k][column]
    const int64_t base = (int64_t)blockIdx.y * 2 * m;
    if (base + m >= n) return;
    const int nt = m / TILE, i0 = blockIdx.x / nt * TILE, j0 = blockIdx.x % nt * TILE;
    TF *I = inv + base / B * ((int64_t)B * B);
    const int o = (int)(base % B);
    TF *X11 = I + (int64_t)o * B + o, *T = X11 + m, *X21 = X11 + (int64_t)m * B, *X22 = X21 + m;
    if (base + m + i0 >= n) {   // rows past the matrix (X21 there is never read; T is, by phase 1)
        if (phase == 0)
            for (int e = threadIdx.x; e < TILE * TILE; e += 256)
                T[(int64_t)(i0 + e / TILE) * B + j0 + e % TILE] = TF(0);
        return;
    }
    const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
    TF acc[Q][Q];
#pragma unroll
    for (int p = 0; p < Q; p++)
#pragma unroll
        for (int q = 0; q < Q; q++) acc[p][q] = TF(0);
    const int k0 = phase == 0 ? j0 : 0, k1 = phase == 0 ? m : i0 + TILE;
    // the next chunk's entries are loaded into registers while this one's product runs
    constexpr int E = KC * TILE / 256;
    TF pa[E], pb[E];
    auto load = [&](int kc) {
#pragma unroll
        for (int q = 0; q < E; q++) {
            const int e = threadIdx.x + 256 * q;
            const int r = e / KC, k = e % KC, kb = e / TILE, c = e % TILE;
            const int64_t row = base + m + i0 + r;
            pa[q] = phase == 0 ? (row < n ? __ldg(L + row * n + base + kc + k) : TF(0))
                               : X22[(int64_t)(i0 + r) * B + kc + k];
            pb[q] = (phase == 0 ? X11 : T)[(int64_t)(kc + kb) * B + j0 + c];
        }
    };
    load(k0);
    for (int kc = k0; kc < k1; kc += KC) {
        __syncthreads();   // the previous chunk has been read
#pragma unroll
        for (int q = 0; q < E; q++) {
            const int e = threadIdx.x + 256 * q;
            as[e % KC][e / KC] = pa[q];
            bs[e / TILE][e % TILE] = pb[q];
        }
        __syncthreads();
        if (kc + KC < k1) load(kc + KC);
#pragma unroll
        for (int k = 0; k < KC; k++) {
            TF u[Q], v[Q];
#pragma unroll
            for (int q = 0; q < Q; q++) {
                u[q] = as[k][ty * Q + q];
                v[q] = bs[k][tx * Q + q];
            }
#pragma unroll
            for (int p = 0; p < Q; p++)
#pragma unroll
                for (int q = 0; q < Q; q++) acc[p][q] = fma(u[p], v[q], acc[p][q]);
        }
    }
    TF *out = phase == 0 ? T : X21;
#pragma unroll
    for (int p = 0; p < Q; p++)
#pragma unroll
        for (int q = 0; q < Q; q++)
            out[(int64_t)(i0 + ty * Q + p) * B + j0 + tx * Q + q] = phase == 0 ? acc[p][q] : -acc[p][q];
}

// rows of M times the block x (column-major, ld n): TRI = false: t -= M x over K columns; true:
// y = M x with M lower triangular.  A warp takes R rows, its lanes the columns.
template <class TF, int NR, int R, bool TRI>
__global__ void __launch_bounds__(kTriThreads) k_tri_rows(const TF *__restrict__ M, int64_t ldm,
                                                          int64_t rows, int K,
                                                          const TF *x, int64_t n,
                                                          int nrhs, TF *out) {
    const int lane = threadIdx.x & 31;
    const int64_t r0 = ((int64_t)blockIdx.x * kTriWarps + (threadIdx.x >> 5)) * R;
    if (r0 >= rows) return;
    TF acc[R][NR];
#pragma unroll
    for (int q = 0; q < R; q++)
#pragma unroll
        for (int v = 0; v < NR; v++) acc[q][v] = TF(0);
    const TF *Mr = M + r0 * ldm;
    const int kend = TRI ? (int)min((int64_t)K, r0 + R) : K;
    chain_next();
#pragma unroll
    for (int q = 0; q < R; q++)
        if (r0 + q < rows)
            for (int k = lane * (128 / (int)sizeof(TF)); k < kend; k += 32 * (128 / (int)sizeof(TF)))
                fetch_l2(Mr + q * ldm + k);
    chain_wait();
#pragma unroll(R == 1 ? 4 : 2)
    for (int k = lane; k < kend; k += 32) {
        TF a[R];
#pragma unroll
        for (int q = 0; q < R; q++)
            a[q] = (r0 + q < rows && (!TRI || k <= r0 + q)) ? __ldg(Mr + q * ldm + k) : TF(0);
#pragma unroll
        for (int v = 0; v < NR; v++) {
            const TF xv = NR == 1 || v < nrhs ? x[(int64_t)v * n + k] : TF(0);
#pragma unroll
            for (int q = 0; q < R; q++) acc[q][v] = fma(a[q], xv, acc[q][v]);
        }
    }
    // the lanes' sums; lane (q NR + v) mod 32 writes element (q, v)
#pragma unroll
    for (int q = 0; q < R; q++)
#pragma unroll
        for (int v = 0; v < NR; v++) {
            TF s = acc[q][v];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == (q * NR + v) % 32 && r0 + q < rows && v < nrhs) {
                TF *p = out + (int64_t)v * n + r0 + q;
                *p = TRI ? s : *p - s;
            }
        }
}

// columns of M (rows x cols) times the block x: TRI = false: t -= M^T x; true: y = M^T x, M
// lower triangular.  A CTA takes 32 columns (lanes along them), its warps share the rows; x
// goes through the warp's shared memory in pieces of 32 rows, read back as broadcasts.
template <class TF, int NR> struct ColCfg {
    static constexpr int PAD = NR == 1 ? 1 : (NR + 3) / 4 * 4;
    static constexpr size_t kSmem = sizeof(TF) * kColWarps * 32 * PAD;
};
template <class TF, int NR, bool TRI>
__global__ void __launch_bounds__(kColThreads) k_tri_cols(const TF *__restrict__ M, int64_t ldm,
                                                          int rows, int64_t cols,
                                                          const TF *x, int64_t n,
                                                          int nrhs, TF *out) {
    constexpr int PAD = ColCfg<TF, NR>::PAD, U = 16;   // rows in flight
    extern __shared__ __align__(16) unsigned char sm_cols[];   // x of the warps' rows, then sums
    TF(*xs)[PAD] = reinterpret_cast<TF(*)[PAD]>(sm_cols) + (threadIdx.x >> 5) * 32;
    TF(*red)[NR][32] = reinterpret_cast<TF(*)[NR][32]>(sm_cols);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t c = (int64_t)blockIdx.x * 32 + lane;
    const bool in = c < cols;
    TF acc[NR];
#pragma unroll
    for (int v = 0; v < NR; v++) acc[v] = TF(0);
    // rows from the CTA's first column on when triangular
    const int first = TRI ? blockIdx.x : 0, pieces = (rows + 31) / 32;
    chain_next();
    for (int i = 32 * first + threadIdx.x; i < rows; i += kColThreads)
        fetch_l2(M + (int64_t)i * ldm + (int64_t)blockIdx.x * 32);
    chain_wait();
    for (int pc = first + warp; pc < pieces; pc += kColWarps) {
        const int i0 = 32 * pc;
        const TF *Mc = M + (int64_t)i0 * ldm + c;
        auto load = [&](int i, TF a[U]) {
#pragma unroll
            for (int q = 0; q < U; q++)
                a[q] = in && i0 + i + q < rows && (!TRI || i0 + i + q >= c)
                           ? __ldg(Mc + (int64_t)(i + q) * ldm)
                           : TF(0);
        };
        TF a[U];
        load(0, a);
#pragma unroll
        for (int v = 0; v < NR; v++)
            xs[lane][v] = i0 + lane < rows && v < nrhs ? x[(int64_t)v * n + i0 + lane] : TF(0);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 32; i += U) {
            TF b[U];
            if (i + U < 32) load(i + U, b);
#pragma unroll
            for (int q = 0; q < U; q++)
#pragma unroll
                for (int v = 0; v < NR; v++) acc[v] = fma(a[q], xs[i + q][v], acc[v]);
#pragma unroll
            for (int q = 0; q < U; q++) a[q] = b[q];
        }
        __syncwarp();
    }
    __syncthreads();
#pragma unroll
    for (int v = 0; v < NR; v++) red[warp][v][lane] = acc[v];
    __syncthreads();
    for (int e = threadIdx.x; e < 32 * NR; e += kColThreads) {
        const int v = e >> 5, l = e & 31;
        const int64_t cc = (int64_t)blockIdx.x * 32 + l;
        if (v >= nrhs || cc >= cols) continue;
        TF s = red[0][v][l];
#pragma unroll
        for (int w = 1; w < kColWarps; w++) s += red[w][v][l];
        TF *p = out + (int64_t)v * n + cc;
        *p = TRI ? s : *p - s;
    }
}

// FP32 updates with several columns: t -= M x (TRANS: M^T x) for 32 outputs per CTA over all K.
// Chunks of 128 of K go through shared memory, the next one's loads (16 per thread) in flight
// meanwhile; thread = (four outputs, a quarter of the columns, an eighth of the chunk), the
// eighths added at the end.  k_tri_rows and k_tri_cols re-read x for every one or four rows: 17
// columns at n = 12,167 took them 114 and 38 us a launch, 23 and 31 us here.
constexpr int kTileOut = 32, kTileK = 128;
constexpr size_t kTileRed = 24 * 1024;   // room of the final sums (24 columns)
template <int NR, bool TRANS>
__global__ void __launch_bounds__(256) k_tri_tile(const float *__restrict__ M, int64_t ldm,
                                                  int64_t outs, int K, const float *x,
                                                  int64_t n, int nrhs, float *out) {
    static_assert(NR % 4 == 0, "four column groups");
    constexpr int NV = NR / 4, LM = TRANS ? kTileOut + 4 : kTileK + 4, LX = kTileK + 4;
    constexpr int EM = kTileOut * kTileK / 256, EX = (NR * kTileK + 255) / 256;
    constexpr int W = TRANS ? kTileOut : kTileK;   // width of the chunk's rows in M
    __shared__ __align__(16) float ms[kTileRed / sizeof(float)];   // the chunk of M, then the sums
    __shared__ __align__(16) float xs[NR * LX];
    static_assert(sizeof(float) * (TRANS ? kTileK : kTileOut) * LM <= kTileRed, "chunk room");
    const int tid = threadIdx.x, og = tid & 7, vg = (tid >> 3) & 3, kg = tid >> 5;
    const int64_t o0 = (int64_t)blockIdx.x * kTileOut;
    float acc[4][NV], pm[EM], px[EX];
#pragma unroll
    for (int q = 0; q < 4; q++)
#pragma unroll
        for (int v = 0; v < NV; v++) acc[q][v] = 0.f;
    auto load_m = [&](int kc) {
#pragma unroll
        for (int q = 0; q < EM; q++) {
            const int e = tid + 256 * q, r = e / W, c = e % W;
            const int64_t o = o0 + (TRANS ? c : r);
            const int k = kc + (TRANS ? r : c);
            pm[q] = o < outs && k < K ? __ldg(M + (TRANS ? k * ldm + o : o * ldm + k)) : 0.f;
        }
    };
    auto load_x = [&](int kc) {
#pragma unroll
        for (int q = 0; q < EX; q++) {
            const int e = tid + 256 * q, v = e / kTileK, k = kc + e % kTileK;
            px[q] = v < nrhs && k < K ? x[(int64_t)v * n + k] : 0.f;
        }
    };
    chain_next();
    load_m(0);
    // the rest of the CTA's part of M, a line of 32 entries per fetch
    for (int e = tid + (TRANS ? kTileK : kTileOut * (kTileK / 32)); e < K * kTileOut / 32; e += 256) {
        const int64_t o = o0 + (TRANS ? 0 : e % kTileOut);
        const int k = TRANS ? e : e / kTileOut * 32;
        if (o < outs && k < K) fetch_l2(M + (TRANS ? k * ldm + o : o * ldm + k));
    }
    chain_wait();
    load_x(0);
    for (int kc = 0; kc < K; kc += kTileK) {
        __syncthreads();   // the previous chunk has been read
#pragma unroll
        for (int q = 0; q < EM; q++) {
            const int e = tid + 256 * q;
            ms[e / W * LM + e % W] = pm[q];
        }
#pragma unroll
        for (int q = 0; q < EX; q++) {
            const int e = tid + 256 * q;
            if (e < NR * kTileK) xs[e / kTileK * LX + e % kTileK] = px[q];
        }
        __syncthreads();
        if (kc + kTileK < K) {
            load_m(kc + kTileK);
            load_x(kc + kTileK);
        }
#pragma unroll
        for (int kk = 0; kk < 16; kk += 4) {
            const int k = kg * 16 + kk;
            float4 m[4];   // TRANS: [k + q][the four outputs]; else [output og + 8 q][k .. k + 3]
#pragma unroll
            for (int q = 0; q < 4; q++)
                m[q] = *reinterpret_cast<const float4 *>(
                    TRANS ? &ms[(k + q) * LM + 4 * og] : &ms[(og + 8 * q) * LM + k]);
#pragma unroll
            for (int v = 0; v < NV; v++) {
                const float4 xv = *reinterpret_cast<const float4 *>(&xs[(vg * NV + v) * LX + k]);
                if constexpr (TRANS) {
                    acc[0][v] = fmaf(m[0].x, xv.x, fmaf(m[1].x, xv.y, fmaf(m[2].x, xv.z, fmaf(m[3].x, xv.w, acc[0][v]))));
                    acc[1][v] = fmaf(m[0].y, xv.x, fmaf(m[1].y, xv.y, fmaf(m[2].y, xv.z, fmaf(m[3].y, xv.w, acc[1][v]))));
                    acc[2][v] = fmaf(m[0].z, xv.x, fmaf(m[1].z, xv.y, fmaf(m[2].z, xv.z, fmaf(m[3].z, xv.w, acc[2][v]))));
                    acc[3][v] = fmaf(m[0].w, xv.x, fmaf(m[1].w, xv.y, fmaf(m[2].w, xv.z, fmaf(m[3].w, xv.w, acc[3][v]))));
                } else {
#pragma unroll
                    for (int q = 0; q < 4; q++)
                        acc[q][v] = fmaf(m[q].x, xv.x, fmaf(m[q].y, xv.y, fmaf(m[q].z, xv.z, fmaf(m[q].w, xv.w, acc[q][v]))));
                }
            }
        }
    }
    __syncthreads();
    // the eighths' sums [8][NR][32]
    float *red = ms;
    static_assert(sizeof(float) * 8 * NR * kTileOut <= kTileRed, "reduction room");
#pragma unroll
    for (int q = 0; q < 4; q++)
#pragma unroll
        for (int v = 0; v < NV; v++)
            red[(kg * NR + vg * NV + v) * kTileOut + (TRANS ? 4 * og + q : og + 8 * q)] = acc[q][v];
    __syncthreads();
    for (int e = tid; e < NR * kTileOut; e += 256) {
        const int v = e / kTileOut;
        const int64_t o = o0 + e % kTileOut;
        if (v >= nrhs || o >= outs) continue;
        float t = red[e];
#pragma unroll
        for (int w = 1; w < 8; w++) t += red[w * NR * kTileOut + e];
        out[(int64_t)v * n + o] -= t;
    }
}

template <class TF> int tri_width(int64_t n) {
    int64_t B = sizeof(TF) == 4 ? (n <= 4096 ? 512 : 1024) : (n <= 512 ? 512 : 256);
    while (B > 64 && B / 2 >= n) B /= 2;
    return (int)B;
}

// rows of a launch: one per warp until that fills the chip (about eight warps per SM; a triangular
// block's 1,024 rows never do), then four (NR sums each), which share the reads of x
template <class TF, int NR, bool TRI>
int launch_rows(const TF *M, int64_t ldm, int64_t rows, int K, const TF *x, int64_t n, int nrhs,
                TF *out, cudaStream_t s, bool first = false) {
    if constexpr (!TRI)
        if (rows > 4 * 1216)
            return launch_chained(first, k_tri_rows<TF, NR, 4, TRI>,
                                  (rows + 4 * kTriWarps - 1) / (4 * kTriWarps), kTriThreads, 0, s, M,
                                  ldm, rows, K, x, n, nrhs, out);
    return launch_chained(first, k_tri_rows<TF, NR, 1, TRI>, (rows + kTriWarps - 1) / kTriWarps,
                          kTriThreads, 0, s, M, ldm, rows, K, x, n, nrhs, out);
}

template <class TF, int NR, bool TRI>
int launch_cols(const TF *M, int64_t ldm, int rows, int64_t cols, const TF *x, int64_t n, int nrhs,
                TF *out, cudaStream_t s) {
    constexpr size_t sh = ColCfg<TF, NR>::kSmem;
    if (sh > 48 * 1024) FEM3_CUDA(device_smem((const void *)k_tri_cols<TF, NR, TRI>, sh));
    return launch_chained(false, k_tri_cols<TF, NR, TRI>, (cols + 31) / 32, kColThreads, sh, s, M, ldm,
                          rows, cols, x, n, nrhs, out);
}

// t -= M x or M^T x
template <class TF, int NR, bool TRANS>
int launch_update(const TF *M, int64_t ldm, int64_t outs, int K, const TF *x, int64_t n, int nrhs,
                  TF *out, cudaStream_t s) {
    if constexpr (sizeof(TF) == 4 && NR > 1) {
        constexpr int NP = (NR + 3) / 4 * 4;
        return launch_chained(false, k_tri_tile<NP, TRANS>, (outs + kTileOut - 1) / kTileOut, 256, 0, s,
                              M, ldm, outs, K, x, n, nrhs, out);
    } else if constexpr (TRANS) {
        return launch_cols<TF, NR, false>(M, ldm, K, outs, x, n, nrhs, out, s);
    } else {
        return launch_rows<TF, NR, false>(M, ldm, outs, K, x, n, nrhs, out, s);
    }
}

template <class TF, int NR>
int solve_blocks(Mesh *m, const TF *L, int64_t n, TF *Y, int nrhs) {
    cudaStream_t s = m->stream;
    const int B = tri_width<TF>(n);
    const int nb = (int)((n + B - 1) / B);
    const TF *inv = reinterpret_cast<const TF *>(m->tri_inv);
    TF *W = reinterpret_cast<TF *>(m->solve_ws);
    kc_begin(m, KC_CHAIN);
    for (int j = 0; j < nb; j++) {   // Y -> W
        const int64_t c0 = (int64_t)j * B, w = std::min<int64_t>(B, n - c0), rest = n - c0 - w;
        FEM3_TRY((launch_rows<TF, NR, true>(inv + (int64_t)j * B * B, B, w, (int)w, Y + c0, n, nrhs,
                                            W + c0, s, j == 0)));
        if (rest > 0)
            FEM3_TRY((launch_update<TF, NR, false>(L + (c0 + w) * n + c0, n, rest, (int)w, W + c0, n,
                                                   nrhs, Y + c0 + w, s)));
    }
    for (int j = nb - 1; j >= 0; j--) {   // W -> Y
        const int64_t c0 = (int64_t)j * B, w = std::min<int64_t>(B, n - c0);
        FEM3_TRY((launch_cols<TF, NR, true>(inv + (int64_t)j * B * B, B, (int)w, w, W + c0, n, nrhs,
                                            Y + c0, s)));
        if (c0 > 0)
            FEM3_TRY((launch_update<TF, NR, true>(L + c0 * n, n, c0, (int)w, Y + c0, n, nrhs, W, s)));
    }
    kc_end(m, KC_CHAIN);
    m->launches += 4 * nb - 2;
    FEM3_CUDA(cudaGetLastError());
    return FEM3_OK;
}

}  // namespace

template <class TF> int tri_prepare(Mesh *m, const TF *L, int64_t n) {
    if (n <= 0) return FEM3_OK;
    cudaStream_t s = m->stream;
    const int B = tri_width<TF>(n), n64 = (int)((n + 63) / 64);
    if (!m->tri_inv) {   // room for either type: nothing is allocated when the precision changes
        const auto bytes = [n](size_t size, int64_t b) { return size * (size_t)((n + b - 1) / b * b * b); };
        FEM3_TRY(dev_alloc(m, &m->tri_inv, std::max(bytes(sizeof(float), tri_width<float>(n)),
                                                    bytes(sizeof(double), tri_width<double>(n)))));
    }
    if (!m->solve_ws) FEM3_TRY(dev_alloc(m, &m->solve_ws, sizeof(double) * kTriRhs * (size_t)n));
    TF *inv = reinterpret_cast<TF *>(m->tri_inv);
    k_tri_seed<TF><<<n64, 256, 0, s>>>(reinterpret_cast<const TF *>(m->dinv), B, inv);
    note_launch(m);
    for (int w = 64; w < B && w < n; w *= 2) {
        constexpr int TILE = sizeof(TF) == 4 ? 64 : 16, Q = TILE / 16;
        const dim3 grid((unsigned)((w / TILE) * (w / TILE)), (unsigned)((n + 2 * w - 1) / (2 * w)));
        for (int phase = 0; phase < 2; phase++) {
            k_tri_double<TF, TILE, Q><<<grid, 256, 0, s>>>(L, n, B, w, phase, inv);
            note_launch(m);
        }
    }
    FEM3_CUDA(cudaGetLastError());
    return FEM3_OK;
}

template <class TF> int tri_solve(Mesh *m, const TF *L, int64_t n, TF *Y, int nrhs) {
    if (n <= 0) return FEM3_OK;
    for (int c0 = 0; c0 < nrhs; c0 += kTriRhs) {
        const int cnt = std::min(kTriRhs, nrhs - c0);
        TF *y = Y + (int64_t)c0 * n;
        if (cnt == 1) FEM3_TRY((solve_blocks<TF, 1>(m, L, n, y, cnt)));
        else if (cnt <= 4) FEM3_TRY((solve_blocks<TF, 4>(m, L, n, y, cnt)));
        else if (cnt <= 8) FEM3_TRY((solve_blocks<TF, 8>(m, L, n, y, cnt)));
        else if (cnt <= 17) FEM3_TRY((solve_blocks<TF, 17>(m, L, n, y, cnt)));
        else FEM3_TRY((solve_blocks<TF, 24>(m, L, n, y, cnt)));
    }
    return FEM3_OK;
}

template int tri_prepare<float>(Mesh *, const float *, int64_t);
template int tri_prepare<double>(Mesh *, const double *, int64_t);
template int tri_solve<float>(Mesh *, const float *, int64_t, float *, int);
template int tri_solve<double>(Mesh *, const double *, int64_t, double *, int);

}  // namespace fem3
