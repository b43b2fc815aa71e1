// Device code of the dense Cholesky factorisation shared by the tile-task factorisation
// (solve.cu) and the blocked factorisation with tensor-core trailing updates (chol_tc.cu):
// release/acquire flag helpers, pivots, and the 64 x 64 FP32 diagonal-block factor-and-invert
// routine.  Included inside `namespace fem3 { namespace {`
// by each translation unit (every unit gets its own internal copy).

constexpr int NB = 64;   // block width of the FP32 factorisations and of the triangular solves

// ---------------------------------------------------------------------------------
// Cholesky
// ---------------------------------------------------------------------------------
constexpr int kSpinLimit = 1 << 22;   // x >= 64 ns sleep: > 0.25 s before giving up

__device__ __forceinline__ int ld_acquire_gpu(const int *p) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_gpu(int *p, int v) {
    asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// FP32: hardware estimate plus one Newton step y <- y + y (1 - x y^2) / 2, so that the
// factor is as accurate as one built from a correctly rounded square root (refinement
// then converges in as many sweeps).
__device__ __forceinline__ float rsqrt_newton(float x) {
    const float y = rsqrtf(x);
    const float r = fmaf(-x * y, y, 1.0f);
    return fmaf(0.5f * y, r, y);
}

// a positive pivot (false for NaN); FP64 by its bits, since a comparison takes the FP64 pipe
__device__ __forceinline__ bool pivot_pos(float d) { return d > 0.f; }
__device__ __forceinline__ bool pivot_pos(double d) {
    const long long b = __double_as_longlong(d);
    return b > 0 && b <= 0x7FF0000000000000LL;
}

// 1 / d of a positive pivot, the only function on the serial path of the diagonal factor.
// FP64: the FP32 reciprocal estimate of the leading 24 bits of d (together below 2^-21 off)
// as the start and one cubic Newton step y <- y (1 + e + e^2), e = 1 - d y (error e^3 <
// 2^-63): three dependent FP64 operations where the division takes several more.
template <class TF> __device__ __forceinline__ TF recip_t(TF d);
template <> __device__ __forceinline__ float recip_t<float>(float d) { return __frcp_rn(d); }
template <> __device__ __forceinline__ double recip_t<double>(double d) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(d);
    const int e = (int)(b >> 52);   // d > 0: the sign bit is 0
    if (e < 8 || e > 2038) return 1.0 / d;
    const float m = __uint_as_float(0x3F800000u | (uint32_t)((b >> 29) & 0x7FFFFFu));
    float ym;   // in [0.5, 1]
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(ym) : "f"(m));
    const uint32_t y32 = __float_as_uint(ym);
    const double y = __longlong_as_double(
        (long long)(((unsigned long long)((int)(y32 >> 23) + 896 + 1023 - e) << 52) |
                    ((unsigned long long)(y32 & 0x7FFFFFu) << 29)));
    const double r = fma(-d, y, 1.0);
    return fma(y, fma(r, r, r), y);
}

__device__ __forceinline__ void lds4(const float *p, float v[4]) {   // 16-byte aligned
    const float4 q = *reinterpret_cast<const float4 *>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
__device__ __forceinline__ void lds2(const float *p, float v[2]) {
    const float2 q = *reinterpret_cast<const float2 *>(p);
    v[0] = q.x; v[1] = q.y;
}

constexpr int PB = 16;   // panel width inside the diagonal block

// named barriers of the diagonal factor (0 is __syncthreads)
constexpr int kBarPanelReady = 1;   // warp 0 -> update warps: block p factored and inverted
constexpr int kBarNextReady = 2;    // update warps -> warp 0: block p + 1 fully updated
constexpr int kBarUpdate = 3;       // among the 15 update warps
__device__ __forceinline__ void bar_sync_n(int id, int count) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive_n(int id, int count) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(count) : "memory");
}

// warp 0: 16 x 16 Cholesky of block p of a_s and its inverse in one pass.  Lanes 0..15 hold
// row r of the block (lower part), lanes 16..31 column r of the identity; step j broadcasts
// the pivot column (a_kj, k >= j, from lanes k) and every lane applies the same update,
// x_k -= (x_j / a_jj) a_kj (k > j): on the rows this is the right-looking factorisation, on
// the identity's columns forward substitution with the new column of L_pp, so the inverse
// needs no pass of its own.  The square roots stay off this serial path: column j (row j of
// the inverse) is scaled by 1 / sqrt(a_jj) after the last step, all sixteen roots at once on
// the lanes.  Entries above the diagonal of the row lanes are never read.  Writes L_pp into
// a_s, L_pp^{-1} into x_s and lt[k][c] = L_pp^{-1}[c][k].
__device__ __forceinline__ void chol_inv16(float (*a_s)[NB + 1], float (*x_s)[NB + 1], float (*lt)[PB + 4],
                                           int P, int nb, int64_t k0, int32_t *err) {
    const int lane = threadIdx.x & 31;
    const int r = lane & (PB - 1);
    const bool inv = lane >= PB;
    float x[PB];
#pragma unroll
    for (int c = 0; c < PB; c++)
        x[c] = inv ? (c == r ? 1.f : 0.f) : (c <= r ? a_s[P + r][P + c] : 0.f);
    int bad = -1;
    float dr = 1.f;   // pivot r (of lane r)
#pragma unroll
    for (int j = 0; j < PB; j++) {
        float col[PB];
#pragma unroll
        for (int k = j; k < PB; k++) col[k] = __shfl_sync(0xffffffffu, x[j], k);
        const float d = col[j];
        const bool pos = pivot_pos(d);
        if (!pos && bad < 0) bad = j;
        const float f = x[j] * (pos ? recip_t(d) : 1.f);
        if (r == j) dr = d;
#pragma unroll
        for (int k = j + 1; k < PB; k++) x[k] -= f * col[k];
    }
    const float rs = pivot_pos(dr) ? rsqrt_newton(dr) : 1.f;
#pragma unroll
    for (int j = 0; j < PB; j++) x[j] *= __shfl_sync(0xffffffffu, rs, j);
    if (bad >= 0 && lane == 0 && P + bad < nb)
        atomicCAS(&err[ERR_NOT_SPD], 0, (int32_t)(k0 + P + bad + 1));
    if (!inv) {
#pragma unroll
        for (int c = 0; c < PB; c++)
            if (c <= r) a_s[P + r][P + c] = x[c];
    } else {
#pragma unroll
        for (int i = 0; i < PB; i++) {
            x_s[P + i][P + r] = i >= r ? x[i] : 0.f;
            lt[r][i] = x[i];
        }
    }
}

// Diagonal block: factor A_kk = L_kk L_kk^T and form L_kk^{-1} (64 x 64; 512 threads), blocked by
// 16 with look-ahead.  Warp 0 factors and inverts the 16 x 16 diagonal block p; 12 other
// warps then (a) solve the 16 rows of block p + 1 in panel p (L_{p+1,p} = A L_pp^{-T})
// and update diagonal block p + 1, which releases warp 0 for block p + 1 at once, and
// (b) meanwhile solve the rest of panel p, finish the inverse's block row p,
// (L^{-1})_pJ = -L_pp^{-1} T_pJ, apply the rest of the trailing update (2 x 2 blocks per
// thread) and form T_{p+1,J} = sum_K L_{p+1,K} (L^{-1})_KJ, which needs nothing of block
// p + 1 and so overlaps its factorisation.  The blocks of L^{-1} above the diagonal are
// zeroed first, while block 0 is factored.  a_s holds the block (rows and columns >= nb
// padded with the identity) and receives L (lower triangle); x_s receives L^{-1} in full
// (zero above the diagonal); the caller stores them.  A non-positive pivot records 1 + its
// global column (k0 + local).  Needs exactly 512 threads, all of the CTA; ends with a
// barrier.
__device__ void potrf_inv_smem(float (*a_s)[NB + 1], float (*x_s)[NB + 1], int nb, int64_t k0,
                               int32_t *err) {
    // warps 4, 8 and 12 share warp 0's SM sub-partition and sit out: the 12 other warps
    // do the update work, so warp 0's serial factor competes with no issuing neighbour
    constexpr int NT = 416, NU = 384, NP = NB / PB;
    __shared__ __align__(16) float lt[2][PB][PB + 4];     // lt[p & 1][k][c] = L_pp^{-1}[c][k]
    __shared__ __align__(16) float pant[PB][NB + 4];      // pant[k][r] = L[r][P + k], r >= P + 16
    __shared__ __align__(16) float tq[PB][NB - PB + 4];   // T_pJ, columns c < P
    const int tid = threadIdx.x;
    if (tid < 32) {
        for (int p = 0; p < NP; p++) {
            if (p > 0) bar_sync_n(kBarNextReady, NT);
            chol_inv16(a_s, x_s, lt[p & 1], p * PB, nb, k0, err);
            __syncwarp();
            bar_arrive_n(kBarPanelReady, NT);
        }
    } else if (((tid >> 5) & 3) != 0) {
        const int ut = ((tid >> 5) - 1 - (tid >> 7)) * 32 + (tid & 31);   // 0 .. NU - 1
        for (int e = ut; e < NB * NB; e += NU) {
            const int i = e / NB, c = e & (NB - 1);
            if (c >= ((i >> 4) + 1) * PB) x_s[i][c] = 0.f;
        }
        for (int p = 0; p < NP; p++) {
            const int P = p * PB;
            bar_sync_n(kBarPanelReady, NT);
            const float(*L16)[PB + 4] = lt[p & 1];
            // (a) block p + 1: its rows of panel p, then its diagonal update
            const int R0 = P + PB;
            if (p + 1 < NP) {
                float xv = 0.f;
                const int xr = R0 + (ut >> 4), xc = ut & 15;
                if (ut < PB * PB) {
#pragma unroll
                    for (int k = 0; k < PB; k++) xv += a_s[xr][P + k] * L16[k][xc];
                }
                bar_sync_n(kBarUpdate, NU);
                if (ut < PB * PB) {
                    a_s[xr][P + xc] = xv;
                    pant[xc][xr] = xv;
                }
                bar_sync_n(kBarUpdate, NU);
                if (ut < PB * PB && xc + R0 <= xr) {
                    float acc = 0.f;
#pragma unroll
                    for (int k = 0; k < PB; k++) acc += pant[k][xr] * pant[k][R0 + xc];
                    a_s[xr][R0 + xc] -= acc;
                }
                bar_arrive_n(kBarNextReady, NT);
            }
            // (b1) rows below block p + 1 (four columns per thread); the inverse's block
            // row p from T_pJ (formed in the previous panel)
            const int R1 = R0 + PB, m2 = NB - R1;
            const bool panel = m2 > 0 && ut < 4 * m2;
            const int pr = R1 + (ut >> 2), pc = (ut & 3) * 4;
            float pv[4] = {0.f, 0.f, 0.f, 0.f};
            if (panel) {
#pragma unroll
                for (int k = 0; k < PB; k++) {
                    const float av = a_s[pr][P + k];
                    float lv[4];
                    lds4(&L16[k][pc], lv);
#pragma unroll
                    for (int q = 0; q < 4; q++) pv[q] += av * lv[q];
                }
            }
            float iv[2] = {0.f, 0.f};
            if (p > 0) {
#pragma unroll
                for (int s2 = 0; s2 < 2; s2++) {
                    const int e = ut + NU * s2;
                    if (e < PB * P) {
                        const int i = e / P, c = e - i * P;
                        float acc = 0.f;
#pragma unroll
                        for (int k = 0; k < PB; k++)
                            if (k <= i) acc += x_s[P + i][P + k] * tq[k][c];
                        iv[s2] = -acc;
                    }
                }
            }
            bar_sync_n(kBarUpdate, NU);
            // (b2) store the rows and the inverse's block row
            if (panel) {
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    a_s[pr][P + pc + q] = pv[q];
                    pant[pc + q][pr] = pv[q];
                }
            }
            if (p > 0) {
#pragma unroll
                for (int s2 = 0; s2 < 2; s2++) {
                    const int e = ut + NU * s2;
                    if (e < PB * P) {
                        const int i = e / P, c = e - i * P;
                        x_s[P + i][c] = iv[s2];
                    }
                }
            }
            if (p + 1 == NP) break;
            bar_sync_n(kBarUpdate, NU);
            // (b3) T_{p+1,J}[i][c] = sum_{k = c}^{R0 - 1} L[R0 + i][k] (L^{-1})[k][c], c < R0
            for (int e = ut; e < PB * R0; e += NU) {
                const int i = e / R0, c = e - i * R0;
                float acc = 0.f;
                for (int kb = c & ~(PB - 1); kb < R0; kb += PB) {
#pragma unroll
                    for (int k = 0; k < PB; k++)
                        if (kb + k >= c) acc += a_s[R0 + i][kb + k] * x_s[kb + k][c];
                }
                tq[i][c] = acc;
            }
            // trailing update of blocks (i, k), i >= k >= p + 1, except block (p + 1, p + 1),
            // in 2 x 2 blocks (rows i0, i0 + 1 >= R1; columns j0, j0 + 1 >= R0)
            const int mr = (NB - R1) / 2, mc = (NB - R0) / 2;
            for (int e = ut; e < mr * mc; e += NU) {
                const int i0 = R1 + 2 * (e / mc), j0 = R0 + 2 * (e % mc);
                if (j0 > i0) continue;
                float c00 = 0.f, c01 = 0.f, c10 = 0.f, c11 = 0.f;
#pragma unroll
                for (int k = 0; k < PB; k++) {
                    float pi[2], pj[2];
                    lds2(&pant[k][i0], pi);
                    lds2(&pant[k][j0], pj);
                    c00 += pi[0] * pj[0];
                    c01 += pi[0] * pj[1];
                    c10 += pi[1] * pj[0];
                    c11 += pi[1] * pj[1];
                }
                a_s[i0][j0] -= c00;
                if (j0 + 1 <= i0) a_s[i0][j0 + 1] -= c01;
                a_s[i0 + 1][j0] -= c10;
                a_s[i0 + 1][j0 + 1] -= c11;
            }
        }
    }
    __syncthreads();
}
