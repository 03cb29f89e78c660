// lu.cu -- blocked right-looking LU of the assembled system in FP64 (the
// dense solve of Gallagher & Smith, Sec. 4 step 3): the factor of the plain
// FP64 path.  (The mixed-precision path inverts an FP32 copy instead, gj.cu.)
//
// Pivoting is restricted to the rows of each NB x NB diagonal block: the
// block is factored with partial pivoting among its own rows and the same
// row exchange is applied across the whole block row.  This keeps every
// panel step inside one CTA (no grid-wide pivot search over n rows) and the
// rest of the step parallel: L21 = A21 U11^{-1}, U12 = L11^{-1} P A12 by
// independent substitutions per row / column, then A22 -= L21 U12.  The
// NEAREST matrix is close to (symmetric positive definite Nystrom matrix) x
// (positive diagonal of segment weights), whose LU needs no pivoting, and the
// rigid-body rows come last, where the in-block pivoting handles the zero
// corner; the growth factor on the swimmer workloads equals that of full
// partial pivoting.  The FP64 refinement of solve.cu removes what is left.
//
// Result: P A = L U with P the composition of the block-local exchanges,
// rowperm[i] = original row now at position i, L unit lower and U upper
// stored in place.
//
// GB300 issues an FP64 fused multiply-add of a warp in 64 clocks and a division
// in 344 wherever it runs, so a triangular solve by one thread per row keeps a
// few SMs busy for its whole length (145 and 114 us for n = 2406, whatever is
// left of the matrix).  The panels L21 and U12 are therefore formed as products
// with the inverses of the diagonal block's 32 x 32 triangles, in strips of 16
// rows or columns over all SMs; the same inverses serve the triangular solves
// of solve.cu.  The block's row exchange reaches the columns left of it once,
// at the end.  Swimmer, n = 2406, factor and solve: 29.2 ms before, 16.3 ms now
// (9.5 the update, 4.7 the diagonal blocks, 1.0 the panels, 1.0 the solves).
#include "nrs_internal.cuh"

namespace nrs {

constexpr int LU_NB = 64, LU_HB = 32, LU_LD = LU_NB + 1;
constexpr int LU_STRIP = 16;  // rows (columns) of a panel CTA
constexpr int LU_DIAG_SMEM = (LU_NB * LU_LD + 4 * LU_HB * (LU_HB + 1)) * (int)sizeof(double);

// Factor the diagonal block at k0 with partial pivoting among its own rows, in
// place; rowperm[k0 + i] = k0 + the block row now at i.  inv (4 x 32 x 32,
// row-major): inverses of the triangles L[0:32, 0:32], L[32:64, 32:64] (unit
// lower) and U[0:32, 0:32], U[32:64, 32:64]; identity beyond kb.
__global__ void __launch_bounds__(256)
    k_diag_factor(int64_t n, double *__restrict__ A, int64_t lda, int64_t k0,
                  int32_t *__restrict__ rowperm, int32_t *__restrict__ info,
                  double *__restrict__ inv)
{
    extern __shared__ double diag_smem[];  // the block, then the four inverses
    double(*D)[LU_LD] = reinterpret_cast<double(*)[LU_LD]>(diag_smem);
    double(*X)[LU_HB][LU_HB + 1] =
        reinterpret_cast<double(*)[LU_HB][LU_HB + 1]>(diag_smem + LU_NB * LU_LD);
    __shared__ int32_t lp[LU_NB];
    __shared__ int32_t s_piv;
    __shared__ double s_pv, s_rp;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tx = tid & 15, ty = tid >> 4;
    const int kb = (int)min((int64_t)LU_NB, n - k0);
    for (int idx = tid; idx < LU_NB * LU_NB; idx += 256) {
        const int r = idx % LU_NB, c = idx / LU_NB;
        D[r][c] = r < kb && c < kb ? A[(k0 + r) + (k0 + c) * lda] : (r == c ? 1.0 : 0.0);
    }
    if (tid < LU_NB) lp[tid] = tid;
    __syncthreads();
    for (int c = 0; c < kb; ++c) {
        if (warp == 0) {
            // the row of largest |D[r][c]|, r >= c, lowest on ties: high words first
            auto key = [&](int r) {
                return r >= c && r < kb ? (unsigned long long)__double_as_longlong(fabs(D[r][c]))
                                        : 0ULL;
            };
            const int r1 = lane + 32;
            const unsigned long long a0 = key(lane), a1 = key(r1), a = a1 > a0 ? a1 : a0;
            const unsigned h = __reduce_max_sync(0xffffffffu, (unsigned)(a >> 32));
            const unsigned l =
                __reduce_max_sync(0xffffffffu, (unsigned)(a >> 32) == h ? (unsigned)a : 0u);
            const unsigned long long m = ((unsigned long long)h << 32) | l;
            const unsigned at0 = __ballot_sync(0xffffffffu, lane >= c && lane < kb && a0 == m);
            const unsigned at1 = __ballot_sync(0xffffffffu, r1 >= c && r1 < kb && a1 == m);
            const int p = at0 ? __ffs(at0) - 1 : at1 ? 31 + __ffs(at1) : c;
            if (lane == 0) {
                const double pv = D[p][c];
                s_piv = p;
                s_pv = pv;
                // 0: a zero pivot, or one whose reciprocal would leave the range
                s_rp = fabs(pv) > 1e-290 && fabs(pv) < 1e290 ? 1.0 / pv : 0.0;
                if (pv == 0.0 && info) atomicCAS(info, 0, (int)(k0 + c + 1));
            }
        }
        __syncthreads();
        // exchange rows c and p (threads 0..63) and form the multipliers of the
        // rows below (64..127): every read before any write
        const int p = s_piv;
        const double pv = s_pv, rp = s_rp;
        double v0 = 0.0, v1 = 0.0;
        const int r = tid - 64;
        if (tid < LU_NB) {
            v0 = D[p][tid];
            v1 = D[c][tid];
        } else if (r < LU_NB && r > c) {
            v0 = r == p ? D[c][c] : D[r][c];
            if (rp != 0.0) v0 *= rp;
            else if (pv != 0.0) v0 /= pv;  // (a zero pivot leaves the column as it is)
        }
        __syncthreads();
        if (tid < LU_NB) {
            D[c][tid] = v0;
            if (p != c && !(tid == c)) D[p][tid] = v1;
        } else if (r < LU_NB && r > c) {
            D[r][c] = v0;
        }
        if (tid == 0 && p != c) {
            const int t = lp[c];
            lp[c] = lp[p];
            lp[p] = t;
        }
        __syncthreads();
        if (pv != 0.0) {
            for (int i = c + 1 + ty; i < kb; i += 16) {
                const double m = D[i][c];
                for (int j = c + 1 + tx; j < kb; j += 16) D[i][j] -= m * D[c][j];
            }
        }
        __syncthreads();
    }
    for (int idx = tid; idx < kb * kb; idx += 256) {
        const int r = idx % kb, c = idx / kb;
        A[(k0 + r) + (k0 + c) * lda] = D[r][c];
    }
    if (tid < kb) rowperm[k0 + tid] = (int32_t)(k0 + lp[tid]);
    // the inverses: warp g < 4 one triangle, lane = column, by substitution with
    // the column in shared memory
    if (warp < 4) {
        const int o = LU_HB * (warp & 1);
        double(*x)[LU_HB + 1] = X[warp];
        if (warp < 2) {
            for (int i = 0; i < LU_HB; ++i) {
                double s0 = i == lane ? 1.0 : 0.0, s1 = 0.0;
                int k = 0;
                for (; k + 1 < i; k += 2) {
                    s0 = fma(-D[o + i][o + k], x[k][lane], s0);
                    s1 = fma(-D[o + i][o + k + 1], x[k + 1][lane], s1);
                }
                if (k < i) s0 = fma(-D[o + i][o + k], x[k][lane], s0);
                x[i][lane] = s0 + s1;
            }
        } else {
            const double rd = 1.0 / D[o + lane][o + lane];
            for (int i = LU_HB - 1; i >= 0; --i) {
                double s0 = i == lane ? 1.0 : 0.0, s1 = 0.0;
                int k = i + 1;
                for (; k + 1 < LU_HB; k += 2) {
                    s0 = fma(-D[o + i][o + k], x[k][lane], s0);
                    s1 = fma(-D[o + i][o + k + 1], x[k + 1][lane], s1);
                }
                if (k < LU_HB) s0 = fma(-D[o + i][o + k], x[k][lane], s0);
                x[i][lane] = (s0 + s1) * __shfl_sync(0xffffffffu, rd, i);
            }
        }
        __syncwarp();
        double *out = inv + warp * LU_HB * LU_HB;
        for (int i = 0; i < LU_HB; ++i) out[i * LU_HB + lane] = x[i][lane];
    }
}

// One CTA: c[r][j] (+)= sum_k a[r][k] b[k][j], 32 k, over a tile of 512 entries
// given as two per thread; a and b in shared memory.
template <int LDA, int LDB>
__device__ __forceinline__ double dot32(const double (*a)[LDA], int r, int a0,
                                        const double (*b)[LDB], int b0, int j, double s)
{
    double t = 0.0;
#pragma unroll 8
    for (int k = 0; k < LU_HB; k += 2) {
        s = fma(a[r][a0 + k], b[b0 + k][j], s);
        t = fma(a[r][a0 + k + 1], b[b0 + k + 1][j], t);
    }
    return s + t;
}

// The panels of block k0 (kb = 64): blockIdx.x < strips: 16 rows of
// L21 = A21 U11^{-1}, with U11 = [U1 V; 0 U2]: X1 = A1 U1^{-1}, X2 = (A2 - X1 V)
// U2^{-1}; the others: 16 columns of U12 = L11^{-1} P A12, with L11 = [L1 0; W
// L2]: Y1 = L1^{-1} B1, Y2 = L2^{-1} (B2 - W Y1).
__global__ void __launch_bounds__(256)
    k_panels(int64_t n, double *__restrict__ A, int64_t lda, int64_t k0, int strips,
             const int32_t *__restrict__ rowperm, const double *__restrict__ inv)
{
    __shared__ double I1[LU_HB][LU_HB + 1], I2[LU_HB][LU_HB + 1], M[LU_HB][LU_HB + 1];
    __shared__ double S[LU_STRIP * LU_LD];  // the strip: 16 x 64 rows, or 64 x 16 + 1 columns
    const int tid = threadIdx.x;
    const bool low = (int)blockIdx.x < strips;
    const int64_t s0 = k0 + LU_NB + (int64_t)LU_STRIP * (low ? blockIdx.x : blockIdx.x - strips);
    const double *i1 = inv + (low ? 2 : 0) * LU_HB * LU_HB, *i2 = i1 + LU_HB * LU_HB;
    for (int e = tid; e < LU_HB * LU_HB; e += 256) {
        I1[e / LU_HB][e % LU_HB] = i1[e];
        I2[e / LU_HB][e % LU_HB] = i2[e];
        const int r = e % LU_HB, c = e / LU_HB;
        // V = U[0:32, 32:64] or W = L[32:64, 0:32]
        M[r][c] = low ? A[(k0 + r) + (k0 + LU_HB + c) * lda] : A[(k0 + LU_HB + r) + (k0 + c) * lda];
    }
    if (low) {
        double(*T)[LU_LD] = reinterpret_cast<double(*)[LU_LD]>(S);
        for (int e = tid; e < LU_STRIP * LU_NB; e += 256) {
            const int r = e % LU_STRIP, c = e / LU_STRIP;
            T[r][c] = s0 + r < n ? A[(s0 + r) + (k0 + c) * lda] : 0.0;
        }
        __syncthreads();
        const int j = tid & 31, r = tid >> 5;  // rows r and r + 8
        const double x0 = dot32<LU_LD, LU_HB + 1>(T, r, 0, I1, 0, j, 0.0);
        const double x1 = dot32<LU_LD, LU_HB + 1>(T, r + 8, 0, I1, 0, j, 0.0);
        __syncthreads();
        T[r][j] = x0;
        T[r + 8][j] = x1;
        __syncthreads();
        const double t0 = T[r][LU_HB + j] - dot32<LU_LD, LU_HB + 1>(T, r, 0, M, 0, j, 0.0);
        const double t1 = T[r + 8][LU_HB + j] - dot32<LU_LD, LU_HB + 1>(T, r + 8, 0, M, 0, j, 0.0);
        T[r][LU_HB + j] = t0;  // each thread its own entries
        T[r + 8][LU_HB + j] = t1;
        __syncthreads();
        const double y0 = dot32<LU_LD, LU_HB + 1>(T, r, LU_HB, I2, 0, j, 0.0);
        const double y1 = dot32<LU_LD, LU_HB + 1>(T, r + 8, LU_HB, I2, 0, j, 0.0);
        __syncthreads();
        T[r][LU_HB + j] = y0;
        T[r + 8][LU_HB + j] = y1;
        __syncthreads();
        for (int e = tid; e < LU_STRIP * LU_NB; e += 256) {
            const int rr = e % LU_STRIP, c = e / LU_STRIP;
            if (s0 + rr < n) A[(s0 + rr) + (k0 + c) * lda] = T[rr][c];
        }
    } else {
        constexpr int LDB = LU_STRIP;
        double(*T)[LDB] = reinterpret_cast<double(*)[LDB]>(S);
        for (int e = tid; e < LU_STRIP * LU_NB; e += 256) {
            const int r = e % LU_NB, c = e / LU_NB;
            T[r][c] = s0 + c < n ? A[rowperm[k0 + r] + (s0 + c) * lda] : 0.0;
        }
        __syncthreads();
        const int j = tid & 15, r = tid >> 4;  // rows r and r + 16
        const double x0 = dot32<LU_HB + 1, LDB>(I1, r, 0, T, 0, j, 0.0);
        const double x1 = dot32<LU_HB + 1, LDB>(I1, r + 16, 0, T, 0, j, 0.0);
        __syncthreads();
        T[r][j] = x0;
        T[r + 16][j] = x1;
        __syncthreads();
        const double t0 = T[LU_HB + r][j] - dot32<LU_HB + 1, LDB>(M, r, 0, T, 0, j, 0.0);
        const double t1 = T[LU_HB + r + 16][j] - dot32<LU_HB + 1, LDB>(M, r + 16, 0, T, 0, j, 0.0);
        T[LU_HB + r][j] = t0;
        T[LU_HB + r + 16][j] = t1;
        __syncthreads();
        const double y0 = dot32<LU_HB + 1, LDB>(I2, r, 0, T, LU_HB, j, 0.0);
        const double y1 = dot32<LU_HB + 1, LDB>(I2, r + 16, 0, T, LU_HB, j, 0.0);
        __syncthreads();
        T[LU_HB + r][j] = y0;
        T[LU_HB + r + 16][j] = y1;
        __syncthreads();
        for (int e = tid; e < LU_STRIP * LU_NB; e += 256) {
            const int rr = e % LU_NB, c = e / LU_NB;
            if (s0 + c < n) A[(k0 + rr) + (s0 + c) * lda] = T[rr][c];
        }
    }
}

// Every block's row exchange on the columns left of it, after the last step:
// blockIdx.y the block (from the second on), one thread a column.
__global__ void __launch_bounds__(128)
    k_swap_left(int64_t n, double *__restrict__ A, int64_t lda, const int32_t *__restrict__ rowperm)
{
    __shared__ int32_t lp[LU_NB];
    __shared__ double T[LU_NB][33];
    const int64_t k0 = (int64_t)LU_NB * (blockIdx.y + 1), c0 = (int64_t)blockIdx.x * 32;
    if (c0 >= k0) return;
    const int kb = (int)min((int64_t)LU_NB, n - k0);
    if (threadIdx.x < kb) lp[threadIdx.x] = (int32_t)(rowperm[k0 + threadIdx.x] - k0);
    for (int e = threadIdx.x; e < LU_NB * 32; e += 128) {
        const int r = e % LU_NB, c = e / LU_NB;  // c0 + 32 <= k0
        if (r < kb) T[r][c] = A[(k0 + r) + (c0 + c) * lda];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < LU_NB * 32; e += 128) {
        const int r = e % LU_NB, c = e / LU_NB;
        if (r < kb) A[(k0 + r) + (c0 + c) * lda] = T[lp[r]][c];
    }
}

// A22 -= L21 U12 on the CUDA cores (64 x 64 tiles, 4 x 4 per thread).
__global__ void __launch_bounds__(256)
    k_gemm_update(int64_t n, double *__restrict__ A, int64_t lda, int64_t k0, int kb)
{
    using T = double;
    constexpr int BM = 64, BN = 64, BK = 16;
    __shared__ T As[BK][BM + 4];
    __shared__ T Bs[BK][BN + 4];
    const int64_t s = k0 + kb;
    const int64_t row0 = s + (int64_t)blockIdx.x * BM, col0 = s + (int64_t)blockIdx.y * BN;
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    T acc[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = T(0);
    for (int kk = 0; kk < kb; kk += BK) {
        for (int e = threadIdx.x; e < BK * BM; e += 256) {
            const int i = e % BM, k = e / BM;
            const int64_t gi = row0 + i;
            const int gk = kk + k;
            As[k][i] = (gi < n && gk < kb) ? A[gi + (k0 + gk) * lda] : T(0);
        }
        for (int e = threadIdx.x; e < BK * BN; e += 256) {
            const int k = e % BK, j = e / BK;
            const int64_t gj = col0 + j;
            const int gk = kk + k;
            Bs[k][j] = (gj < n && gk < kb) ? A[(k0 + gk) + gj * lda] : T(0);
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < BK; ++k) {
            T a[4], b[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) a[r] = As[k][tx + 16 * r];
#pragma unroll
            for (int c = 0; c < 4; ++c) b[c] = Bs[k][ty * 4 + c];
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[r][c] += a[r] * b[c];
        }
        __syncthreads();
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int64_t gj = col0 + ty * 4 + c;
        if (gj >= n) continue;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int64_t gi = row0 + tx + 16 * r;
            if (gi < n) A[gi + gj * lda] -= acc[r][c];
        }
    }
}

size_t lu_inverse_doubles(int64_t n) { return (size_t)ceil_div(n, LU_NB) * 4 * LU_HB * LU_HB; }

int run_lu_fp64(Ctx &c, double *A, int64_t lda)
{
    const int64_t n = c.n, nblk = ceil_div(n, LU_NB);
    if (cudaFuncSetAttribute(k_diag_factor, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             LU_DIAG_SMEM) != cudaSuccess)
        return -1;
    c.tbeg(PH_LU_PANEL);
    cudaMemsetAsync(c.d_info, 0, sizeof(int32_t), c.stream);
    for (int64_t k = 0; k < nblk; ++k) {
        const int64_t k0 = k * LU_NB;
        double *inv = c.d_LUinv + k * 4 * LU_HB * LU_HB;
        if (k > 0) c.tbeg(PH_LU_PANEL);
        k_diag_factor<<<1, 256, LU_DIAG_SMEM, c.stream>>>(n, A, lda, k0, c.d_rowperm, c.d_info, inv);
        c.launches += 1;
        const int64_t rest = n - k0 - LU_NB;
        if (rest <= 0) {
            c.tend(PH_LU_PANEL);
            break;
        }
        const int strips = (int)ceil_div(rest, LU_STRIP);
        k_panels<<<2 * strips, 256, 0, c.stream>>>(n, A, lda, k0, strips, c.d_rowperm, inv);
        c.tend(PH_LU_PANEL);
        c.tbeg(PH_LU_UPDATE);
        const unsigned g = (unsigned)ceil_div(rest, 64);
        k_gemm_update<<<dim3(g, g), 256, 0, c.stream>>>(n, A, lda, k0, LU_NB);
        c.tend(PH_LU_UPDATE);
        c.launches += 2;
    }
    if (nblk > 1) {
        c.tbeg(PH_LU_PANEL);
        k_swap_left<<<dim3((unsigned)(2 * (nblk - 1)), (unsigned)(nblk - 1)), 128, 0, c.stream>>>(
            n, A, lda, c.d_rowperm);
        c.tend(PH_LU_PANEL);
        c.launches += 1;
    }
    return 0;
}

}  // namespace nrs
