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
// at the end.  Swimmer, n = 2406, factor and solve: 27.8 ms before, 12.0 ms now
// (8.5 the update, of which the FP64 pipe needs 7.4; 1.0 the panels, 1.0 the
// solves; the diagonal blocks, 94 us each, mostly beside the update).
#include "nrs_internal.cuh"

namespace nrs {

constexpr int LU_NB = 64, LU_HB = 32, LU_LD = LU_NB + 1;
constexpr int LU_STRIP = 16;  // rows (columns) of a panel CTA
constexpr int LU_DIAG_SMEM = (LU_NB * LU_LD + 4 * LU_HB * (LU_HB + 1)) * (int)sizeof(double);

constexpr int DF_ROWS = 5;  // rows a warp updates at once

// 1/x within one unit in the last place (rcp_refined): the seed instruction gives
// 20 bits
__device__ __forceinline__ double lu_rcp(double x)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return rcp_refined(x, y);
}

// what its launch asks for: no other CTA of the factorisation fits beside it
constexpr int LU_DIAG_EXCL_SMEM = 190 * 1024;
static_assert(LU_DIAG_SMEM <= LU_DIAG_EXCL_SMEM, "the block fits");

// Factor the diagonal block at k0 with partial pivoting among its own rows, in
// place; rowperm[k0 + i] = k0 + the block row now at i.  inv (4 x 32 x 32,
// row-major): inverses of the triangles L[0:32, 0:32], L[32:64, 32:64] (unit
// lower) and U[0:32, 0:32], U[32:64, 32:64]; identity beyond kb.
//
// One barrier a pivot step: while warps 1 to 7 apply step c to the columns from
// c + 2 on, a row a warp and turn, warp 0 applies it to column c + 1, finds the
// next pivot there and forms the next multipliers.  Rows stay where they are
// until the end; `at` names the row at each position, in two copies like the
// multipliers `F`, since warp 0 is a step ahead.  (With the search, the row
// exchange, the multipliers and the update one after the other, three barriers
// a step, the block took 122 us.)
__global__ void __launch_bounds__(256)
    k_diag_factor(int64_t n, double *__restrict__ A, int64_t lda, int64_t k0,
                  int32_t *__restrict__ rowperm, int32_t *__restrict__ info,
                  double *__restrict__ inv)
{
    extern __shared__ double diag_smem[];  // the block, then the four inverses
    double(*D)[LU_LD] = reinterpret_cast<double(*)[LU_LD]>(diag_smem);
    double(*X)[LU_HB][LU_HB + 1] =
        reinterpret_cast<double(*)[LU_HB][LU_HB + 1]>(diag_smem + LU_NB * LU_LD);
    __shared__ double F[2][LU_NB];  // of positions after the pivot's
    __shared__ int at[2][LU_NB];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int kb = (int)min((int64_t)LU_NB, n - k0);
    for (int idx = tid; idx < LU_NB * LU_NB; idx += 256) {
        const int r = idx % LU_NB, c = idx / LU_NB;
        D[r][c] = r < kb && c < kb ? A[(k0 + r) + (k0 + c) * lda] : (r == c ? 1.0 : 0.0);
    }
    int a0 = lane, a1 = lane + 32;  // warp 0: the rows at positions lane, lane + 32
    __syncthreads();
    // step c = -1 only finds the first pivot
    for (int c = -1; c < kb - 1; ++c) {
        const int b = c & 1, cn = c + 1;
        if (warp == 0) {
            double d0 = D[a0][cn], d1 = D[a1][cn];
            if (c >= 0) {
                const double u = D[at[b][c]][cn];
                if (lane > c) d0 = fma(-F[b][lane], u, d0);
                if (lane + 32 > c) d1 = fma(-F[b][lane + 32], u, d1);
            }
            // the position of largest |d|, lowest on ties: high words first
            const bool in0 = lane >= cn && lane < kb, in1 = lane + 32 >= cn && lane + 32 < kb;
            const unsigned long long k0_ = in0 ? (unsigned long long)__double_as_longlong(fabs(d0)) : 0ULL;
            const unsigned long long k1_ = in1 ? (unsigned long long)__double_as_longlong(fabs(d1)) : 0ULL;
            const unsigned long long km = k1_ > k0_ ? k1_ : k0_;
            const unsigned h = __reduce_max_sync(0xffffffffu, (unsigned)(km >> 32));
            const unsigned l =
                __reduce_max_sync(0xffffffffu, (unsigned)(km >> 32) == h ? (unsigned)km : 0u);
            const unsigned long long m = ((unsigned long long)h << 32) | l;
            const unsigned at0 = __ballot_sync(0xffffffffu, in0 && k0_ == m);
            const unsigned at1 = __ballot_sync(0xffffffffu, in1 && k1_ == m);
            const int p = at0 ? __ffs(at0) - 1 : 31 + __ffs(at1);
            const int src = p & 31, cs = cn & 31;
            const double pv = __shfl_sync(0xffffffffu, p < 32 ? d0 : d1, src);
            const double dc = __shfl_sync(0xffffffffu, cn < 32 ? d0 : d1, cs);
            const int rp = __shfl_sync(0xffffffffu, p < 32 ? a0 : a1, src);
            const int rc = __shfl_sync(0xffffffffu, cn < 32 ? a0 : a1, cs);
            // exchange positions cn and p
            if (lane == src) (p < 32 ? d0 : d1) = dc, (p < 32 ? a0 : a1) = rc;
            if (lane == cs) (cn < 32 ? d0 : d1) = pv, (cn < 32 ? a0 : a1) = rp;
            // multipliers (a zero pivot leaves the column as it is); m has |pv|'s bits,
            // and comparing them spares the FP64 pipe
            if (m == 0) {
                if (lane == 0 && info) atomicCAS(info, 0, (int)(k0 + cn + 1));
            } else if (h > (60u << 20) && h < (1986u << 20)) {  // 2^-963 to 2^963
                const double r = lu_rcp(pv);
                if (lane > cn) d0 *= r;
                if (lane + 32 > cn) d1 *= r;
            } else {
                if (lane > cn) d0 /= pv;
                if (lane + 32 > cn) d1 /= pv;
            }
            F[b ^ 1][lane] = m == 0 ? 0.0 : d0;
            F[b ^ 1][lane + 32] = m == 0 ? 0.0 : d1;
            at[b ^ 1][lane] = a0;
            at[b ^ 1][lane + 32] = a1;
            D[a0][cn] = d0;
            D[a1][cn] = d1;
        } else if (c >= 0) {
            const double *u = D[at[b][c]];
            const int j = c + 2 + lane;
            const double u0 = j < kb ? u[j] : 0.0, u1 = j + 32 < kb ? u[j + 32] : 0.0;
            // five rows at a time, all their loads before the first store
            for (int i0 = c + warp; i0 < kb; i0 += 7 * DF_ROWS) {
                double *row[DF_ROWS], f[DF_ROWS], x0[DF_ROWS], x1[DF_ROWS];
#pragma unroll
                for (int q = 0; q < DF_ROWS; ++q) {
                    const int i = min(i0 + 7 * q, kb - 1);
                    f[q] = -F[b][i];
                    row[q] = D[at[b][i]];
                }
#pragma unroll
                for (int q = 0; q < DF_ROWS; ++q) {
                    x0[q] = j < kb ? row[q][j] : 0.0;
                    x1[q] = j + 32 < kb ? row[q][j + 32] : 0.0;
                }
#pragma unroll
                for (int q = 0; q < DF_ROWS; ++q) {
                    if (i0 + 7 * q >= kb) break;
                    if (j < kb) row[q][j] = fma(f[q], u0, x0[q]);
                    if (j + 32 < kb) row[q][j + 32] = fma(f[q], u1, x1[q]);
                }
            }
        }
        __syncthreads();
    }
    // the rows to their places
    const int *order = at[(kb - 1) & 1];
    {
        double v[LU_NB * LU_NB / 256];
#pragma unroll
        for (int q = 0; q < LU_NB * LU_NB / 256; ++q) {
            const int idx = tid + 256 * q;
            v[q] = D[order[idx / LU_NB]][idx % LU_NB];
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < LU_NB * LU_NB / 256; ++q) {
            const int idx = tid + 256 * q;
            D[idx / LU_NB][idx % LU_NB] = v[q];
        }
        __syncthreads();
    }
    for (int idx = tid; idx < kb * kb; idx += 256) {
        const int r = idx % kb, c = idx / kb;
        A[(k0 + r) + (k0 + c) * lda] = D[r][c];
    }
    if (tid < kb) rowperm[k0 + tid] = (int32_t)(k0 + order[tid]);
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

// A22 -= L21 U12 on the FP64 pipe, which bounds it (64 clocks a warp's fused
// multiply-add): a tile of 32 x 64 with all of its 64 products a sum at once in
// shared memory, 2 x 4 entries a thread.  Small tiles because a step's tiles
// rarely divide by the SMs (64 x 64: at n = 2406 the updates took 9.5 ms, of
// which the pipe needs 7.4).
constexpr int GU_ROWS = 32, GU_LDA = GU_ROWS + 1, GU_LDB = LU_NB + 1;
constexpr int GU_SMEM = LU_NB * (GU_LDA + GU_LDB) * (int)sizeof(double);
// The leading 64 x 64 block is k_lead_update's.
__global__ void __launch_bounds__(256, 4)
    k_gemm_update(int64_t n, double *__restrict__ A, int64_t lda, int64_t k0)
{
    if (blockIdx.y == 0 && blockIdx.x < LU_NB / GU_ROWS) return;
    extern __shared__ double gu_smem[];
    double(*As)[GU_LDA] = reinterpret_cast<double(*)[GU_LDA]>(gu_smem);
    double(*Bs)[GU_LDB] = reinterpret_cast<double(*)[GU_LDB]>(gu_smem + LU_NB * GU_LDA);
    const int64_t s = k0 + LU_NB;
    const int64_t row0 = s + (int64_t)blockIdx.x * GU_ROWS, col0 = s + (int64_t)blockIdx.y * LU_NB;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
#pragma unroll 8
    for (int e = tid; e < LU_NB * GU_ROWS; e += 256) {
        const int i = e % GU_ROWS, k = e / GU_ROWS;
        As[k][i] = row0 + i < n ? A[row0 + i + (k0 + k) * lda] : 0.0;
    }
#pragma unroll 8
    for (int e = tid; e < LU_NB * LU_NB; e += 256) {
        const int k = e % LU_NB, j = e / LU_NB;
        Bs[k][j] = col0 + j < n ? A[(k0 + k) + (col0 + j) * lda] : 0.0;
    }
    double acc[2][4] = {};
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < LU_NB; ++k) {
        const double x0 = As[k][tx], x1 = As[k][tx + 16];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const double y = Bs[k][4 * ty + c];
            acc[0][c] = fma(x0, y, acc[0][c]);
            acc[1][c] = fma(x1, y, acc[1][c]);
        }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int64_t gj = col0 + ty * 4 + c;
        if (gj >= n) continue;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int64_t gi = row0 + tx + 16 * r;
            if (gi < n) A[gi + gj * lda] -= acc[r][c];
        }
    }
}

// The same for the leading 64 x 64 block of A22, the next diagonal block, in 16
// tiles of 16 x 16, one entry a thread: the sums run in the same order.
__global__ void __launch_bounds__(256)
    k_lead_update(int64_t n, double *__restrict__ A, int64_t lda, int64_t k0)
{
    __shared__ double As[LU_NB][17], Bs[LU_NB][17];
    const int64_t s = k0 + LU_NB;
    const int64_t row0 = s + 16 * (blockIdx.x & 3), col0 = s + 16 * (blockIdx.x >> 2);
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int k = ty + 16 * q;
        As[k][tx] = row0 + tx < n ? A[row0 + tx + (k0 + k) * lda] : 0.0;
        const int e = tid + 256 * q, kk = e % LU_NB, j = e / LU_NB;
        Bs[kk][j] = col0 + j < n ? A[(k0 + kk) + (col0 + j) * lda] : 0.0;
    }
    __syncthreads();
    double acc = 0.0;
#pragma unroll 16
    for (int k = 0; k < LU_NB; ++k) acc = fma(As[k][tx], Bs[k][ty], acc);
    if (row0 + tx < n && col0 + ty < n) A[row0 + tx + (col0 + ty) * lda] -= acc;
}

size_t lu_inverse_doubles(int64_t n) { return (size_t)ceil_div(n, LU_NB) * 4 * LU_HB * LU_HB; }

// One factorisation.  The diagonal block of step k + 1 needs only the leading
// block of step k's update: that is brought up to date first, and then the block
// is factored on the main stream while a side stream does the rest of the
// update.  The factorisation of a block is one latency-bound CTA; it asks for
// enough shared memory to have its SM to itself, and starts first.
int run_lu_fp64(Ctx &c, double *A, int64_t lda)
{
    const int64_t n = c.n, nblk = ceil_div(n, LU_NB);
    if (cudaFuncSetAttribute(k_diag_factor, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             LU_DIAG_EXCL_SMEM) != cudaSuccess ||
        cudaFuncSetAttribute(k_gemm_update, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             GU_SMEM) != cudaSuccess)
        return -1;
    c.tbeg(PH_LU_DIAG);
    cudaMemsetAsync(c.d_info, 0, sizeof(int32_t), c.stream);
    for (int64_t k = 0; k < nblk; ++k) {
        const int64_t k0 = k * LU_NB;
        double *inv = c.d_LUinv + k * 4 * LU_HB * LU_HB;
        if (k > 0) c.tbeg(PH_LU_DIAG);
        k_diag_factor<<<1, 256, LU_DIAG_EXCL_SMEM, c.stream>>>(n, A, lda, k0, c.d_rowperm, c.d_info,
                                                              inv);
        c.tend(PH_LU_DIAG);
        c.launches += 1;
        if (k > 0) cudaStreamWaitEvent(c.stream, c.ev_upd, 0);
        const int64_t rest = n - k0 - LU_NB;
        if (rest <= 0) break;
        const int strips = (int)ceil_div(rest, LU_STRIP);
        c.tbeg(PH_LU_PANEL);
        k_panels<<<2 * strips, 256, 0, c.stream>>>(n, A, lda, k0, strips, c.d_rowperm, inv);
        k_lead_update<<<16, 256, 0, c.stream>>>(n, A, lda, k0);
        c.tend(PH_LU_PANEL);
        cudaEventRecord(c.ev_diag, c.stream);
        cudaStreamWaitEvent(c.stream2, c.ev_diag, 0);
        c.tbeg(PH_LU_UPDATE, c.stream2);
        k_gemm_update<<<dim3((unsigned)ceil_div(rest, GU_ROWS), (unsigned)ceil_div(rest, LU_NB)), 256,
                        GU_SMEM, c.stream2>>>(n, A, lda, k0);
        c.tend(PH_LU_UPDATE, c.stream2);
        cudaEventRecord(c.ev_upd, c.stream2);
        c.launches += 3;
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
