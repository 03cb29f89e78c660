// mlp.cu -- learned starting guess for the refinement: a point-wise MLP that
// predicts each force point's force density f_m (in its body's frame) from
// local features, trained with Adam on the solutions the method produces.
// The paper has no learned component; the prediction only changes where the
// refinement of Sec. 4 step 3 starts, never what it converges to.
//
// Architecture: x (17) -> W1 x + b1 -> SiLU -> W2 h1 + b2 -> SiLU -> W3 h2 + b3 (3),
// SiLU(z) = z / (1 + e^-z).  Parameter vector (FP32, NRS_MLP_PARAMS entries):
//   W1 [64][17] row-major, b1 [64], W2 [64][64], b2 [64], W3 [3][64], b3 [3].
// Features of force point m of body b (body frame; L, V, F are the scales):
//   0-2   xi_m / L                 3-5   xidot_m / V
//   6     s = (m - n_off[b]) / max(1, N_b - 1)  (position in the body's point order)
//   7     W_m / mean_b(W)          8-10  one-hot body kind (free, prescribed, static)
//   11-13 B^T U / V                14-16 B^T Omega L / V
// with (U, Omega) the previous stage's solution for a free body, the
// prescribed motion for a prescribed body, zero for a static one.
// Target: B^T f_m / F.  Loss: mean over points and components of the squared error.
//
// Every sum over points (weight gradients, loss, scales) has a fixed order
// that depends only on the number of points: results are deterministic.
#include <math.h>

#include "nrs_internal.cuh"

namespace nrs {

constexpr int MI = NRS_MLP_IN, MH = NRS_MLP_HID, MO = NRS_MLP_OUT, MP = NRS_MLP_PARAMS;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + MH * MI, OFF_W2 = OFF_B1 + MH,
              OFF_B2 = OFF_W2 + MH * MH, OFF_W3 = OFF_B2 + MH, OFF_B3 = OFF_W3 + MO * MH;
static_assert(OFF_B3 + MO == MP, "parameter layout");

constexpr int ML_THREADS = 128;   // 4 warps; one warp evaluates ML_P points at a time
constexpr int GR_THREADS = 256;   // gradient kernel: threads per block
constexpr int GR_POINTS = 32;     // points per block (chunk) of the gradient sums
constexpr int RD_THREADS = 256;   // single-block reductions

// SiLU(z) = z * sigmoid(z), rounded the same way in every kernel
__device__ __forceinline__ float sigmoid(float z) { return 1.0f / (1.0f + expf(-z)); }
__device__ __forceinline__ float silu(float z) { return z * sigmoid(z); }

// Parameters in shared memory for the forward and backward kernels, W1 and W2
// as stored with rows of odd length: a warp reads a row (lane = column) and a
// column (lane = row) without bank conflicts, and the copy in is straight.
struct SmemNet {
    float w1[MH][MI];       // MI = 17 is odd
    float w2[MH][MH + 1];
    float w3[MO][MH];
    float b1[MH], b2[MH], b3[MO];
};

__device__ __forceinline__ void load_net(SmemNet &n, const float *__restrict__ P)
{
    for (int k = threadIdx.x; k < MH * MI; k += blockDim.x) (&n.w1[0][0])[k] = P[OFF_W1 + k];
#pragma unroll 8
    for (int k = threadIdx.x; k < MH * MH; k += blockDim.x) n.w2[k / MH][k % MH] = P[OFF_W2 + k];
    for (int k = threadIdx.x; k < MO * MH; k += blockDim.x) n.w3[k / MH][k % MH] = P[OFF_W3 + k];
    for (int k = threadIdx.x; k < MH; k += blockDim.x) {
        n.b1[k] = P[OFF_B1 + k];
        n.b2[k] = P[OFF_B2 + k];
    }
    if (threadIdx.x < MO) n.b3[threadIdx.x] = P[OFF_B3 + threadIdx.x];
    __syncthreads();
}

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// One warp evaluates ML_P points together: lane j owns hidden units j and
// j + 32 of each.  The layers' products read two weights and, in one broadcast
// load, the ML_P points' input from shared memory for 2 ML_P fused
// multiply-adds; with one point a warp they were bound by these loads (9200
// points, forward and backward: 47 us, 18 us so).  A point's sums run in the same order
// whatever ML_P is.
constexpr int ML_P = 4;
static_assert(ML_P == 4, "the points' values travel as float4");

struct Points {  // one value of each of the warp's points
    float v[ML_P];
};

__device__ __forceinline__ void store4(float4 *s, const Points &a)
{
    *s = make_float4(a.v[0], a.v[1], a.v[2], a.v[3]);
}

// za += sum_i w[lane][i] s[i], zb += sum_i w[lane + 32][i] s[i], or with TRANS
// the columns w[i][lane], w[i][lane + 32]
template <bool TRANS, int LEN, int LD>
__device__ __forceinline__ void layer(const float (*w)[LD], const float4 *s, int lane, Points &za,
                                      Points &zb)
{
#pragma unroll 8
    for (int i = 0; i < LEN; ++i) {
        const float4 h = s[i];
        const float wa = TRANS ? w[i][lane] : w[lane][i];
        const float wb = TRANS ? w[i][lane + 32] : w[lane + 32][i];
        const float hv[ML_P] = {h.x, h.y, h.z, h.w};
#pragma unroll
        for (int p = 0; p < ML_P; ++p) {
            za.v[p] = fmaf(wa, hv[p], za.v[p]);
            zb.v[p] = fmaf(wb, hv[p], zb.v[p]);
        }
    }
}

// The warp's inputs x (MI per point) of points p0 .. p0 + ML_P - 1 into s[i],
// zero beyond npts
__device__ __forceinline__ void load_points(const float *__restrict__ X, int64_t p0, int64_t npts,
                                            int lane, float4 *s)
{
    Points x;
#pragma unroll
    for (int p = 0; p < ML_P; ++p)
        x.v[p] = lane < MI && p0 + p < npts ? X[(p0 + p) * MI + lane] : 0.0f;
    if (lane < MI) store4(&s[lane], x);
    __syncwarp();
}

// Forward pass.  Same operations in the same order as the forward half of
// k_mlp_fwd_bwd.
__global__ void __launch_bounds__(ML_THREADS)
    k_mlp_forward(int64_t npts, const float *__restrict__ P, const float *__restrict__ X,
                  float *__restrict__ Y)
{
    __shared__ SmemNet net;
    __shared__ float4 sv[ML_THREADS / 32][MH];
    load_net(net, P);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t stride = (int64_t)gridDim.x * (ML_THREADS / 32) * ML_P;
    for (int64_t p0 = ((int64_t)blockIdx.x * (ML_THREADS / 32) + w) * ML_P; p0 < npts; p0 += stride) {
        load_points(X, p0, npts, lane, sv[w]);
        Points za, zb;
#pragma unroll
        for (int p = 0; p < ML_P; ++p) za.v[p] = net.b1[lane], zb.v[p] = net.b1[lane + 32];
        layer<false, MI, MI>(net.w1, sv[w], lane, za, zb);
        __syncwarp();
#pragma unroll
        for (int p = 0; p < ML_P; ++p) za.v[p] = silu(za.v[p]), zb.v[p] = silu(zb.v[p]);
        store4(&sv[w][lane], za);
        store4(&sv[w][lane + 32], zb);
        __syncwarp();
#pragma unroll
        for (int p = 0; p < ML_P; ++p) za.v[p] = net.b2[lane], zb.v[p] = net.b2[lane + 32];
        layer<false, MH, MH + 1>(net.w2, sv[w], lane, za, zb);
        __syncwarp();
#pragma unroll
        for (int p = 0; p < ML_P; ++p) {
            const float ha = silu(za.v[p]), hb = silu(zb.v[p]);
#pragma unroll
            for (int o = 0; o < MO; ++o) {
                const float part = warp_sum(fmaf(net.w3[o][lane], ha, net.w3[o][lane + 32] * hb));
                if (lane == 0 && p0 + p < npts) Y[(p0 + p) * MO + o] = part + net.b3[o];
            }
        }
    }
}

// Forward and backward pass of the training loss:
//   Z1 = W1 x + b1, H1 = SiLU(Z1), Z2 = W2 H1 + b2, H2 = SiLU(Z2), Y = W3 H2 + b3,
//   dY = 2 (Y - T) / (3 npts),  D2 = (W3^T dY) * SiLU'(Z2),  D1 = (W2^T D2) * SiLU'(Z1),
// with SiLU'(z) = s (1 + z (1 - s)), s = 1 / (1 + e^-z).  Writes H1, H2, DY,
// D1, D2 for the parameter-gradient sums, and Y when it is not NULL.
__global__ void __launch_bounds__(ML_THREADS)
    k_mlp_fwd_bwd(int64_t npts, const float *__restrict__ P, const float *__restrict__ X,
                  const float *__restrict__ T, float *__restrict__ Y, float *__restrict__ H1,
                  float *__restrict__ H2, float *__restrict__ DY, float *__restrict__ D1,
                  float *__restrict__ D2)
{
    __shared__ SmemNet net;
    __shared__ float4 sv[ML_THREADS / 32][MH];
    load_net(net, P);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const float scale = 2.0f / (float)(3 * npts);
    const int64_t stride = (int64_t)gridDim.x * (ML_THREADS / 32) * ML_P;
    for (int64_t p0 = ((int64_t)blockIdx.x * (ML_THREADS / 32) + w) * ML_P; p0 < npts; p0 += stride) {
        load_points(X, p0, npts, lane, sv[w]);
        Points z1a, z1b, z2a, z2b, s1a, s1b, s2a, s2b, ha, hb;
#pragma unroll
        for (int p = 0; p < ML_P; ++p) z1a.v[p] = net.b1[lane], z1b.v[p] = net.b1[lane + 32];
        layer<false, MI, MI>(net.w1, sv[w], lane, z1a, z1b);
        __syncwarp();
#pragma unroll
        for (int p = 0; p < ML_P; ++p) {
            s1a.v[p] = sigmoid(z1a.v[p]);
            s1b.v[p] = sigmoid(z1b.v[p]);
            ha.v[p] = z1a.v[p] * s1a.v[p];
            hb.v[p] = z1b.v[p] * s1b.v[p];
            if (p0 + p < npts) {
                H1[(p0 + p) * MH + lane] = ha.v[p];
                H1[(p0 + p) * MH + lane + 32] = hb.v[p];
            }
        }
        store4(&sv[w][lane], ha);
        store4(&sv[w][lane + 32], hb);
        __syncwarp();
#pragma unroll
        for (int p = 0; p < ML_P; ++p) z2a.v[p] = net.b2[lane], z2b.v[p] = net.b2[lane + 32];
        layer<false, MH, MH + 1>(net.w2, sv[w], lane, z2a, z2b);
        __syncwarp();
        Points da, db;
#pragma unroll
        for (int p = 0; p < ML_P; ++p) {
            const bool in = p0 + p < npts;
            s2a.v[p] = sigmoid(z2a.v[p]);
            s2b.v[p] = sigmoid(z2b.v[p]);
            const float h2a = z2a.v[p] * s2a.v[p], h2b = z2b.v[p] * s2b.v[p];
            if (in) {
                H2[(p0 + p) * MH + lane] = h2a;
                H2[(p0 + p) * MH + lane + 32] = h2b;
            }
            float dy[MO], ga = 0.0f, gb = 0.0f;
#pragma unroll
            for (int o = 0; o < MO; ++o) {
                const float y = warp_sum(fmaf(net.w3[o][lane], h2a, net.w3[o][lane + 32] * h2b)) +
                                net.b3[o];
                if (Y && lane == 0 && in) Y[(p0 + p) * MO + o] = y;
                dy[o] = in ? scale * (y - T[(p0 + p) * MO + o]) : 0.0f;
            }
            if (lane < MO && in)
                DY[(p0 + p) * MO + lane] = lane == 0 ? dy[0] : (lane == 1 ? dy[1] : dy[2]);
#pragma unroll
            for (int o = 0; o < MO; ++o) {
                ga = fmaf(net.w3[o][lane], dy[o], ga);
                gb = fmaf(net.w3[o][lane + 32], dy[o], gb);
            }
            da.v[p] = ga * (s2a.v[p] * (1.0f + z2a.v[p] * (1.0f - s2a.v[p])));
            db.v[p] = gb * (s2b.v[p] * (1.0f + z2b.v[p] * (1.0f - s2b.v[p])));
            if (in) {
                D2[(p0 + p) * MH + lane] = da.v[p];
                D2[(p0 + p) * MH + lane + 32] = db.v[p];
            }
        }
        store4(&sv[w][lane], da);
        store4(&sv[w][lane + 32], db);
        __syncwarp();
        Points ga, gb;
#pragma unroll
        for (int p = 0; p < ML_P; ++p) ga.v[p] = gb.v[p] = 0.0f;
        layer<true, MH, MH + 1>(net.w2, sv[w], lane, ga, gb);
        __syncwarp();
#pragma unroll
        for (int p = 0; p < ML_P; ++p)
            if (p0 + p < npts) {
                D1[(p0 + p) * MH + lane] =
                    ga.v[p] * (s1a.v[p] * (1.0f + z1a.v[p] * (1.0f - s1a.v[p])));
                D1[(p0 + p) * MH + lane + 32] =
                    gb.v[p] * (s1b.v[p] * (1.0f + z1b.v[p] * (1.0f - s1b.v[p])));
            }
    }
}

// Partial parameter gradients of GR_POINTS points (one block), summed in
// point order in FP32 from shared-memory tiles:
//   W1[j][i]: D1[p][j] X[p][i]    b1[j]: D1[p][j]    W2[j][i]: D2[p][j] H1[p][i]
//   b2[j]: D2[p][j]               W3[o][j]: DY[p][o] H2[p][j]    b3[o]: DY[p][o]
// W2 in 4 x 4 tiles, one per thread (two 16-byte shared loads for 16 fused
// multiply-adds, 12 us for 9200 points; one entry a thread at a time took 21), the
// rest one entry a thread.
__global__ void __launch_bounds__(GR_THREADS)
    k_mlp_grad_part(int64_t npts, const float *__restrict__ X, const float *__restrict__ H1,
                    const float *__restrict__ H2, const float *__restrict__ DY,
                    const float *__restrict__ D1, const float *__restrict__ D2,
                    float *__restrict__ part)
{
    __shared__ __align__(16) float sx[GR_POINTS][MI], sh1[GR_POINTS][MH], sh2[GR_POINTS][MH];
    __shared__ __align__(16) float sd1[GR_POINTS][MH], sd2[GR_POINTS][MH], sdy[GR_POINTS][MO];
    const int64_t p0 = (int64_t)blockIdx.x * GR_POINTS;
    const int np = (int)min((int64_t)GR_POINTS, npts - p0);
    const int tid = threadIdx.x;
#pragma unroll
    for (int k = tid; k < GR_POINTS * MH / 4; k += GR_THREADS) {
        const int q = k / (MH / 4), j = 4 * (k % (MH / 4));
        const bool in = q < np;
        const int64_t g = (p0 + q) * MH + j;
        const float4 z = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        const float4 a = in ? *reinterpret_cast<const float4 *>(H1 + g) : z;
        const float4 b = in ? *reinterpret_cast<const float4 *>(H2 + g) : z;
        const float4 c = in ? *reinterpret_cast<const float4 *>(D1 + g) : z;
        const float4 d = in ? *reinterpret_cast<const float4 *>(D2 + g) : z;
        *reinterpret_cast<float4 *>(&sh1[q][j]) = a;
        *reinterpret_cast<float4 *>(&sh2[q][j]) = b;
        *reinterpret_cast<float4 *>(&sd1[q][j]) = c;
        *reinterpret_cast<float4 *>(&sd2[q][j]) = d;
    }
    for (int k = tid; k < GR_POINTS * MI; k += GR_THREADS) {
        const int q = k / MI, i = k % MI;
        sx[q][i] = q < np ? X[(p0 + q) * MI + i] : 0.0f;
    }
    if (tid < GR_POINTS * MO) {
        const int q = tid / MO, o = tid % MO;
        sdy[q][o] = q < np ? DY[(p0 + q) * MO + o] : 0.0f;
    }
    __syncthreads();
    float *out = part + (int64_t)blockIdx.x * MP;
    {
        const int j0 = 4 * (tid >> 4), i0 = 4 * (tid & 15);
        float acc[4][4] = {};
#pragma unroll 4
        for (int q = 0; q < np; ++q) {
            const float4 d = *reinterpret_cast<const float4 *>(&sd2[q][j0]);
            const float4 h = *reinterpret_cast<const float4 *>(&sh1[q][i0]);
            const float dv[4] = {d.x, d.y, d.z, d.w}, hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(dv[a], hv[b], acc[a][b]);
        }
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) out[OFF_W2 + (j0 + a) * MH + i0 + b] = acc[a][b];
    }
    // W1: rows j = tid / 4, columns 4 (tid mod 4) .. + 3, and column 16
    {
        const int j = tid >> 2, i0 = 4 * (tid & 3);
        const bool last = (tid & 3) == 3;
        float acc[5] = {};
#pragma unroll 4
        for (int q = 0; q < np; ++q) {
            const float d = sd1[q][j];
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[b] = fmaf(d, sx[q][i0 + b], acc[b]);
            if (last) acc[4] = fmaf(d, sx[q][MI - 1], acc[4]);
        }
#pragma unroll
        for (int b = 0; b < 4; ++b) out[OFF_W1 + j * MI + i0 + b] = acc[b];
        if (last) out[OFF_W1 + j * MI + MI - 1] = acc[4];
    }
    // W3 (192 entries) and b1 (64), one a thread
    {
        const int o = tid / MH, j = tid % MH;
        float s = 0.0f;
        if (o < MO) {
#pragma unroll 4
            for (int q = 0; q < np; ++q) s = fmaf(sdy[q][o], sh2[q][j], s);
            out[OFF_W3 + tid] = s;
        } else {
#pragma unroll 4
            for (int q = 0; q < np; ++q) s += sd1[q][j];
            out[OFF_B1 + j] = s;
        }
    }
    // b2 and b3
    if (tid < MH + MO) {
        float s = 0.0f;
#pragma unroll 4
        for (int q = 0; q < np; ++q) s += tid < MH ? sd2[q][tid] : sdy[q][tid - MH];
        out[tid < MH ? OFF_B2 + tid : OFF_B3 + tid - MH] = s;
    }
}
static_assert(GR_THREADS == (MO + 1) * MH && GR_THREADS == 4 * MH && MI == 17, "entries a thread");

// Adam (Kingma & Ba 2015) for parameter k: beta1 = 0.9, beta2 = 0.999,
// epsilon = 1e-8; bc1 = 1 - beta1^t and bc2 = 1 - beta2^t are computed on the
// host in FP64.
__device__ __forceinline__ void adam_update(float *__restrict__ P, float *__restrict__ Mo,
                                            float *__restrict__ Ve, int k, float g, float lr,
                                            float bc1, float bc2)
{
    const float m = fmaf(0.9f, Mo[k], 0.1f * g);
    const float v = fmaf(0.999f, Ve[k], 0.001f * (g * g));
    Mo[k] = m;
    Ve[k] = v;
    P[k] -= lr * (m / bc1) / (sqrtf(v / bc2) + 1e-8f);
}

// G[k] = sum over chunks in FP64, the chunks c, c + 8, ... by eight warps (32
// parameters a block), then the eight sums in order; with lr > 0 also one Adam
// step of the parameters.  (One thread a parameter, 288 chunks one after the
// other, took 49 us for 9200 points; this takes 14.)
constexpr int GF_WARPS = 8;
__global__ void __launch_bounds__(32 * GF_WARPS)
    k_mlp_grad_finish(int chunks, const float *__restrict__ part, float *__restrict__ G,
                      float *__restrict__ P, float *__restrict__ Mo, float *__restrict__ Ve,
                      float lr, float bc1, float bc2)
{
    __shared__ double sum[GF_WARPS][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int k = blockIdx.x * 32 + lane;
    double s = 0.0;
    if (k < MP) {
#pragma unroll 4
        for (int c = w; c < chunks; c += GF_WARPS) s += (double)part[(int64_t)c * MP + k];
    }
    sum[w][lane] = s;
    __syncthreads();
    if (w || k >= MP) return;
#pragma unroll
    for (int v = 1; v < GF_WARPS; ++v) s += sum[v][lane];
    const float g = (float)s;
    if (G) G[k] = g;
    if (lr > 0.0f) adam_update(P, Mo, Ve, k, g, lr, bc1, bc2);
}

__device__ double block_sum_fixed(double v)
{
    __shared__ double red[RD_THREADS];
    red[threadIdx.x] = v;
    __syncthreads();
    for (int w = RD_THREADS / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    const double r = red[0];
    __syncthreads();
    return r;
}

__device__ double block_max_fixed(double v)
{
    __shared__ double red[RD_THREADS];
    red[threadIdx.x] = v;
    __syncthreads();
    for (int w = RD_THREADS / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + w]);
        __syncthreads();
    }
    const double r = red[0];
    __syncthreads();
    return r;
}

// loss[0] = mean of (Y - T)^2 and loss[1] = mean of T^2 over the npts * 3
// entries (one block).
__global__ void __launch_bounds__(RD_THREADS)
    k_mlp_loss(int64_t npts, const float *__restrict__ Y, const float *__restrict__ T,
               double *__restrict__ loss)
{
    double s = 0.0, t2 = 0.0;
    for (int64_t i = threadIdx.x; i < npts * MO; i += RD_THREADS) {
        const double d = (double)Y[i] - (double)T[i];
        s += d * d;
        t2 += (double)T[i] * (double)T[i];
    }
    s = block_sum_fixed(s);
    t2 = block_sum_fixed(t2);
    if (threadIdx.x == 0) {
        loss[0] = s / (double)(npts * MO);
        loss[1] = t2 / (double)(npts * MO);
    }
}

// One Adam step with a given gradient G.
__global__ void k_mlp_adam(float *__restrict__ P, float *__restrict__ Mo, float *__restrict__ Ve,
                           const float *__restrict__ G, float lr, float bc1, float bc2)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < MP) adam_update(P, Mo, Ve, k, G[k], lr, bc1, bc2);
}

// Scales from one solved stage: L = max |xi_m|, V = max |b_m| over the force
// rows of the right-hand side, F = sqrt(mean |f_m|^2); a zero scale becomes 1.
__global__ void __launch_bounds__(RD_THREADS)
    k_mlp_scales(int64_t N, const D4 *__restrict__ xi, const double *__restrict__ b,
                 const double *__restrict__ sol, double *__restrict__ out)
{
    double lmax = 0.0, vmax = 0.0, fsum = 0.0;
    for (int64_t m = threadIdx.x; m < N; m += RD_THREADS) {
        const D4 p = xi[m];
        lmax = fmax(lmax, sqrt(p.x * p.x + p.y * p.y + p.z * p.z));
        const double *bm = b + 3 * m, *fm = sol + 3 * m;
        vmax = fmax(vmax, sqrt(bm[0] * bm[0] + bm[1] * bm[1] + bm[2] * bm[2]));
        fsum += fm[0] * fm[0] + fm[1] * fm[1] + fm[2] * fm[2];
    }
    lmax = block_max_fixed(lmax);
    vmax = block_max_fixed(vmax);
    fsum = block_sum_fixed(fsum);
    if (threadIdx.x == 0) {
        const double F = sqrt(fsum / (double)N);
        out[0] = lmax > 0.0 ? lmax : 1.0;
        out[1] = vmax > 0.0 ? vmax : 1.0;
        out[2] = F > 0.0 ? F : 1.0;
    }
}

// Per-body mean of W_n (one thread per body).
__global__ void k_mlp_wmean(int nbodies, const int64_t *__restrict__ n_off,
                            const double *__restrict__ W, double *__restrict__ Wmean)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nbodies) return;
    double s = 0.0;
    for (int64_t m = n_off[b]; m < n_off[b + 1]; ++m) s += W[m];
    const int64_t cnt = n_off[b + 1] - n_off[b];
    Wmean[b] = cnt > 0 ? s / (double)cnt : 0.0;
}

// Features of every force point and, when T is not NULL, the body-frame
// targets from the solution sol = [f (3N); (U, Omega) (6F)].
// B row-major per body with the basis vectors as columns: B^T v has
// components sum_r B[r][k] v_r.
__global__ void k_mlp_features(int64_t N, const D4 *__restrict__ xi, const D4 *__restrict__ xidot,
                               const double *__restrict__ W, const double *__restrict__ Wmean,
                               const int64_t *__restrict__ n_off, const int32_t *__restrict__ body_x,
                               const int32_t *__restrict__ kind,
                               const int32_t *__restrict__ free_index, const double *__restrict__ B,
                               const double *__restrict__ Upres, const double *__restrict__ Ompres,
                               const double *__restrict__ vprev, const double *__restrict__ sol,
                               const double *__restrict__ scales, float *__restrict__ X,
                               float *__restrict__ T)
{
    const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= N) return;
    const double L = scales[0], V = scales[1], F = scales[2];
    const int b = body_x[m];
    const double *Bb = B + 9 * b;
    const D4 p = xi[m], v = xidot[m];
    float *x = X + m * MI;
    x[0] = (float)(p.x / L);
    x[1] = (float)(p.y / L);
    x[2] = (float)(p.z / L);
    x[3] = (float)(v.x / V);
    x[4] = (float)(v.y / V);
    x[5] = (float)(v.z / V);
    const int64_t nb = n_off[b + 1] - n_off[b];
    x[6] = (float)((double)(m - n_off[b]) / (double)(nb > 1 ? nb - 1 : 1));
    x[7] = (float)(Wmean[b] > 0.0 ? W[m] / Wmean[b] : 0.0);
    const int kb = kind[b];
    x[8] = kb == NRS_FREE ? 1.0f : 0.0f;
    x[9] = kb == NRS_PRESCRIBED ? 1.0f : 0.0f;
    x[10] = kb == NRS_STATIC ? 1.0f : 0.0f;
    double U[3] = {0.0, 0.0, 0.0}, Om[3] = {0.0, 0.0, 0.0};
    if (kb == NRS_PRESCRIBED) {
        for (int k = 0; k < 3; ++k) {
            U[k] = Upres[3 * b + k];
            Om[k] = Ompres[3 * b + k];
        }
    } else if (kb == NRS_FREE && vprev) {
        const int f = free_index[b];
        for (int k = 0; k < 3; ++k) {
            U[k] = vprev[6 * f + k];
            Om[k] = vprev[6 * f + 3 + k];
        }
    }
    for (int k = 0; k < 3; ++k) {
        const double ub = Bb[k] * U[0] + Bb[3 + k] * U[1] + Bb[6 + k] * U[2];
        const double ob = Bb[k] * Om[0] + Bb[3 + k] * Om[1] + Bb[6 + k] * Om[2];
        x[11 + k] = (float)(ub / V);
        x[14 + k] = (float)(ob * L / V);
    }
    if (T) {
        const double *fm = sol + 3 * m;
        for (int k = 0; k < 3; ++k)
            T[m * MO + k] =
                (float)((Bb[k] * fm[0] + Bb[3 + k] * fm[1] + Bb[6 + k] * fm[2]) / F);
    }
}

// Start vector from a prediction Y: f_m = F B y_m; (U, Omega) of the free
// bodies from vprev (zero when NULL).  bad[0] is set if any entry is not finite.
__global__ void k_mlp_to_start(int64_t N, int64_t nfree, const float *__restrict__ Y,
                               const int32_t *__restrict__ body_x, const double *__restrict__ B,
                               const double *__restrict__ vprev, const double *__restrict__ scales,
                               double *__restrict__ x0, int32_t *__restrict__ bad)
{
    const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const double F = scales[2];
    if (m < N) {
        const double *Bb = B + 9 * body_x[m];
        const double y0 = Y[m * MO], y1 = Y[m * MO + 1], y2 = Y[m * MO + 2];
        bool ok = true;
        for (int r = 0; r < 3; ++r) {
            const double f = F * (Bb[3 * r] * y0 + Bb[3 * r + 1] * y1 + Bb[3 * r + 2] * y2);
            ok = ok && isfinite(f);
            x0[3 * m + r] = f;
        }
        if (!ok) atomicOr(bad, 1);
    } else if (m < N + 6 * nfree) {
        const int64_t k = m - N;
        const double v = vprev ? vprev[k] : 0.0;
        if (!isfinite(v)) atomicOr(bad, 1);
        x0[3 * N + k] = v;
    }
}

// x0 = xp if its residual norm is the smaller one (and it is finite), else xc.
// used[0] records the choice; used[1] is the non-finite flag of k_mlp_to_start.
__global__ void k_pick_start(int64_t n, const double *__restrict__ xp, const double *__restrict__ xc,
                             const double *__restrict__ norms, double *__restrict__ x0,
                             int32_t *__restrict__ used)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool pred = used[1] == 0 && norms[0] < norms[1];
    if (i < n) x0[i] = pred ? xp[i] : xc[i];
    if (i == 0) used[0] = pred ? 1 : 0;
}

// ---- host side ---------------------------------------------------------------

int mlp_grad_chunks(int64_t npts) { return (int)ceil_div(npts, GR_POINTS); }

static unsigned warp_grid(const Ctx &c, int64_t npts)
{
    // ML_P points per warp, at most four blocks of 4 warps per SM (each block
    // stages all parameters in shared memory first)
    return (unsigned)std::max<int64_t>(
        1, std::min<int64_t>(ceil_div(npts, ML_P * (ML_THREADS / 32)), 4 * (int64_t)c.num_sms));
}

static void bias_corrections(int t, float *bc1, float *bc2)
{
    *bc1 = (float)(1.0 - pow(0.9, (double)t));
    *bc2 = (float)(1.0 - pow(0.999, (double)t));
}

void mlp_eval(Ctx &c, const float *X, int64_t npts, const float *T, float *Y, float *G,
              double *loss_dev)
{
    if (!T || !G) {
        k_mlp_forward<<<warp_grid(c, npts), ML_THREADS, 0, c.stream>>>(npts, c.d_mlp_params, X, Y);
        c.launches += 1;
        if (T && loss_dev) {
            k_mlp_loss<<<1, RD_THREADS, 0, c.stream>>>(npts, Y, T, loss_dev);
            c.launches += 1;
        }
    }
    if (T && G) mlp_train_step(c, X, npts, T, G, 0.0f, Y);
    if (T && G && loss_dev) {
        k_mlp_loss<<<1, RD_THREADS, 0, c.stream>>>(npts, Y, T, loss_dev);
        c.launches += 1;
    }
}

void mlp_train_step(Ctx &c, const float *X, int64_t npts, const float *T, float *G, float lr,
                    float *Y)
{
    k_mlp_fwd_bwd<<<warp_grid(c, npts), ML_THREADS, 0, c.stream>>>(
        npts, c.d_mlp_params, X, T, Y, c.d_mlp_z1, c.d_mlp_z2, c.d_mlp_dy, c.d_mlp_d1, c.d_mlp_d2);
    const int chunks = mlp_grad_chunks(npts);
    k_mlp_grad_part<<<(unsigned)chunks, GR_THREADS, 0, c.stream>>>(
        npts, X, c.d_mlp_z1, c.d_mlp_z2, c.d_mlp_dy, c.d_mlp_d1, c.d_mlp_d2, c.d_mlp_part);
    float bc1 = 1.0f, bc2 = 1.0f;
    if (lr > 0.0f) {
        c.mlp_t += 1;
        bias_corrections(c.mlp_t, &bc1, &bc2);
    }
    k_mlp_grad_finish<<<(unsigned)ceil_div(MP, 32), 32 * GF_WARPS, 0, c.stream>>>(
        chunks, c.d_mlp_part, G, c.d_mlp_params, c.d_mlp_m, c.d_mlp_v, lr, bc1, bc2);
    c.launches += 3;
}

void mlp_adam(Ctx &c, const float *G, float lr)
{
    c.mlp_t += 1;
    float bc1, bc2;
    bias_corrections(c.mlp_t, &bc1, &bc2);
    k_mlp_adam<<<(unsigned)ceil_div(MP, 256), 256, 0, c.stream>>>(c.d_mlp_params, c.d_mlp_m,
                                                                  c.d_mlp_v, G, lr, bc1, bc2);
    c.launches += 1;
}

void mlp_scales(Ctx &c, const D4 *xi, const double *b, const double *sol, double *out)
{
    k_mlp_scales<<<1, RD_THREADS, 0, c.stream>>>(c.N, xi, b, sol, out);
    c.launches += 1;
}

void mlp_features(Ctx &c, const D4 *xi, const D4 *xidot, const double *vprev, const double *sol,
                  float *X, float *T)
{
    k_mlp_wmean<<<(unsigned)ceil_div(c.nbodies, 64), 64, 0, c.stream>>>(c.nbodies, c.d_n_off, c.d_W,
                                                                         c.d_mlp_wmean);
    k_mlp_features<<<(unsigned)ceil_div(c.N, 128), 128, 0, c.stream>>>(
        c.N, xi, xidot, c.d_W, c.d_mlp_wmean, c.d_n_off, c.d_body_x, c.d_kind, c.d_free_index,
        c.d_B, c.d_U, c.d_Om, vprev, sol, c.d_mlp_scal, X, T);
    c.launches += 2;
}

void mlp_start(Ctx &c, const float *Y, const double *vprev, double *x0)
{
    cudaMemsetAsync(c.d_mlp_used, 0, 2 * sizeof(int32_t), c.stream);
    k_mlp_to_start<<<(unsigned)ceil_div(c.N + 6 * c.F, 128), 128, 0, c.stream>>>(
        c.N, c.F, Y, c.d_body_x, c.d_B, vprev, c.d_mlp_scal, x0, c.d_mlp_used + 1);
    c.launches += 1;
}

void pick_start(Ctx &c, const double *xp, const double *xc, const double *norms, double *x0)
{
    k_pick_start<<<(unsigned)ceil_div(c.n, 256), 256, 0, c.stream>>>(c.n, xp, xc, norms, x0,
                                                                       c.d_mlp_used);
    c.launches += 1;
}

}  // namespace nrs
