// velocity.cu -- the fluid velocity at field points and the passive tracers
// it carries (the particle tracking of Gallagher & Smith's mouse-node and
// sperm examples): the NEAREST boundary integral of Sec. 3 evaluated off the
// body,
//   u(x_p) = (1/(8 pi mu)) sum_q S^eps(x_p - X_q) w_q f_{n(q)},
// with f the force density of the stage's solve and n(q) the nearest force
// point of quadrature point q.
//
// One CTA takes 128 field points and a contiguous range of quadrature points
// (staged through shared memory with their weighted f_{n(q)} gathered), one
// thread per field point accumulating the three components in FP64.  The
// ranges' partial sums are added in ascending order by a second kernel:
// deterministic.
//
// The FP64 pipe bounds it (64 clocks a warp and scheduler for a fused
// multiply-add, 76 for a plain operation, 572 and 344 for the correctly rounded
// square root and division), so a term is arranged for few operations there:
//   u_j += s (|r|^2 + 2 eps^2) (w f_j) + s (r . w f) r_j,   s = rho^(-3/2),
// 19 fused multiply-adds, with s from a 30-bit 1/sqrt(rho) refined once, and
// that seed's powers and the product s (|r|^2 + 2 eps^2) on the integer pipe
// (fp64_int.cuh).  Every step is rounded in FP64 (s to about 2 units) and the
// sums are taken in groups, so the result is no further from exact than with
// every S_jk w f_k formed and added on its own.  2000 field
// points and 92000 quadrature points: 21.1 ms with all six products S_jk w
// formed as the assembly forms them, 6.4 ms so.
#include "fp64_int.cuh"
#include "nrs_internal.cuh"

namespace nrs {

namespace {

constexpr int VL_THREADS = 128;
constexpr int VL_CHUNK = 256;     // quadrature points staged at a time
constexpr int VL_MIN_RANGE = 64;  // quadrature points of a range, at least
constexpr int VL_GROUP = 16;      // consecutive quadrature points summed apart

// A staged quadrature point: position and w f_{n(q)}.
struct alignas(16) VelPoint {
    double x, y, z, fx, fy, fz;
};

// s = rho^(-3/2) and s dg on the FP64 pipe: rho outside [2^-100, 2^100)
__device__ __noinline__ double2 inv_cube_fp64(double rho, double dg)
{
    const double s = 1.0 / (rho * sqrt(rho));
    return make_double2(s, s * dg);
}

// part[(s * P + p) * 3 + j] = sum over quadrature points q of range s of
// S_jk w_q f_k(n(q)), q ascending in groups of VL_GROUP.  one = 1.0, nz = -0.0
// (run-time values, so that a fused multiply-add stays one).  N force points;
// a quadrature point without a nearest one (no distance was finite: k_nearest
// marks it -1) has no density, and the velocity is NaN.
__global__ void __launch_bounds__(VL_THREADS)
    k_velocity_part(int64_t P, const D4 *__restrict__ xp, int64_t Q, const D4 *__restrict__ Xw,
                    const int32_t *__restrict__ nn, int64_t N, const double *__restrict__ f, double eps2,
                    int64_t q_per_split, double one, double nz, double *__restrict__ part)
{
    __shared__ VelPoint sX[VL_CHUNK];
    const int64_t p = (int64_t)blockIdx.x * VL_THREADS + threadIdx.x;
    const int64_t s = blockIdx.y;
    const int64_t q0 = s * q_per_split, q1 = min(Q, q0 + q_per_split);
    const bool active = p < P;
    const bool idle = p - (threadIdx.x & 31) >= P;  // none of the warp's points exists
    double px = 0.0, py = 0.0, pz = 0.0;
    if (active) {
        const D4 v = xp[p];
        px = v.x;
        py = v.y;
        pz = v.z;
    }
    double a0 = 0.0, a1 = 0.0, a2 = 0.0;
    for (int64_t c0 = q0; c0 < q1; c0 += VL_CHUNK) {
        const int cnt = (int)min((int64_t)VL_CHUNK, q1 - c0);
        __syncthreads();
        for (int i = threadIdx.x; i < cnt; i += VL_THREADS) {
            const D4 X = Xw[c0 + i];
            const int64_t n = nn[c0 + i];
            const bool has = n >= 0 && n < N;
            const double *fq = f + (has ? 3 * n : 0);
            const double w = has ? X.w : __longlong_as_double(0x7ff8000000000000LL);
            sX[i] = VelPoint{X.x, X.y, X.z, w * fq[0], w * fq[1], w * fq[2]};
        }
        __syncthreads();
        if (idle) continue;
        for (int i0 = 0; i0 < cnt; i0 += VL_GROUP) {
            // a group's terms are summed apart: the long sums then take one rounding
            // a group, not two a term
            double t0 = 0.0, t1 = 0.0, t2 = 0.0;
            const int i1 = min(cnt, i0 + VL_GROUP);
#pragma unroll 2
            for (int i = i0; i < i1; ++i) {
                const VelPoint X = sX[i];
                const double rx = fma(X.x, -one, px), ry = fma(X.y, -one, py), rz = fma(X.z, -one, pz);
                const double rho = fma(rx, rx, fma(ry, ry, fma(rz, rz, eps2)));
                const double dg = fma(rho, one, eps2);  // |r|^2 + 2 eps^2
                double inv, sd;
                if ((hi32(double_bits(rho)) - (923u << 20)) < (200u << 20)) {
                    double y2, y3;
                    rsqrt_powers(rho, y2, y3);
                    const double e = fma(-rho, y2, one);
                    inv = fma(1.5, fma(y3, e, nz), y3);
                    bool tie = false;  // (a tie rounds either way here)
                    const Sig d = unpack(dg);
                    sd = pack(mul_sig(unpack(inv), d.m << 1, d.f, tie));
                } else {
                    const double2 v = inv_cube_fp64(rho, dg);
                    inv = v.x;
                    sd = v.y;
                }
                const double rf = fma(rx, X.fx, fma(ry, X.fy, fma(rz, X.fz, nz)));
                const double sr = fma(inv, rf, nz);
                t0 = fma(sd, X.fx, fma(sr, rx, t0));
                t1 = fma(sd, X.fy, fma(sr, ry, t1));
                t2 = fma(sd, X.fz, fma(sr, rz, t2));
            }
            a0 = fma(t0, one, a0);
            a1 = fma(t1, one, a1);
            a2 = fma(t2, one, a2);
        }
    }
    if (active) {
        double *o = part + (s * P + p) * 3;
        o[0] = a0;
        o[1] = a1;
        o[2] = a2;
    }
}

// u[p] = (c sum_s part[s][p], 0), the ranges added in ascending order; one
// thread per component
__global__ void k_velocity_finish(int64_t P, int splits, const double *__restrict__ part, double c,
                                  double *__restrict__ u)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 3 * P) return;
    double a = 0.0;
#pragma unroll 8
    for (int s = 0; s < splits; ++s) a = __dadd_rn(a, part[(int64_t)s * 3 * P + i]);
    const int64_t p = i / 3;
    const int j = (int)(i % 3);
    u[4 * p + j] = __dmul_rn(a, c);
    if (j == 2) u[4 * p + 3] = 0.0;
}

// Tracer positions of the explicit midpoint: stage 0 x = x_save + dt/2 u,
// stage 1 x = x_save + dt u (column 3 kept).
__global__ void k_tracer_update(int64_t P, int stage, double dt, const D4 *__restrict__ x_save,
                                const D4 *__restrict__ u, D4 *__restrict__ x)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= P) return;
    const double h = stage == 0 ? __dmul_rn(0.5, dt) : dt;
    const D4 a = x_save[p], v = u[p];
    D4 r;
    r.x = __dadd_rn(a.x, __dmul_rn(h, v.x));
    r.y = __dadd_rn(a.y, __dmul_rn(h, v.y));
    r.z = __dadd_rn(a.z, __dmul_rn(h, v.z));
    r.w = a.w;
    x[p] = r;
}

}  // namespace

// Quadrature-range splits of the velocity kernel for P field points: about
// four CTAs per SM in all, each range at least VL_MIN_RANGE points (a range's
// terms follow one another; few field points need many ranges to fill the GPU).
int velocity_splits(const Ctx &c, int64_t P)
{
    const int64_t tiles = ceil_div(P, VL_THREADS);
    int64_t s = ceil_div(4 * (int64_t)c.num_sms, tiles);
    s = std::min<int64_t>(s, ceil_div(c.Q, VL_MIN_RANGE));
    return (int)std::max<int64_t>(1, std::min<int64_t>(s, 1024));
}

// u (device [P*4]) at xp (device [P*4]) from the force density f (device,
// 3 per force point), the lab-frame quadrature points Xw (device [Q*4]) and
// the context's nearest-neighbour map; part: device workspace of
// velocity_splits(c, P) * P * 3 doubles.
void launch_velocity(Ctx &c, const D4 *Xw, const D4 *xp, int64_t P, const double *f, D4 *u,
                     double *part, cudaStream_t s)
{
    if (P <= 0) return;
    const int splits = velocity_splits(c, P);
    const int64_t qps = ceil_div(c.Q, splits);
    const double coef = 1.0 / (8.0 * kPi * c.mu);
    dim3 grid((unsigned)ceil_div(P, VL_THREADS), (unsigned)splits);
    k_velocity_part<<<grid, VL_THREADS, 0, s>>>(P, xp, c.Q, Xw, c.d_nn, c.N, f, c.eps * c.eps,
                                                qps, 1.0, -0.0, part);
    k_velocity_finish<<<(unsigned)ceil_div(3 * P, 128), 128, 0, s>>>(
        P, splits, part, coef, reinterpret_cast<double *>(u));
    c.launches += 2;
}

void launch_tracer_update(Ctx &c, int stage, double dt, cudaStream_t s)
{
    k_tracer_update<<<(unsigned)ceil_div(c.n_tracers, 256), 256, 0, s>>>(
        c.n_tracers, stage, dt, c.d_tr_save, c.d_tr_u, c.d_tr);
    c.launches += 1;
}

}  // namespace nrs
