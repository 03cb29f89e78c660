// geometry.cu -- kinematics, nearest neighbours, segments of nu, rigid-body
// border and the explicit-midpoint state update (Gallagher & Smith, Sec. 3
// and Sec. 4).
#include <math.h>

#include "fp64_int.cuh"
#include "nrs_internal.cuh"

namespace nrs {

// ---------------------------------------------------------------------------
// kinematics (Sec. 4: the state Y = [X0; B] places each body)
// ---------------------------------------------------------------------------

// x0 + ((B_r0 p0 + B_r1 p1) + B_r2 p2), rounded step by step (no fused
// multiply-add) so that lab-frame clouds are reproducible bit for bit.
__device__ __forceinline__ double rigid_row(const double *x0, const double *B, int r, double p0,
                                            double p1, double p2)
{
    double s = __dadd_rn(__dmul_rn(B[3 * r + 0], p0), __dmul_rn(B[3 * r + 1], p1));
    s = __dadd_rn(s, __dmul_rn(B[3 * r + 2], p2));
    return __dadd_rn(x0[r], s);
}

__global__ void k_kinematics(int64_t N, int64_t Q, int64_t F, const D4 *__restrict__ xi,
                             const D4 *__restrict__ Xiw, const D4 *__restrict__ xidot,
                             const int32_t *__restrict__ body_x, const int32_t *__restrict__ body_X,
                             const int32_t *__restrict__ kind, const double *__restrict__ x0,
                             const double *__restrict__ B, const double *__restrict__ U,
                             const double *__restrict__ Om, const double *__restrict__ ext,
                             D4 *__restrict__ x, D4 *__restrict__ Xw, double *__restrict__ b)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N) {
        int bd = body_x[i];
        const double *o = x0 + 3 * bd;
        const double *Bb = B + 9 * bd;
        D4 p = xi[i];
        D4 r;
        r.x = rigid_row(o, Bb, 0, p.x, p.y, p.z);
        r.y = rigid_row(o, Bb, 1, p.x, p.y, p.z);
        r.z = rigid_row(o, Bb, 2, p.x, p.y, p.z);
        r.w = p.w;
        x[i] = r;
        double v[3] = {0.0, 0.0, 0.0};
        int kd = kind[bd];
        if (kd != NRS_STATIC) {
            D4 d = xidot[i];
            for (int k = 0; k < 3; ++k) {
                double s = __dadd_rn(__dmul_rn(Bb[3 * k + 0], d.x), __dmul_rn(Bb[3 * k + 1], d.y));
                v[k] = __dadd_rn(s, __dmul_rn(Bb[3 * k + 2], d.z));
            }
        }
        if (kd == NRS_PRESCRIBED) {
            double rr[3] = {__dsub_rn(r.x, o[0]), __dsub_rn(r.y, o[1]), __dsub_rn(r.z, o[2])};
            const double *w = Om + 3 * bd;
            double oxr[3] = {__dsub_rn(__dmul_rn(w[1], rr[2]), __dmul_rn(w[2], rr[1])),
                             __dsub_rn(__dmul_rn(w[2], rr[0]), __dmul_rn(w[0], rr[2])),
                             __dsub_rn(__dmul_rn(w[0], rr[1]), __dmul_rn(w[1], rr[0]))};
            for (int k = 0; k < 3; ++k) v[k] = __dadd_rn(v[k], __dadd_rn(U[3 * bd + k], oxr[k]));
        }
        b[3 * i + 0] = v[0];
        b[3 * i + 1] = v[1];
        b[3 * i + 2] = v[2];
    } else if (i < N + Q) {
        int64_t q = i - N;
        int bd = body_X[q];
        const double *o = x0 + 3 * bd;
        const double *Bb = B + 9 * bd;
        D4 p = Xiw[q];
        D4 r;
        r.x = rigid_row(o, Bb, 0, p.x, p.y, p.z);
        r.y = rigid_row(o, Bb, 1, p.x, p.y, p.z);
        r.z = rigid_row(o, Bb, 2, p.x, p.y, p.z);
        r.w = p.w;
        Xw[q] = r;
    } else if (i < N + Q + 6 * F) {
        int64_t c = i - N - Q;
        b[3 * N + c] = ext[c];
    }
}

void launch_kinematics(Ctx &c, const D4 *xi, const D4 *Xiw, const D4 *xidot, D4 *x, D4 *Xw,
                       double *b)
{
    if (x == c.d_x) join_assembly(c);  // (the side stream reads it)
    int64_t total = c.N + c.Q + 6 * c.F;
    int threads = 256;
    c.tbeg(PH_KINEMATICS);
    k_kinematics<<<(unsigned)ceil_div(total, threads), threads, 0, c.stream>>>(
        c.N, c.Q, c.F, xi, Xiw, xidot, c.d_body_x, c.d_body_X, c.d_kind, c.d_x0, c.d_B, c.d_U,
        c.d_Om, c.d_ext, x, Xw, b);
    c.tend(PH_KINEMATICS);
    c.launches += 1;
}

// ---------------------------------------------------------------------------
// nearest neighbours (Sec. 3: n-hat(q) = argmin_n |x[n] - X[q]|)
// ---------------------------------------------------------------------------
//
// The force points are boxed 32 at a time (k_nn_boxes), and a warp only looks
// at the boxes that can hold a nearest neighbour of one of its 8 quadrature
// points: it evaluates the box whose centre is closest to that of its own
// points' box, which bounds every point's distance from above, and keeps the
// boxes whose distance from its own box does not exceed the largest of these
// bounds.  The block stages the boxes that any of its warps kept, each warp
// scans its own.  Points that are neighbours in index order are neighbours in
// space on lattices and curves, so few boxes remain; for points in arbitrary
// order all do: the scan is the full one, and what comes on top is a test of
// every box a warp.  9200 force points and 92000 quadrature points of the
// channel, over all bodies, map and segments with a cold L2: 970 us for the scan
// of all pairs, 150 with boxes kept by warps (270 to 129 us of search when they
// were kept for a whole block: those that straddle two faces keep nearly all).
// Both clouds shuffled: 1029 and 1030 us, force points alone 987 and 1004,
// quadrature points alone 1030 and 347; 9200 x 92000 random points 999 and 957;
// 4000 x 32000 on 1728 lattice places (8 equally near force points on average) 513
// and 353.  (Shuffled clouds took 1164 us when every point was asked whatever the
// boxes looked like and a warp's kept boxes were looked up one by one, lattice
// places 966 when more than four candidates a lane meant all force points again.)
//
// Two passes over the kept force points, staged through shared memory.
// Pass 1 finds m_f, the smallest FP32 squared distance.  With C the largest
// coordinate magnitude involved, every FP32 difference component is within
// delta = 2^-24 (|x| + |X| + |dx|) <= 4.01 * 2^-24 * C of the exact one, so
// the difference vector is within e = sqrt(3) delta <= 4.2e-7 C of exact and
// the FP32 squared distance within 4 u of its rounded components.  A force
// point can be (or tie with) the FP64 minimiser only if
//     sqrt(d2_f) <= (sqrt(m_f) (1 + 1e-6) + 2 e) (1 + 1e-6);
// pass 2 evaluates exactly those candidates in FP64 with the operation order
// ((dx*dx + dy*dy) + dz*dz), keeping the first strict minimum in ascending
// index order.  The 1e-6 factors dominate every FP32 rounding of the bound
// itself (u = 2^-24 ~ 6e-8), so the result equals an exhaustive FP64 search.
// The same bound on a distance from above, taken over the warp, is compared
// with the boxes' squared distances from below: the boxes are rounded outward,
// and the FP32 rounding of the distance between two boxes (relative, 6 u) is
// again inside the 1e-6 factors.

constexpr int NN_TILE = 512;                       // force points staged at a time
constexpr int NN_BOXES = NN_TILE / NN_BOX;         // boxes staged at a time
static_assert(NN_BOX == 32 && NN_TILE == NN_THREADS, "a warp stages a box");

__device__ __forceinline__ float warp_min(float v)
{
    for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__device__ __forceinline__ float warp_max(float v)
{
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// v rounded to the nearest float (a tie away from zero): on the integer pipe,
// because an FP64 conversion takes the FP64 pipe 68 clocks
__device__ __forceinline__ float nearest_float(double v)
{
    float hi, lo;
    if (split_pair(v, hi, lo)) return hi;
    return v == 0.0 ? 0.0f : __double2float_rn(v);
}

// floats below and above whatever rounds to f (not a number for infinite f)
__device__ __forceinline__ float below(float f) { return f - (fabsf(f) * 1.2e-7f + 1e-44f); }
__device__ __forceinline__ float above(float f) { return f + (fabsf(f) * 1.2e-7f + 1e-44f); }

// boxes[2 k], boxes[2 k + 1]: lower and upper corner of force points
// [32 k, 32 k + 32), rounded outward (NaN coordinates left out: such a point is
// never a nearest neighbour)
__global__ void __launch_bounds__(256)
    k_nn_boxes(int64_t N, const D4 *__restrict__ x, float4 *__restrict__ boxes)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const float inf = __int_as_float(0x7f800000);
    float4 lo = make_float4(inf, inf, inf, 0.0f), hi = make_float4(-inf, -inf, -inf, 0.0f);
    if (i < N) {
        const D4 p = x[i];
        lo = make_float4(fminf(__double2float_rd(p.x), inf), fminf(__double2float_rd(p.y), inf),
                         fminf(__double2float_rd(p.z), inf), 0.0f);
        hi = make_float4(fmaxf(__double2float_ru(p.x), -inf), fmaxf(__double2float_ru(p.y), -inf),
                         fmaxf(__double2float_ru(p.z), -inf), 0.0f);
    }
    lo = make_float4(warp_min(lo.x), warp_min(lo.y), warp_min(lo.z), 0.0f);
    hi = make_float4(warp_max(hi.x), warp_max(hi.y), warp_max(hi.z), 0.0f);
    if ((threadIdx.x & 31) == 0 && i < N) {
        boxes[2 * (i / NN_BOX)] = lo;
        boxes[2 * (i / NN_BOX) + 1] = hi;
    }
}

// The NN_SPLIT threads of a quadrature point are consecutive lanes; each scans
// the candidates i = sub, sub + NN_SPLIT, ... of every tile in ascending order,
// and the lanes combine their results: the FP32 minimum (exact, order-free)
// and, in pass 2, the lexicographic minimum of (FP64 distance, index), which
// is the first strict minimum of the ascending scan.
__global__ void __launch_bounds__(NN_THREADS)
    k_nearest(const NNTask *__restrict__ tasks, const int64_t *__restrict__ n_off, int nbodies,
              int global, const D4 *__restrict__ x, const D4 *__restrict__ X,
              const float4 *__restrict__ boxes, int32_t *__restrict__ nn, int32_t *status)
{
    constexpr int WARPS = NN_THREADS / 32, WORDS = NN_THREADS / 32;
    __shared__ float4 tile[NN_TILE];
    __shared__ int32_t list[NN_THREADS];         // boxes of a chunk that some warp kept, ascending
    __shared__ unsigned int mask[WARPS][WORDS];  // each warp's kept boxes of the chunk
    __shared__ unsigned int s_cmax;
    __shared__ int s_cnt[WARPS];
    const NNTask t = tasks[blockIdx.x];
    const int64_t n_lo = global ? 0 : n_off[t.body];
    const int64_t n_hi = global ? n_off[nbodies] : n_off[t.body + 1];
    const int64_t b_lo = n_lo / NN_BOX, b_hi = ceil_div(n_hi, NN_BOX);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int sub = tid % NN_SPLIT;
    const int64_t q = (int64_t)t.q0 + tid / NN_SPLIT;
    const bool active = q < t.q1;
    const float inf = __int_as_float(0x7f800000), nan = __int_as_float(0x7fffffff);
    double qx = 0.0, qy = 0.0, qz = 0.0;
    float4 ql = make_float4(inf, inf, inf, 0.0f), qh = make_float4(-inf, -inf, -inf, 0.0f);
    if (active) {
        D4 p = X[q];
        qx = p.x;
        qy = p.y;
        qz = p.z;
    }
    const float fx = nearest_float(qx), fy = nearest_float(qy), fz = nearest_float(qz);
    if (active) {
        ql = make_float4(below(fx), below(fy), below(fz), 0.0f);
        qh = make_float4(above(fx), above(fy), above(fz), 0.0f);
    }
    if (tid == 0) s_cmax = 0u;
    // the box of the warp's quadrature points
    ql = make_float4(warp_min(ql.x), warp_min(ql.y), warp_min(ql.z), 0.0f);
    qh = make_float4(warp_max(qh.x), warp_max(qh.y), warp_max(qh.z), 0.0f);
    // the box whose centre is closest: lexicographic minimum of (distance, index)
    int64_t seed;
    {
        unsigned key = 0xffffffffu, at = 0u;
        for (int64_t k = b_lo + lane; k < b_hi; k += 32) {
            const float4 l = boxes[2 * k], h = boxes[2 * k + 1];
            const float cx = (l.x + h.x) - (ql.x + qh.x), cy = (l.y + h.y) - (ql.y + qh.y);
            const float cz = (l.z + h.z) - (ql.z + qh.z);
            const unsigned d = __float_as_uint(cx * cx + cy * cy + cz * cz) & 0x7fffffffu;
            if (d < key) {
                key = d;
                at = (unsigned)(k - b_lo);
            }
        }
        const unsigned wk = __reduce_min_sync(0xffffffffu, key);
        seed = b_lo + __reduce_min_sync(0xffffffffu, key == wk ? at : 0xffffffffu);
    }
    float best = inf;
    __syncthreads();  // s_cmax is set
    // box k into this warp's slice of the tile
    auto stage = [&](int64_t k) {
        const int64_t i = k * NN_BOX + lane;
        float4 v = make_float4(nan, nan, nan, 0.0f);
        float lmax = 0.0f;
        if (i >= n_lo && i < n_hi) {
            const D4 p = x[i];
            v = make_float4(nearest_float(p.x), nearest_float(p.y), nearest_float(p.z), 0.0f);
            lmax = fmaxf(fabsf(v.x), fmaxf(fabsf(v.y), fabsf(v.z)));
        }
        tile[tid] = v;
        lmax = warp_max(lmax);
        if (lane == 0) atomicMax(&s_cmax, __float_as_uint(lmax));
    };
    auto scan = [&](int slot) {
        if (active) {
#pragma unroll
            for (int i = sub; i < NN_BOX; i += NN_SPLIT) {
                const float4 v = tile[slot * NN_BOX + i];
                const float dx = v.x - fx, dy = v.y - fy, dz = v.z - fz;
                best = fminf(best, dx * dx + dy * dy + dz * dz);
            }
        }
    };
    // the first cnt boxes of the tile in one run (a box at a time takes a tenth longer)
    auto scan_all = [&](int cnt) {
        if (active) {
#pragma unroll 16
            for (int i = sub; i < cnt * NN_BOX; i += NN_SPLIT) {
                const float4 v = tile[i];
                const float dx = v.x - fx, dy = v.y - fy, dz = v.z - fz;
                best = fminf(best, dx * dx + dy * dy + dz * dz);
            }
        }
    };
    // the squared bound above for the smallest distance so far, and 1e-43 for the
    // absolute rounding of squares that are subnormal (distances below 1e-19)
    auto bound = [&]() {
#pragma unroll
        for (int o = 1; o < NN_SPLIT; o <<= 1)
            best = fminf(best, __shfl_xor_sync(0xffffffffu, best, o));
        const float cmax =
            fmaxf(__uint_as_float(s_cmax), fmaxf(fabsf(fx), fmaxf(fabsf(fy), fabsf(fz))));
        const float e = 4.2e-7f * cmax;
        const float th = (sqrtf(best) * (1.0f + 1e-6f) + 2.0f * e + 1e-30f) * (1.0f + 1e-6f);
        return th * th + 1e-43f;
    };
    // the largest of the warp's bounds (a point that is not a number has none)
    auto warp_bound = [&](float th) {
        return __uint_as_float(
            __reduce_max_sync(0xffffffffu, active && th >= 0.0f ? __float_as_uint(th) : 0u));
    };
    // each quadrature point's own closest box (by centre), evaluated for it: for
    // warps whose points lie far apart, which one box serves badly
    auto seed_each = [&]() {
        unsigned key = 0xffffffffu, at = 0u;
        for (int64_t k = b_lo + sub; k < b_hi; k += NN_SPLIT) {
            const float4 l = boxes[2 * k], h = boxes[2 * k + 1];
            const float cx = (l.x + h.x) - 2.0f * fx, cy = (l.y + h.y) - 2.0f * fy;
            const float cz = (l.z + h.z) - 2.0f * fz;
            const unsigned d = __float_as_uint(cx * cx + cy * cy + cz * cz) & 0x7fffffffu;
            if (d < key) {
                key = d;
                at = (unsigned)(k - b_lo);
            }
        }
#pragma unroll
        for (int o = 1; o < NN_SPLIT; o <<= 1) {
            const unsigned ok = __shfl_xor_sync(0xffffffffu, key, o);
            const unsigned oa = __shfl_xor_sync(0xffffffffu, at, o);
            if (ok < key || (ok == key && oa < at)) {
                key = ok;
                at = oa;
            }
        }
        for (int j = 0; j < 32 / NN_SPLIT; ++j) {
            stage(b_lo + __shfl_sync(0xffffffffu, at, NN_SPLIT * j));
            __syncwarp();
            if (lane / NN_SPLIT == j) scan(warp);
            __syncwarp();
        }
    };
    constexpr int NN_MANY = 16;  // kept boxes of a chunk from which on each point is asked
    // whether asking can leave boxes out: not if half of those kept hold the warp's
    // first point (force points in no spatial order: every box is the whole cloud)
    auto worth_asking = [&](int64_t k0, int words, unsigned mine) {
        const float px = __shfl_sync(0xffffffffu, fx, 0), py = __shfl_sync(0xffffffffu, fy, 0);
        const float pz = __shfl_sync(0xffffffffu, fz, 0);
        int all = 0, hold = 0;
        for (int w = 0; w < words; ++w) {
            const unsigned bits = __shfl_sync(0xffffffffu, mine, w);
            if (!bits) continue;
            bool in = (bits >> lane) & 1u;
            if (in) {
                const int64_t k = k0 + 32 * w + lane;
                const float4 l = boxes[2 * k], h = boxes[2 * k + 1];
                in = l.x <= px && px <= h.x && l.y <= py && py <= h.y && l.z <= pz && pz <= h.z;
            }
            hold += __popc(__ballot_sync(0xffffffffu, in));
            all += __popc(bits);
        }
        return 2 * hold < all;
    };
    bool seeded = false;
    // keeps, of the chunk of NN_THREADS boxes from k0 on, those within th of one
    // of the warp's points; returns how many some warp of the block kept
    auto keep = [&](int64_t k0, float &th) {
        const int words = (int)min((int64_t)WORDS, ceil_div(b_hi - k0, 32));
        const float u2 = warp_bound(th);
        unsigned mine = 0u;
        for (int w = 0; w < words; ++w) {
            const int64_t k = k0 + 32 * w + lane;
            bool in = false;
            if (k < b_hi) {
                const float4 l = boxes[2 * k], h = boxes[2 * k + 1];
                const float dx = fmaxf(0.0f, fmaxf(l.x - qh.x, ql.x - h.x));
                const float dy = fmaxf(0.0f, fmaxf(l.y - qh.y, ql.y - h.y));
                const float dz = fmaxf(0.0f, fmaxf(l.z - qh.z, ql.z - h.z));
                in = !((dx * dx + dy * dy + dz * dz) * (1.0f - 1e-6f) > u2);
            }
            const unsigned bal = __ballot_sync(0xffffffffu, in);
            if (lane == w) mine = bal;
        }
        if (__reduce_add_sync(0xffffffffu, __popc(mine)) > NN_MANY &&
            worth_asking(k0, words, mine)) {
            // (in the first chunk, where no other warp looks at this one's slice of
            // the tile)
            if (!seeded && k0 == b_lo) {
                seed_each();
                th = bound();
                seeded = true;
            }
            for (int w = 0; w < words; ++w) {
                const int64_t k = k0 + 32 * w + lane;
                bool in = (__shfl_sync(0xffffffffu, mine, w) >> lane) & 1u;
                if (!__any_sync(0xffffffffu, in)) continue;
                float4 l = make_float4(0.0f, 0.0f, 0.0f, 0.0f), h = l;
                if (in) {
                    l = boxes[2 * k];
                    h = boxes[2 * k + 1];
                }
                bool any = false;
                for (int j = 0; j < 32 / NN_SPLIT; ++j) {
                    const float px = __shfl_sync(0xffffffffu, fx, NN_SPLIT * j);
                    const float py = __shfl_sync(0xffffffffu, fy, NN_SPLIT * j);
                    const float pz = __shfl_sync(0xffffffffu, fz, NN_SPLIT * j);
                    const float pt = __shfl_sync(0xffffffffu, active ? th : -1.0f, NN_SPLIT * j);
                    const float dx = fmaxf(0.0f, fmaxf(l.x - above(px), below(px) - h.x));
                    const float dy = fmaxf(0.0f, fmaxf(l.y - above(py), below(py) - h.y));
                    const float dz = fmaxf(0.0f, fmaxf(l.z - above(pz), below(pz) - h.z));
                    any |= !((dx * dx + dy * dy + dz * dz) * (1.0f - 1e-6f) > pt) && !(pt < 0.0f);
                }
                const unsigned bal = __ballot_sync(0xffffffffu, in && any);
                if (lane == w) mine = bal;
            }
        }
        __syncthreads();  // everyone is done with the list, the masks and the tile
        if (lane < WORDS) mask[warp][lane] = mine;
        __syncthreads();
        unsigned any = 0u;  // word `warp` of the union
        for (int w = 0; w < WARPS; ++w) any |= mask[w][warp];
        if (lane == 0) s_cnt[warp] = __popc(any);
        __syncthreads();
        int before = 0, total = 0;
        for (int w = 0; w < WARPS; ++w) {
            if (w < warp) before += s_cnt[w];
            total += s_cnt[w];
        }
        if ((any >> lane) & 1u) list[before + __popc(any & ((1u << lane) - 1u))] = tid;
        __syncthreads();
        return total;
    };
    // which of the cnt staged boxes list[j], ... this warp kept
    auto mine_of = [&](int j, int cnt) {
        const int r = lane < cnt ? list[j + lane] : 0;
        return __ballot_sync(0xffffffffu, lane < cnt && ((mask[warp][r >> 5] >> (r & 31)) & 1u));
    };

    if (b_hi > b_lo) {
        stage(seed);
        __syncwarp();
        scan(warp);
    }
    float th = bound();
    const bool one_chunk = b_hi - b_lo <= NN_THREADS;
    int kept = 0;
    for (int64_t k0 = b_lo; k0 < b_hi; k0 += NN_THREADS) {
        kept = keep(k0, th);
        for (int j = 0; j < kept; j += NN_BOXES) {
            if (j) __syncthreads();  // the previous boxes are scanned
            const int cnt = min(NN_BOXES, kept - j);
            if (warp < cnt) stage(k0 + list[j + warp]);
            __syncthreads();
            const unsigned todo = mine_of(j, cnt);
            if (todo == (1u << cnt) - 1u) {
                scan_all(cnt);
            } else {
                for (unsigned m = todo; m; m &= m - 1) scan(__ffs(m) - 1);
            }
        }
        if (!one_chunk) th = bound();
    }
    __syncthreads();  // s_cmax is final
    th = bound();

    double best64 = __longlong_as_double(0x7ff0000000000000LL);
    int64_t arg = -1;
    // (the candidates do not come in ascending order: the lowest index of equal ones)
    auto try64 = [&](int64_t n) {
        const D4 p = x[n];
        double ex = __dsub_rn(p.x, qx), ey = __dsub_rn(p.y, qy), ez = __dsub_rn(p.z, qz);
        double s = __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez));
        if (s < best64 || (s == best64 && n < arg)) {
            best64 = s;
            arg = n;
        }
    };
    // this lane's candidates: how many, and the first four (from n_lo on); more, of
    // force points at nearly the same distance, are decided at once
    int found = 0;
    int32_t cand[4] = {0, 0, 0, 0};
    auto decide = [&](int slot, int64_t k) {
        if (active) {
            unsigned near = 0u;
#pragma unroll
            for (int u = 0; u < NN_BOX / NN_SPLIT; ++u) {
                const float4 v = tile[slot * NN_BOX + sub + NN_SPLIT * u];
                const float dx = v.x - fx, dy = v.y - fy, dz = v.z - fz;
                if (dx * dx + dy * dy + dz * dz <= th) near |= 1u << u;
            }
            for (; near; near &= near - 1u) {
                const int32_t n = (int32_t)(k * NN_BOX + sub + NN_SPLIT * (__ffs(near) - 1) - n_lo);
                if (found == 0) cand[0] = n;
                if (found == 1) cand[1] = n;
                if (found == 2) cand[2] = n;
                if (found == 3) cand[3] = n;
                if (found > 3) try64(n_lo + n);
                ++found;
            }
        }
    };
    if (one_chunk && kept <= NN_BOXES) {
        // the tile still holds them all
        for (unsigned m = mine_of(0, kept); m; m &= m - 1) {
            const int s = __ffs(m) - 1;
            decide(s, b_lo + list[s]);
        }
    } else {
        seeded = true;  // every distance is known: th stays
        for (int64_t k0 = b_lo; k0 < b_hi; k0 += NN_THREADS) {
            kept = keep(k0, th);
            for (int j = 0; j < kept; j += NN_BOXES) {
                if (j) __syncthreads();
                const int cnt = min(NN_BOXES, kept - j);
                if (warp < cnt) stage(k0 + list[j + warp]);
                __syncthreads();
                for (unsigned m = mine_of(j, cnt); m; m &= m - 1) {
                    const int s = __ffs(m) - 1;
                    decide(s, k0 + list[j + s]);
                }
            }
        }
    }
    // One candidate in all, at a finite distance, is the neighbour; more are
    // decided in FP64 (76 clocks of the pipe an operation: only then).
    int total = found;
#pragma unroll
    for (int o = 1; o < NN_SPLIT; o <<= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
    if (total == 1 && best < inf) {
        if (found) {
            arg = n_lo + cand[0];
            best64 = 0.0;
        }
    } else {
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (c < found) try64(n_lo + cand[c]);
    }
#pragma unroll
    for (int o = 1; o < NN_SPLIT; o <<= 1) {
        const double os = __shfl_xor_sync(0xffffffffu, best64, o);
        const int64_t oa = __shfl_xor_sync(0xffffffffu, arg, o);
        if (oa >= 0 && (arg < 0 || os < best64 || (os == best64 && oa < arg))) {
            best64 = os;
            arg = oa;
        }
    }
    if (active && sub == 0) {
        nn[q] = (int32_t)arg;  // -1 only when no distance was finite (NaN/Inf input)
        if (arg < 0) atomicOr(status, ST_NONFINITE);
    }
}

void launch_nearest(Ctx &c, const D4 *x, const D4 *Xw, int32_t *nn, bool only_deforming)
{
    const NNTask *tasks = only_deforming ? c.d_tasks_deform : c.d_tasks_all;
    int count = only_deforming ? c.n_tasks_deform : c.n_tasks_all;
    if (count == 0) return;
    c.tbeg(PH_NEAREST);
    k_nn_boxes<<<(unsigned)ceil_div(c.N, 256), 256, 0, c.stream>>>(c.N, x, c.d_nn_box);
    k_nearest<<<count, NN_THREADS, 0, c.stream>>>(tasks, c.d_n_off, c.nbodies, c.nn_global, x, Xw,
                                                   c.d_nn_box, nn, c.d_status);
    c.tend(PH_NEAREST);
    c.launches += 2;
}

// ---------------------------------------------------------------------------
// segments of nu: stable counting sort of q by n-hat(q)
// ---------------------------------------------------------------------------

// Quadrature points without a valid nearest force point (non-finite input,
// flagged by k_nearest) are left out of every segment.
__global__ void k_count(int64_t Q, int64_t N, const int32_t *__restrict__ nn,
                        int32_t *__restrict__ cnt)
{
    int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q < Q) {
        const int32_t k = nn[q];
        if (k >= 0 && k < N) atomicAdd(&cnt[k], 1);
    }
}

// Exclusive scan of cnt[0..N) into seg_ptr[0..N] and cursor[0..N] (one block of
// 1024 threads; cnt may alias cursor).  A warp takes 256 consecutive counts as
// 8 rows of 32, so that every access is coalesced.
__global__ void __launch_bounds__(1024)
    k_scan(int64_t N, const int32_t *cnt, int32_t *__restrict__ seg_ptr, int32_t *cursor)
{
    __shared__ int32_t part[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int32_t run = 0;  // sum of the tiles before
    for (int64_t base = 0; base < N; base += 8192) {
        const int64_t i0 = base + 256 * warp + lane;
        int32_t v[8], inc[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) inc[r] = v[r] = i0 + 32 * r < N ? cnt[i0 + 32 * r] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1)
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int32_t u = __shfl_up_sync(0xffffffffu, inc[r], o);
                if (lane >= o) inc[r] += u;
            }
        int32_t sum = 0;  // of the warp's rows before
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int32_t t = __shfl_sync(0xffffffffu, inc[r], 31);
            inc[r] += sum - v[r];
            sum += t;
        }
        if (lane == 31) part[warp] = sum;
        __syncthreads();
        int32_t w = part[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t u = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += u;
        }
        const int32_t before = __shfl_sync(0xffffffffu, w, max(warp - 1, 0));
        const int32_t at = run + (warp ? before : 0);
#pragma unroll
        for (int r = 0; r < 8; ++r)
            if (i0 + 32 * r < N) {
                seg_ptr[i0 + 32 * r] = at + inc[r];
                cursor[i0 + 32 * r] = at + inc[r];
            }
        run += __shfl_sync(0xffffffffu, w, 31);
        __syncthreads();  // part is free for the next tile
    }
    if (tid == 0) {
        seg_ptr[N] = run;
        cursor[N] = run;
    }
}

__global__ void k_scatter(int64_t Q, int64_t N, const int32_t *__restrict__ nn,
                          int32_t *__restrict__ cursor, int32_t *__restrict__ perm)
{
    int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q < Q) {
        const int32_t k = nn[q];
        if (k < 0 || k >= N) return;
        int32_t pos = atomicAdd(&cursor[k], 1);
        perm[pos] = (int32_t)q;
    }
}

// Order each segment by ascending q.  Segments hold about Q / N points: a warp
// ranks up to 32 (each lane counts the smaller values by shuffles; one thread
// per segment with an insertion sort in global memory took 24 us for 9200
// segments), its first lane sorts a longer one by insertion.
__global__ void k_sort_segments(int64_t N, const int32_t *__restrict__ seg_ptr,
                                int32_t *__restrict__ perm)
{
    const int64_t n = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32;
    if (n >= N) return;
    const int lane = threadIdx.x & 31;
    const int32_t lo = seg_ptr[n], hi = seg_ptr[n + 1], len = hi - lo;
    if (len <= 32) {
        const int32_t v = lane < len ? perm[lo + lane] : 0;
        int rank = 0;
        for (int k = 0; k < len; ++k) rank += __shfl_sync(0xffffffffu, v, k) < v;
        if (lane < len) perm[lo + rank] = v;
        return;
    }
    if (lane) return;
    for (int32_t i = lo + 1; i < hi; ++i) {
        int32_t v = perm[i];
        int32_t j = i - 1;
        while (j >= lo && perm[j] > v) {
            perm[j + 1] = perm[j];
            --j;
        }
        perm[j + 1] = v;
    }
}

void launch_segments(Ctx &c, const int32_t *nn, int32_t *seg_ptr, int32_t *perm)
{
    join_assembly(c);  // an assembly still on the side stream reads seg_ptr
    int threads = 256;
    c.tbeg(PH_SEGMENTS);
    cudaMemsetAsync(c.d_cursor, 0, sizeof(int32_t) * (c.N + 1), c.stream);
    cudaMemsetAsync(perm, 0, sizeof(int32_t) * c.Q, c.stream);  // tail stays a valid index
    k_count<<<(unsigned)ceil_div(c.Q, threads), threads, 0, c.stream>>>(c.Q, c.N, nn, c.d_cursor);
    // the counts are read from d_cursor, scanned into seg_ptr and back into d_cursor
    k_scan<<<1, 1024, 0, c.stream>>>(c.N, c.d_cursor, seg_ptr, c.d_cursor);
    k_scatter<<<(unsigned)ceil_div(c.Q, threads), threads, 0, c.stream>>>(c.Q, c.N, nn, c.d_cursor,
                                                                          perm);
    k_sort_segments<<<(unsigned)ceil_div(32 * c.N, threads), threads, 0, c.stream>>>(c.N, seg_ptr,
                                                                                      perm);
    c.tend(PH_SEGMENTS);
    c.launches += 4;
}

// Lab-frame quadrature points in segment order, and per-segment moments
// W_n = sum w_q, R_n = sum w_q (X_q - x0_b) accumulated in ascending q: one
// thread per segment gathers its points and sums them.  Quadrature points
// left out of every segment (no valid nearest force point) are not gathered.
__global__ void k_gather_moments(int64_t N, const int32_t *__restrict__ seg_ptr,
                                 const int32_t *__restrict__ perm, const D4 *__restrict__ Xw,
                                 D4 *__restrict__ Xs, const int32_t *__restrict__ body_x,
                                 const double *__restrict__ x0, double *__restrict__ W,
                                 double *__restrict__ R)
{
    int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const double *o = x0 + 3 * body_x[n];
    double w_sum = 0.0, r0 = 0.0, r1 = 0.0, r2 = 0.0;
    for (int32_t p = seg_ptr[n]; p < seg_ptr[n + 1]; ++p) {
        const D4 X = Xw[perm[p]];
        Xs[p] = X;
        w_sum = __dadd_rn(w_sum, X.w);
        r0 = __dadd_rn(r0, __dmul_rn(X.w, __dsub_rn(X.x, o[0])));
        r1 = __dadd_rn(r1, __dmul_rn(X.w, __dsub_rn(X.y, o[1])));
        r2 = __dadd_rn(r2, __dmul_rn(X.w, __dsub_rn(X.z, o[2])));
    }
    W[n] = w_sum;
    R[3 * n + 0] = r0;
    R[3 * n + 1] = r1;
    R[3 * n + 2] = r2;
}

void launch_gather(Ctx &c, const D4 *Xw_lab, const int32_t *seg_ptr, const int32_t *perm)
{
    join_assembly(c);  // and the gathered points
    int threads = 128;
    c.tbeg(PH_SEGMENTS);
    k_gather_moments<<<(unsigned)ceil_div(c.N, threads), threads, 0, c.stream>>>(
        c.N, seg_ptr, perm, Xw_lab, c.d_Xs, c.d_body_x, c.d_x0, c.d_W, c.d_R);
    c.tend(PH_SEGMENTS);
    c.launches += 1;
}

// ---------------------------------------------------------------------------
// rigid-body border (Sec. 4: unknown U, Omega; force and moment balance)
// ---------------------------------------------------------------------------

__device__ __forceinline__ double cross_entry(const double v[3], int j, int k)
{
    // [v]x = [[0,-v2,v1],[v2,0,-v0],[-v1,v0,0]]
    if (j == k) return 0.0;
    if (j == 0) return k == 1 ? -v[2] : v[1];
    if (j == 1) return k == 0 ? v[2] : -v[0];
    return k == 0 ? -v[1] : v[0];
}

__global__ void k_border(int64_t N, int64_t n, const int32_t *__restrict__ free_body,
                         const int32_t *__restrict__ body_x, const D4 *__restrict__ x,
                         const double *__restrict__ x0, const double *__restrict__ W,
                         const double *__restrict__ R, double *__restrict__ A64,
                         float *__restrict__ A32, float2 *__restrict__ Adf, int64_t lda)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int c = blockIdx.y;  // border unknown / row 0 .. 6F-1
    const int f = c / 6, cc = c % 6;
    const int bd = free_body[f];
    const int64_t base = 3 * N + 6 * (int64_t)f;
    double col = 0.0, row = 0.0;
    if (i < 3 * N) {
        const int64_t m = i / 3;
        const int jk = (int)(i % 3);
        if (body_x[m] == bd) {
            if (cc < 3) {
                col = (jk == cc) ? -1.0 : 0.0;
                row = (jk == cc) ? W[m] : 0.0;
            } else {
                D4 p = x[m];
                double r[3] = {__dsub_rn(p.x, x0[3 * bd + 0]), __dsub_rn(p.y, x0[3 * bd + 1]),
                               __dsub_rn(p.z, x0[3 * bd + 2])};
                col = cross_entry(r, jk, cc - 3);
                double Rm[3] = {R[3 * m + 0], R[3 * m + 1], R[3 * m + 2]};
                row = cross_entry(Rm, cc - 3, jk);
            }
        }
    }
    A64[i + (base + cc) * lda] = col;
    A64[(base + cc) + i * lda] = row;
    if (A32) {
        A32[i + (base + cc) * lda] = (float)col;
        A32[(base + cc) + i * lda] = (float)row;
    }
    if (Adf) {
        Adf[i + (base + cc) * lda] = df_split(col);
        Adf[(base + cc) + i * lda] = df_split(row);
    }
}

void launch_border(Ctx &c, const D4 *x_lab, double *A64, float *A32, int64_t lda)
{
    if (c.F == 0) return;
    int threads = 256;
    dim3 grid((unsigned)ceil_div(c.n, threads), (unsigned)(6 * c.F));
    // d_free_index holds nbodies entries (body -> free index) then F entries (free index -> body)
    c.tbeg(PH_BORDER);
    k_border<<<grid, threads, 0, c.stream>>>(c.N, c.n, c.d_free_index + c.nbodies, c.d_body_x, x_lab,
                                             c.d_x0, c.d_W, c.d_R, A64, A32,
                                             (c.arnoldi_df && A64 == c.d_A64) ? c.d_Adf : nullptr,
                                             lda);
    c.tend(PH_BORDER);
    c.launches += 1;
}

// ---------------------------------------------------------------------------
// explicit midpoint update of Y = [X0; B] (Sec. 4), B by modified Gram-Schmidt
// ---------------------------------------------------------------------------

__global__ void k_rk2(int stage, double dt, int nbodies, int64_t N,
                      const int32_t *__restrict__ kind, const int32_t *__restrict__ free_index,
                      const double *__restrict__ sol, const double *__restrict__ U,
                      const double *__restrict__ Om, const double *__restrict__ x0_save,
                      const double *__restrict__ B_save, double *__restrict__ x0,
                      double *__restrict__ B)
{
    int bd = blockIdx.x * blockDim.x + threadIdx.x;
    if (bd >= nbodies) return;
    int kd = kind[bd];
    if (kd == NRS_STATIC) return;
    double u[3], w[3];
    if (kd == NRS_FREE) {
        const double *v = sol + 3 * N + 6 * (int64_t)free_index[bd];
        for (int k = 0; k < 3; ++k) {
            u[k] = v[k];
            w[k] = v[3 + k];
        }
    } else {
        for (int k = 0; k < 3; ++k) {
            u[k] = U[3 * bd + k];
            w[k] = Om[3 * bd + k];
        }
    }
    const double h = stage == 0 ? 0.5 * dt : dt;
    double Bc[9], Bn[9];
    for (int k = 0; k < 9; ++k) Bc[k] = B[9 * bd + k];
    // dB = [w]x Bc ; Bn = B_save + h dB
    for (int r = 0; r < 3; ++r)
        for (int col = 0; col < 3; ++col) {
            double d = 0.0;
            for (int k = 0; k < 3; ++k) {
                double wx = (r == k) ? 0.0
                            : (r == 0) ? (k == 1 ? -w[2] : w[1])
                            : (r == 1) ? (k == 0 ? w[2] : -w[0])
                                       : (k == 0 ? -w[1] : w[0]);
                d += wx * Bc[3 * k + col];
            }
            Bn[3 * r + col] = B_save[9 * bd + 3 * r + col] + h * d;
        }
    for (int k = 0; k < 3; ++k) x0[3 * bd + k] = x0_save[3 * bd + k] + h * u[k];
    // modified Gram-Schmidt on the columns
    for (int j = 0; j < 3; ++j) {
        for (int i = 0; i < j; ++i) {
            double dot = Bn[i] * Bn[j] + Bn[3 + i] * Bn[3 + j] + Bn[6 + i] * Bn[6 + j];
            for (int r = 0; r < 3; ++r) Bn[3 * r + j] -= dot * Bn[3 * r + i];
        }
        double nrm = sqrt(Bn[j] * Bn[j] + Bn[3 + j] * Bn[3 + j] + Bn[6 + j] * Bn[6 + j]);
        for (int r = 0; r < 3; ++r) Bn[3 * r + j] /= nrm;
    }
    for (int k = 0; k < 9; ++k) B[9 * bd + k] = Bn[k];
}

void launch_rk2(Ctx &c, int stage, double dt, const double *sol)
{
    c.tbeg(PH_UPDATE);
    k_rk2<<<(unsigned)ceil_div(c.nbodies, 64), 64, 0, c.stream>>>(
        stage, dt, c.nbodies, c.N, c.d_kind, c.d_free_index, sol, c.d_U, c.d_Om, c.d_x0_save,
        c.d_B_save, c.d_x0, c.d_B);
    c.tend(PH_UPDATE);
    c.launches += 1;
}

}  // namespace nrs
