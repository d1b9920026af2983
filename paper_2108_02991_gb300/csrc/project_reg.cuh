// Per-shot projection with the FISTA state in registers (fixed iterations):
// device code of the kernels in project.cu.  Same iteration as
// project_dev.cuh, arranged so that a sample costs ~63 FP64 operations
// instead of ~100, and written over a number type R:
//
//   double  FP64 samples;
//   Df      FP32 samples: every value is an unevaluated sum of two floats
//           (hi + lo, ~48 bits).  On GB300 the FP64 pipe runs at 1/64 of the
//           FP32 rate, so ~500 FP32 operations take a ninth of the time of
//           those FP64 operations; the FP32 output keeps only the first 24
//           of the 48 bits.
//
// Arrangement.  Duals are kept divided by tau (Y = y / tau), so the radii are
// alpha and beta and Z = Y + D s needs no product.  With
//   p[m]  = Y1[m] + Y2[m-1] - Y2[m]
//   s[m]  = pin(clip(k[m] - tau (p[m-1] - p[m])))      (= k - tau D^T Y)
// (FP64: the differences of Y1 and of e[m] = Y2[m-1] - Y2[m] apart, which are
// exact where neighbours are close: rounding p costs half as much again in the
// result's error),
//   d[m]  = s[m+1] - s[m]
//   Z1[m] = Y1[m] + d[m],   Z2[m] = Y2[m] + (d[m+1] - d[m])
// every difference is formed once.  The extrapolation
//   Y+ = q+ + mom (q+ - q),  q+ = f Z,  f = max(0, 1 - radius / |Z|)
// takes mom from a table: it is the same for every row and call (a square
// root and a division in FP64 per thread and iteration otherwise).
//
// A thread owns M consecutive samples; neighbours exchange duals to the right
// and (s, d) to the left by shuffles, across warps through one slot a
// warp in shared memory -- across the CTAs of a cluster through distributed
// shared memory -- with two barriers an iteration.
//
// Bound: FP32 issue (two floats; 594 instructions a sample and iteration, 81 %
// of the issue slots at 512 samples a shot) or the FP64 pipe.  Measured, 100
// iterations, form with its state in memory -> this one: 4096 x 2560 FP32
// samples 192.9 -> 24.5 ms, 64 x 1024 3.15 -> 0.24 ms, 32 x 64 ~0.5 ms -> 86 us;
// 127 x 2047 FP64 samples (200 iterations) 11.65 -> 7.7 ms.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>
#include <type_traits>

#include "kernels.h"
#include "ptx.cuh"

namespace sparkling {
namespace {

// ---- two-float numbers ------------------------------------------------------

// hi + lo.  Sums and products below round the exact result to ~2^-48 of the
// largest operand; explicit _rn operations, so that no product is contracted
// into a sum whose rounding error is formed from its rounded value.
struct Df {
    float h, l;
};

__device__ __forceinline__ Df df_two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}

// |a| >= |b| (or a = 0)
__device__ __forceinline__ Df df_renorm(float a, float b)
{
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

// a +- b without the final renormalisation (an operand of one more sum)
__device__ __forceinline__ Df r_add_raw(Df a, Df b)
{
    const Df s = df_two_sum(a.h, b.h);
    return {s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l))};
}
__device__ __forceinline__ Df r_neg(Df a) { return {-a.h, -a.l}; }
// the sign bit alone (a subtraction would take the FP64 pipe)
__device__ __forceinline__ double r_neg(double a)
{
    return __longlong_as_double(__double_as_longlong(a) ^ (long long)0x8000000000000000ULL);
}
__device__ __forceinline__ Df r_sub_raw(Df a, Df b) { return r_add_raw(a, r_neg(b)); }
__device__ __forceinline__ Df r_norm(Df a) { return df_renorm(a.h, a.l); }
__device__ __forceinline__ Df r_add(Df a, Df b) { return r_norm(r_add_raw(a, b)); }
__device__ __forceinline__ Df r_mul_raw(Df a, Df b)
{
    const float p = __fmul_rn(a.h, b.h);
    return {p, fmaf(a.h, b.h, -p) + fmaf(a.h, b.l, a.l * b.h)};
}
__device__ __forceinline__ Df r_mul(Df a, Df b) { return r_norm(r_mul_raw(a, b)); }
// a * b - c
__device__ __forceinline__ Df r_mulsub(Df a, Df b, Df c)
{
    const Df p = r_mul_raw(a, b);
    const Df s = df_two_sum(p.h, -c.h);
    return df_renorm(s.h, __fadd_rn(s.l, __fsub_rn(p.l, c.l)));
}
// c - a * b
__device__ __forceinline__ Df r_submul(Df c, Df a, Df b)
{
    const Df p = r_mul_raw(a, b);
    const Df s = df_two_sum(c.h, -p.h);
    return df_renorm(s.h, __fadd_rn(s.l, __fsub_rn(c.l, p.l)));
}

__device__ __forceinline__ double r_add_raw(double a, double b) { return a + b; }
__device__ __forceinline__ double r_sub_raw(double a, double b) { return a - b; }
__device__ __forceinline__ double r_add(double a, double b) { return a + b; }
__device__ __forceinline__ double r_mul(double a, double b) { return a * b; }
__device__ __forceinline__ double r_mulsub(double a, double b, double c) { return fma(a, b, -c); }
__device__ __forceinline__ double r_submul(double c, double a, double b) { return fma(-a, b, c); }

template <class R> __device__ __forceinline__ R r_from(double v);
template <> __device__ __forceinline__ double r_from<double>(double v) { return v; }
template <> __device__ __forceinline__ Df r_from<Df>(double v)
{
    const float h = (float)v;
    return {h, (float)(v - (double)h)};
}

__device__ __forceinline__ double r_value(double v) { return v; }
__device__ __forceinline__ float r_value(Df v) { return v.h; }   // normalised: the nearest float

template <class R> __device__ __forceinline__ R r_zero();
template <> __device__ __forceinline__ double r_zero<double>() { return 0.0; }
template <> __device__ __forceinline__ Df r_zero<Df>() { return {0.f, 0.f}; }

__device__ __forceinline__ double r_shfl_up(double v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ double r_shfl_down(double v) { return __shfl_down_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ Df r_shfl_up(Df v)
{
    return {__shfl_up_sync(0xffffffffu, v.h, 1), __shfl_up_sync(0xffffffffu, v.l, 1)};
}
__device__ __forceinline__ Df r_shfl_down(Df v)
{
    return {__shfl_down_sync(0xffffffffu, v.h, 1), __shfl_down_sync(0xffffffffu, v.l, 1)};
}

// Clip to [-box, box]; NaN passes.
__device__ __forceinline__ double r_clip(double v, double box)
{
    return v > box ? box : (v < -box ? -box : v);
}
__device__ __forceinline__ Df r_clip(Df v, Df box)
{
    const bool hi = v.h > box.h || (v.h == box.h && v.l > box.l);
    const bool lo = v.h < -box.h || (v.h == -box.h && v.l < -box.l);
    return hi ? box : (lo ? r_neg(box) : v);
}
// Whether a component may lie outside the box (never false when one does): on
// the leading words, off the FP64 pipe.
__device__ __forceinline__ bool r_near(const double *v, double box)
{
    const int m = max(max(__double2hiint(v[0]) & 0x7fffffff, __double2hiint(v[1]) & 0x7fffffff),
                      __double2hiint(v[2]) & 0x7fffffff);
    return m >= __double2hiint(box);
}
__device__ __forceinline__ bool r_near(const Df *v, Df box)
{
    return fmaxf(fmaxf(fabsf(v[0].h), fabsf(v[1].h)), fabsf(v[2].h)) >= box.h;
}

// Update of one row: q+ = f z with f = max(0, 1 - r / |z|) (0 for a row that
// does not exist), extrapolated with the previous iteration's q.  1/|z| is the
// hardware estimate and one step of Halley's method for x^-1/2 (third order:
// x (1 + e/2 + 3 e^2/8), e = 1 - zz x^2).
//
// FP64: q itself is kept, Y+ = q+ + mom (q+ - q).  A warp whose rows all lie
// inside the ball skips the factor (the FP64 pipe bounds this form).
__device__ __forceinline__ void r_update(const double *z, double r, double r2, const double2 m,
                                         bool exists, double *q, double *y)
{
    const double zz = fma(z[0], z[0], fma(z[1], z[1], z[2] * z[2]));
    double f = 0.0;
    // both non-negative: integer comparison (NaN compares above)
    const bool on = exists && __double_as_longlong(zz) > __double_as_longlong(r2);
    if (on) {
        double x;
        asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(zz));
        const double e = fma(-zz * x, x, 1.0);
        x = fma(x * e, fma(0.375, e, 0.5), x);
        f = fma(-r, x, 1.0);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double qn = on ? z[c] * f : 0.0;
        y[c] = fma(m.x, qn - q[c], qn);
        q[c] = qn;
    }
}

// Two floats: W = mom q is kept, Y+ = ((1 + mom) f) z - W and W+ = (mom+ f) z
// (q+ itself in the last iteration).  No branch: both rows of a sample and
// their long dependent chains run side by side.
__device__ __forceinline__ void r_update(const Df *z, Df r, float r2, const float4 m, bool exists,
                                         Df *w, Df *y)
{
    Df q[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float p = __fmul_rn(z[c].h, z[c].h);
        q[c] = {p, fmaf(z[c].h + z[c].h, z[c].l, fmaf(z[c].h, z[c].h, -p))};
    }
    const Df zz = r_add(r_add_raw(q[0], q[1]), q[2]);
    const float x = rsqrt_sfu(zz.h);
    // e = 1 - zz x^2 with x^2 as an exact pair
    const float t = __fmul_rn(x, x), tl = fmaf(x, x, -t);
    float e = fmaf(-zz.h, t, 1.f);
    e = fmaf(-zz.h, tl, fmaf(-zz.l, t, e));
    const Df g = r_mul_raw(r, Df{x, x * (e * fmaf(0.375f, e, 0.5f))});
    const Df s = df_renorm(1.f, -g.h);          // g <= 1 up to rounding
    Df f = df_renorm(s.h, __fsub_rn(s.l, g.l));
    // inside the ball (or no such row): 0; NaN goes on, and stays
    if (!exists || zz.h <= r2 || f.h < 0.f) f = {0.f, 0.f};
    const Df a = r_mul(f, Df{m.x, m.y}), b = r_mul(f, Df{m.z, m.w});
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        y[c] = r_mulsub(z[c], a, w[c]);
        w[c] = r_mul(z[c], b);
    }
}

// Momentum of an iteration: (mom_it, -) in FP64; (1 + mom_it, mom_{it+1}) as
// two-float sums, mom_{it+1} = 1 in the last one (W is then q+).
__device__ __forceinline__ double2 momentum_of(const MomentumTables &m, int it, bool, double)
{
    return __ldg(m.d + it);
}
__device__ __forceinline__ float4 momentum_of(const MomentumTables &m, int it, bool final, Df)
{
    float4 v = __ldg(m.f + it);
    if (final) { v.z = 1.f; v.w = 0.f; }
    return v;
}

// Squared radius as the type the comparison takes.
__device__ __forceinline__ double r_square(double r) { return r * r; }
__device__ __forceinline__ float r_square(Df r) { return r.h * r.h; }

// ---- the projection ---------------------------------------------------------

// One slot of the exchange across warps: of the sample left of a warp's first
// one Y2 and p (two floats) or Y2, e and Y1 (FP64); (s, d) of the sample right
// of its last one.
template <class R> struct EdgeSlot {
    R a[9], b[6];
};
constexpr int kSlotWords = 15;          // 8-byte words of a slot

struct RegShot {
    int Ns, n_iter, pin_index;
    double alpha, beta, box;
    double pin[3];
};

// Project one shot, all threads of the CTA (of the cluster's CTAs) calling.
// m0: first of the thread's M samples.  edge: the CTA's slots, one a warp;
// left_a / right_b: the neighbour slots this warp writes (its right
// neighbour's a, its left neighbour's b; null at the ends of the shot),
// possibly in another CTA of the cluster.  first / last: no warp on that
// side; the slots nobody writes are zero.  loadk(m, kv) gives the FP64 input; store(m, s) takes the result.
// refresh(it, y1, y2, w1, w2) may replace the state after iteration it (-1:
// once the input is loaded).
template <class R, int M, class Sync, class Refresh, class LoadK, class Store>
__device__ __forceinline__ void project_registers(const RegShot &p, const MomentumTables &mom, int m0,
                                                  EdgeSlot<R> *mine,
                                                  EdgeSlot<R> *to_right, EdgeSlot<R> *to_left,
                                                  bool first, bool last, Sync sync, Refresh refresh,
                                                  LoadK loadk, Store store)
{
    constexpr bool kTwoFloat = std::is_same<R, Df>::value;
    const int lane = threadIdx.x & 31;
    const R tau = r_from<R>(1.0 / 20.0);
    const R alpha = r_from<R>(p.alpha), beta = r_from<R>(p.beta), box = r_from<R>(p.box);
    const auto a2 = r_square(alpha);
    const auto b2 = r_square(beta);
    R y1[M][3], y2[M][3], w1[M][3], w2[M][3], k[M][3], s[M][3];   // w: W, or q in FP64
#pragma unroll
    for (int j = 0; j < M; ++j) {
        double kv[3] = {0.0, 0.0, 0.0};
        if (m0 + j < p.Ns) loadk(m0 + j, kv);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            // a pinned sample's k is never read: it holds the pin.  Beyond any
            // dual term the clip decides: keep the sums finite.
            double v = m0 + j == p.pin_index ? p.pin[c] : kv[c];
            if (kTwoFloat) {
                v = v > kDfHuge ? kDfHuge : v;
                v = v < -kDfHuge ? -kDfHuge : v;
            }
            k[j][c] = r_from<R>(v);
            y1[j][c] = y2[j][c] = w1[j][c] = w2[j][c] = r_zero<R>();
        }
    }
    refresh(-1, y1, y2, w1, w2);
    const bool pinned = p.pin_index >= m0 && p.pin_index < m0 + M;
    for (int it = 0;; ++it) {
        // s from (Y1, Y2): dp[j] = D^T Y of the thread's samples
        R dp[M][3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            R yl = r_shfl_up(y2[M - 1][c]);
            if constexpr (kTwoFloat) {
                R pp[M];
#pragma unroll
                for (int j = 1; j < M; ++j)
                    pp[j] = r_add_raw(y1[j][c], r_sub_raw(y2[j - 1][c], y2[j][c]));
                if (M == 1) pp[0] = r_add_raw(y1[0][c], r_sub_raw(yl, y2[0][c]));
                if (lane == 31 && !last) {
                    to_right->a[c] = y2[M - 1][c];
                    to_right->a[3 + c] = pp[M - 1];
                }
#pragma unroll
                for (int j = 0; j < M; ++j) dp[j][c] = pp[j];
                if (M > 1) dp[0][c] = yl;
            } else {
                if (lane == 31 && !last) {
                    to_right->a[c] = y2[M - 1][c];
                    to_right->a[3 + c] = (M > 1 ? y2[M > 1 ? M - 2 : 0][c] : yl) - y2[M - 1][c];
                    to_right->a[6 + c] = y1[M - 1][c];
                }
                dp[0][c] = yl;
            }
        }
        sync();
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if constexpr (kTwoFloat) {
                R yl = M > 1 ? dp[0][c] : r_shfl_up(y2[0][c]);
                if (lane == 0) yl = mine->a[c];
                dp[0][c] = r_add_raw(y1[0][c], r_sub_raw(yl, y2[0][c]));
                R pl = r_shfl_up(dp[M - 1][c]);
                if (lane == 0) pl = mine->a[3 + c];
#pragma unroll
                for (int j = M - 1; j >= 0; --j)
                    dp[j][c] = r_sub_raw(j ? dp[j ? j - 1 : 0][c] : pl, dp[j][c]);
            } else {
                R yl = dp[0][c], y1l = r_shfl_up(y1[M - 1][c]), el[M + 1];
                if (lane == 0) {
                    yl = mine->a[c];
                    y1l = mine->a[6 + c];
                }
#pragma unroll
                for (int j = 0; j < M; ++j) el[j + 1] = (j ? y2[j ? j - 1 : 0][c] : yl) - y2[j][c];
                el[0] = r_shfl_up(el[M]);
                if (lane == 0) el[0] = mine->a[3 + c];
#pragma unroll
                for (int j = 0; j < M; ++j)
                    dp[j][c] = ((j ? y1[j ? j - 1 : 0][c] : y1l) - y1[j][c]) + (el[j] - el[j + 1]);
            }
        }
#pragma unroll
        for (int j = 0; j < M; ++j) {
#pragma unroll
            for (int c = 0; c < 3; ++c)
                s[j][c] = r_submul(k[j][c], tau, dp[j][c]);
            if (r_near(s[j], box) || pinned)
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    s[j][c] = m0 + j == p.pin_index ? k[j][c] : r_clip(s[j][c], box);
        }
        if (it == p.n_iter) break;
        // duals from s
        R sr[3], dr[3], d[M][3];
        const bool final = it + 1 == p.n_iter;
        const auto mo = momentum_of(mom, it, final, R());
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            sr[c] = r_shfl_down(s[0][c]);
#pragma unroll
            for (int j = 0; j + 1 < M; ++j) d[j][c] = r_sub_raw(s[j + 1][c], s[j][c]);
            if (M == 1) d[0][c] = r_sub_raw(sr[c], s[0][c]);
            if (lane == 0 && !first) {
                to_left->b[c] = s[0][c];
                to_left->b[3 + c] = d[0][c];
            }
        }
        sync();
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (lane == 31) sr[c] = mine->b[c];
            d[M - 1][c] = r_sub_raw(sr[c], s[M - 1][c]);
            dr[c] = r_shfl_down(d[0][c]);
            if (lane == 31) dr[c] = mine->b[3 + c];
        }
#pragma unroll
        for (int j = 0; j < M; ++j) {
            R z1[3], z2[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                z1[c] = r_add(y1[j][c], d[j][c]);
                z2[c] = r_add(y2[j][c], r_sub_raw(j + 1 < M ? d[j + 1][c] : dr[c], d[j][c]));
            }
            r_update(z1, alpha, a2, mo, m0 + j < p.Ns - 1, w1[j], y1[j]);
            r_update(z2, beta, b2, mo, m0 + j < p.Ns - 2, w2[j], y2[j]);
            if (final)            // the output is s(q), not s(Y)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    y1[j][c] = w1[j][c];
                    y2[j][c] = w2[j][c];
                }
        }
        if (!final) refresh(it, y1, y2, w1, w2);
    }
#pragma unroll
    for (int j = 0; j < M; ++j)
        if (m0 + j < p.Ns) store(m0 + j, s[j]);
}

} // namespace
} // namespace sparkling
