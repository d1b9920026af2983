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
// Bound: FP32 issue and the FMA pipe (two floats: ~500 lane operations a sample
// and iteration; x and y share paired instructions, 594 -> ~460 issued) or the
// FP64 pipe.  Measured, 100 iterations, form with its state in memory -> this
// one: 4096 x 2560 FP32 samples 192.9 -> 21.9 ms (25.0 without the pairing),
// 64 x 1024 3.15 -> 0.27 ms, 32 x 64 ~0.5 ms -> 78 us; 127 x 2047 FP64 samples (200
// iterations) 11.65 -> 7.6 ms.
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

__device__ __forceinline__ Df r_norm(Df a) { return df_renorm(a.h, a.l); }
__device__ __forceinline__ Df r_mul_raw(Df a, Df b)
{
    const float p = __fmul_rn(a.h, b.h);
    return {p, fmaf(a.h, b.h, -p) + fmaf(a.h, b.l, a.l * b.h)};
}
__device__ __forceinline__ Df r_mul(Df a, Df b) { return r_norm(r_mul_raw(a, b)); }

template <class R> __device__ __forceinline__ R r_from(double v);
template <> __device__ __forceinline__ double r_from<double>(double v) { return v; }
template <> __device__ __forceinline__ Df r_from<Df>(double v)
{
    const float h = (float)v;
    return {h, (float)(v - (double)h)};
}

// ---- vectors of three -------------------------------------------------------

// Two floats: x and y share 64-bit registers (paired FP32, one instruction for
// both), z stands alone.
struct VecDf {
    f2 h, l;
    float zh, zl;
};
struct VecD {
    double x, y, z;
};
template <class R> struct VecOf;
template <> struct VecOf<double> { typedef VecD type; };
template <> struct VecOf<Df> { typedef VecDf type; };

__device__ __forceinline__ VecD v_zero(double) { return {0.0, 0.0, 0.0}; }
__device__ __forceinline__ VecDf v_zero(Df)
{
    const f2 z = f2_pack(0.f, 0.f);
    return {z, z, 0.f, 0.f};
}
__device__ __forceinline__ VecD v_from(const double *v, double) { return {v[0], v[1], v[2]}; }
__device__ __forceinline__ VecDf v_from(const double *v, Df)
{
    const Df x = r_from<Df>(v[0]), y = r_from<Df>(v[1]), z = r_from<Df>(v[2]);
    return {f2_pack(x.h, y.h), f2_pack(x.l, y.l), z.h, z.l};
}
// The nearest value of the output's type (two floats: the sums are normalised).
__device__ __forceinline__ void v_values(const VecD &v, double *o) { o[0] = v.x; o[1] = v.y; o[2] = v.z; }
__device__ __forceinline__ void v_values(const VecDf &v, float *o)
{
    f2_unpack(v.h, o[0], o[1]);
    o[2] = v.zh;
}

__device__ __forceinline__ VecD v_add(const VecD &a, const VecD &b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ VecD v_sub(const VecD &a, const VecD &b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ VecD v_add_raw(const VecD &a, const VecD &b) { return v_add(a, b); }
__device__ __forceinline__ VecD v_sub_raw(const VecD &a, const VecD &b) { return v_sub(a, b); }
// c - a * b
__device__ __forceinline__ VecD v_submul(const VecD &c, double a, const VecD &b)
{
    return {fma(-a, b.x, c.x), fma(-a, b.y, c.y), fma(-a, b.z, c.z)};
}

// a +- b without the final renormalisation (an operand of one more sum)
__device__ __forceinline__ VecDf v_add_raw(const VecDf &a, const VecDf &b)
{
    VecDf r;
    r.h = f2_add(a.h, b.h);
    const f2 t = f2_sub(r.h, a.h);
    const f2 e = f2_add(f2_sub(a.h, f2_sub(r.h, t)), f2_sub(b.h, t));
    r.l = f2_add(e, f2_add(a.l, b.l));
    const Df z = df_two_sum(a.zh, b.zh);
    r.zh = z.h;
    r.zl = __fadd_rn(z.l, __fadd_rn(a.zl, b.zl));
    return r;
}
__device__ __forceinline__ VecDf v_sub_raw(const VecDf &a, const VecDf &b)
{
    VecDf r;
    r.h = f2_sub(a.h, b.h);
    const f2 t = f2_sub(r.h, a.h);
    const f2 e = f2_sub(f2_sub(a.h, f2_sub(r.h, t)), f2_add(b.h, t));
    r.l = f2_add(e, f2_sub(a.l, b.l));
    const Df z = df_two_sum(a.zh, -b.zh);
    r.zh = z.h;
    r.zl = __fadd_rn(z.l, __fsub_rn(a.zl, b.zl));
    return r;
}
__device__ __forceinline__ VecDf v_norm(const VecDf &a)
{
    VecDf r;
    r.h = f2_add(a.h, a.l);
    r.l = f2_sub(a.l, f2_sub(r.h, a.h));
    const Df z = df_renorm(a.zh, a.zl);
    r.zh = z.h;
    r.zl = z.l;
    return r;
}
__device__ __forceinline__ VecDf v_add(const VecDf &a, const VecDf &b) { return v_norm(v_add_raw(a, b)); }

// A two-float factor of vectors, spread over the pairs.
struct FactorDf {
    f2 h, nh, l;
    Df s;
    __device__ __forceinline__ FactorDf(Df f)
        : h(f2_pack(f.h, f.h)), nh(f2_pack(-f.h, -f.h)), l(f2_pack(f.l, f.l)), s(f) {}
};
__device__ __forceinline__ VecDf v_mul_raw(const VecDf &a, const FactorDf &f)
{
    VecDf r;
    r.h = f2_mul(a.h, f.h);
    const f2 ne = f2_fma(a.h, f.nh, r.h);        // minus the product's rounding error
    r.l = f2_sub(f2_fma(a.h, f.l, f2_mul(a.l, f.h)), ne);
    const Df z = r_mul_raw(Df{a.zh, a.zl}, f.s);
    r.zh = z.h;
    r.zl = z.l;
    return r;
}
__device__ __forceinline__ VecDf v_mul(const VecDf &a, const FactorDf &f) { return v_norm(v_mul_raw(a, f)); }
__device__ __forceinline__ VecDf v_submul(const VecDf &c, const FactorDf &f, const VecDf &b)
{
    return v_norm(v_sub_raw(c, v_mul_raw(b, f)));
}

__device__ __forceinline__ VecD v_shfl_up(const VecD &v)
{
    constexpr unsigned int kAll = 0xffffffffu;
    return {__shfl_up_sync(kAll, v.x, 1), __shfl_up_sync(kAll, v.y, 1), __shfl_up_sync(kAll, v.z, 1)};
}
__device__ __forceinline__ VecD v_shfl_down(const VecD &v)
{
    constexpr unsigned int kAll = 0xffffffffu;
    return {__shfl_down_sync(kAll, v.x, 1), __shfl_down_sync(kAll, v.y, 1), __shfl_down_sync(kAll, v.z, 1)};
}
__device__ __forceinline__ VecDf v_shfl_up(const VecDf &v)
{
    constexpr unsigned int kAll = 0xffffffffu;
    return {__shfl_up_sync(kAll, v.h, 1), __shfl_up_sync(kAll, v.l, 1), __shfl_up_sync(kAll, v.zh, 1),
            __shfl_up_sync(kAll, v.zl, 1)};
}
__device__ __forceinline__ VecDf v_shfl_down(const VecDf &v)
{
    constexpr unsigned int kAll = 0xffffffffu;
    return {__shfl_down_sync(kAll, v.h, 1), __shfl_down_sync(kAll, v.l, 1),
            __shfl_down_sync(kAll, v.zh, 1), __shfl_down_sync(kAll, v.zl, 1)};
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
    return hi ? box : (lo ? Df{-box.h, -box.l} : v);
}
__device__ __forceinline__ VecD v_clip(const VecD &v, double box)
{
    return {r_clip(v.x, box), r_clip(v.y, box), r_clip(v.z, box)};
}
__device__ __forceinline__ VecDf v_clip(const VecDf &v, Df box)
{
    float xh, yh, xl, yl;
    f2_unpack(v.h, xh, yh);
    f2_unpack(v.l, xl, yl);
    const Df x = r_clip(Df{xh, xl}, box), y = r_clip(Df{yh, yl}, box), z = r_clip(Df{v.zh, v.zl}, box);
    return {f2_pack(x.h, y.h), f2_pack(x.l, y.l), z.h, z.l};
}
// Whether a component may lie outside the box (never false when one does): on
// the leading words, off the FP64 pipe.
__device__ __forceinline__ bool v_near(const VecD &v, double box)
{
    const int m = max(max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff),
                      __double2hiint(v.z) & 0x7fffffff);
    return m >= __double2hiint(box);
}
__device__ __forceinline__ bool v_near(const VecDf &v, Df box)
{
    float x, y;
    f2_unpack(v.h, x, y);
    return fmaxf(fmaxf(fabsf(x), fabsf(y)), fabsf(v.zh)) >= box.h;
}

// Update of one row: q+ = f z with f = max(0, 1 - r / |z|) (0 for a row that
// does not exist), extrapolated with the previous iteration's q.  1/|z| is the
// hardware estimate and one step of Halley's method for x^-1/2 (third order:
// x (1 + e/2 + 3 e^2/8), e = 1 - zz x^2).
//
// FP64: q itself is kept, Y+ = q+ + mom (q+ - q).  A warp whose rows all lie
// inside the ball skips the factor (the FP64 pipe bounds this form).
// Where the square overflows 1/|z| is 0, and NaN stays in its component (zz is not
// subnormal: r2 is not).  Selections, not a branch (3 % of 37 x 129 samples): of the
// factor with two samples a thread, of the products with one, whose chain bounds it
// (37 x 129 293 us, selecting the factor 299; 127 x 2047 7.55 ms, factor 7.53).
template <int M>
__device__ __forceinline__ void r_update(const VecD &z, double r, double r2, const double2 m,
                                         bool exists, VecD &q, VecD &y)
{
    const double zz = fma(z.x, z.x, fma(z.y, z.y, z.z * z.z));
    double f = 0.0;
    // both non-negative: comparison as integers, unsigned (a NaN of either sign
    // compares above)
    const unsigned long long zb = (unsigned long long)__double_as_longlong(zz);
    const bool on = exists && zb > (unsigned long long)__double_as_longlong(r2);
    const unsigned int zh = (unsigned int)(zb >> 32);
    if (on) {
        double x;
        asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(zz));
        const double e = fma(-zz * x, x, 1.0);
        x = fma(x * e, fma(0.375, e, 0.5), x);
        f = fma(-r, x, 1.0);
        if (M > 1) f = zh >= 0x7ff00000u ? (zh == 0x7ff00000u ? 1.0 : 0.0) : f;
    }
    const bool odd = M == 1 && on && zh >= 0x7ff00000u;
    auto row = [&](double zc, double &qc, double &yc) {
        double qn = on ? zc * f : 0.0;
        if (M == 1) {
            const bool nan = (__double2hiint(zc) & 0x7fffffff) >= 0x7ff00000;
            qn = odd ? (zh == 0x7ff00000u || nan ? zc : 0.0) : qn;
        }
        yc = fma(m.x, qn - qc, qn);
        qc = qn;
    };
    row(z.x, q.x, y.x);
    row(z.y, q.y, y.y);
    row(z.z, q.z, y.z);
}

// Two floats: W = mom q is kept, Y+ = ((1 + mom) f) z - W and W+ = (mom+ f) z
// (q+ itself in the last iteration).  No branch: both rows of a sample and
// their long dependent chains run side by side.
template <int M>
__device__ __forceinline__ void r_update(const VecDf &z, Df r, float r2, const float4 m, bool exists,
                                         VecDf &w, VecDf &y)
{
    float xh, yh, xl, yl;
    f2_unpack(z.h, xh, yh);
    f2_unpack(z.l, xl, yl);
    auto square = [](float h, float l) -> Df {
        const float p = __fmul_rn(h, h);
        return {p, fmaf(h + h, l, fmaf(h, h, -p))};
    };
    const Df qx = square(xh, xl), qy = square(yh, yl), qz = square(z.zh, z.zl);
    const Df a0 = df_two_sum(qx.h, qy.h), a1 = df_two_sum(a0.h, qz.h);
    const Df zz = df_renorm(a1.h, __fadd_rn(__fadd_rn(a1.l, a0.l), __fadd_rn(__fadd_rn(qx.l, qy.l), qz.l)));
    const float x = rsqrt_sfu(zz.h);
    // e = 1 - zz x^2 with x^2 as an exact pair
    const float t = __fmul_rn(x, x), tl = fmaf(x, x, -t);
    float e = fmaf(-zz.h, t, 1.f);
    e = fmaf(-zz.h, tl, fmaf(-zz.l, t, e));
    const Df g = r_mul_raw(r, Df{x, x * (e * fmaf(0.375f, e, 0.5f))});
    const Df s = df_renorm(1.f, -g.h);          // g <= 1 up to rounding
    Df f = df_renorm(s.h, __fsub_rn(s.l, g.l));
    // inside the ball (or no such row): 0, and for NaN, which stays in its
    // component.  r2 lies a little below the radius squared: near it the sign of f
    // decides, on both words
    if (!exists || zz.h <= r2 || !(f.h >= 0.f)) f = {0.f, 0.f};
    const FactorDf a(r_mul(f, Df{m.x, m.y})), b(r_mul(f, Df{m.z, m.w}));
    y = v_norm(v_sub_raw(v_mul_raw(z, a), w));
    w = v_mul(z, b);
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

__device__ __forceinline__ double factor_of(double f) { return f; }
__device__ __forceinline__ FactorDf factor_of(Df f) { return FactorDf(f); }

// Squared radius as the type the comparison takes; two floats: the square of the
// leading word less 2^-20 of it, so that a row below it is inside for certain
// (infinity stays).
__device__ __forceinline__ double r_square(double r) { return r * r; }
__device__ __forceinline__ float r_square(Df r) { return r.h * r.h * (1.f - 1.f / (1 << 20)); }

// ---- the projection ---------------------------------------------------------

// One slot of the exchange across warps: of the sample left of a warp's first
// one Y2 and p (two floats) or Y2, e and Y1 (FP64); (s, d) of the sample right
// of its last one.
template <class R> struct EdgeSlot {
    typename VecOf<R>::type a[3], b[2];
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
// side; the slots nobody writes are zero.  loadk(m, kv) gives the FP64 input;
// store(m, s) takes the result.
// refresh(it, y1, y2, w1, w2) may replace the state after iteration it (-1:
// once the input is loaded).
template <class R, int M, class Sync, class Refresh, class LoadK, class Store>
__device__ __forceinline__ void project_registers(const RegShot &p, const MomentumTables &mom, int m0,
                                                  EdgeSlot<R> *mine,
                                                  EdgeSlot<R> *to_right, EdgeSlot<R> *to_left,
                                                  bool first, bool last, Sync sync, Refresh refresh,
                                                  LoadK loadk, Store store)
{
    typedef typename VecOf<R>::type V;
    constexpr bool kTwoFloat = std::is_same<R, Df>::value;
    constexpr int L = M - 1, L1 = M > 1 ? M - 2 : 0;       // the thread's last samples
    const int lane = threadIdx.x & 31;
    const auto tau = factor_of(r_from<R>(1.0 / 20.0));
    const R alpha = r_from<R>(p.alpha), beta = r_from<R>(p.beta), box = r_from<R>(p.box);
    const auto a2 = r_square(alpha);
    const auto b2 = r_square(beta);
    V y1[M], y2[M], w1[M], w2[M], k[M], s[M];              // w: W, or q in FP64
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
            kv[c] = v;
        }
        k[j] = v_from(kv, R());
        y1[j] = y2[j] = w1[j] = w2[j] = v_zero(R());
    }
    refresh(-1, y1, y2, w1, w2);
    const bool pinned = p.pin_index >= m0 && p.pin_index < m0 + M;
    for (int it = 0;; ++it) {
        // s from (Y1, Y2): dp[j] = D^T Y of the thread's samples
        V dp[M], yl = v_shfl_up(y2[L]);
        if constexpr (kTwoFloat) {
#pragma unroll
            for (int j = 1; j < M; ++j) dp[j] = v_add_raw(y1[j], v_sub_raw(y2[j - 1], y2[j]));
            if (M == 1) dp[0] = v_add_raw(y1[0], v_sub_raw(yl, y2[0]));
            if (lane == 31 && !last) {
                to_right->a[0] = y2[L];
                to_right->a[1] = dp[L];
            }
        } else if (lane == 31 && !last) {
            to_right->a[0] = y2[L];
            to_right->a[1] = v_sub(M > 1 ? y2[L1] : yl, y2[L]);
            to_right->a[2] = y1[L];
        }
        sync();
        if constexpr (kTwoFloat) {
            if (lane == 0) yl = mine->a[0];
            dp[0] = v_add_raw(y1[0], v_sub_raw(yl, y2[0]));
            V pl = v_shfl_up(dp[L]);
            if (lane == 0) pl = mine->a[1];
#pragma unroll
            for (int j = M - 1; j >= 0; --j) dp[j] = v_sub_raw(j ? dp[j ? j - 1 : 0] : pl, dp[j]);
        } else {
            V y1l = v_shfl_up(y1[L]), el[M + 1];
            if (lane == 0) {
                yl = mine->a[0];
                y1l = mine->a[2];
            }
#pragma unroll
            for (int j = 0; j < M; ++j) el[j + 1] = v_sub(j ? y2[j ? j - 1 : 0] : yl, y2[j]);
            el[0] = v_shfl_up(el[M]);
            if (lane == 0) el[0] = mine->a[1];
#pragma unroll
            for (int j = 0; j < M; ++j)
                dp[j] = v_add(v_sub(j ? y1[j ? j - 1 : 0] : y1l, y1[j]), v_sub(el[j], el[j + 1]));
        }
#pragma unroll
        for (int j = 0; j < M; ++j) {
            s[j] = v_submul(k[j], tau, dp[j]);
            if (v_near(s[j], box) || pinned) s[j] = m0 + j == p.pin_index ? k[j] : v_clip(s[j], box);
        }
        if (it == p.n_iter) break;
        // duals from s
        V sr = v_shfl_down(s[0]), dr, d[M];
        const bool final = it + 1 == p.n_iter;
        const auto mo = momentum_of(mom, it, final, R());
#pragma unroll
        for (int j = 0; j + 1 < M; ++j) d[j] = v_sub_raw(s[j + 1], s[j]);
        if (M == 1) d[0] = v_sub_raw(sr, s[0]);
        if (lane == 0 && !first) {
            to_left->b[0] = s[0];
            to_left->b[1] = d[0];
        }
        sync();
        if (lane == 31) sr = mine->b[0];
        d[L] = v_sub_raw(sr, s[L]);
        dr = v_shfl_down(d[0]);
        if (lane == 31) dr = mine->b[1];
#pragma unroll
        for (int j = 0; j < M; ++j) {
            const V z1 = v_add(y1[j], d[j]);
            const V z2 = v_add(y2[j], v_sub_raw(j + 1 < M ? d[j + 1 < M ? j + 1 : 0] : dr, d[j]));
            r_update<M>(z1, alpha, a2, mo, m0 + j < p.Ns - 1, w1[j], y1[j]);
            r_update<M>(z2, beta, b2, mo, m0 + j < p.Ns - 2, w2[j], y2[j]);
            if (final) {          // the output is s(q), not s(Y)
                y1[j] = w1[j];
                y2[j] = w2[j];
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
