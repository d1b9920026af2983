// Fast repulsion: particle-particle particle-mesh (P3M) summation of
// R_i = sum_{j != i} d_ij / |d_ij|_eps, the O(N^2) bottleneck of Sec. II-C.2
// (the paper takes a fast multipole method there; this is the GB300 path).
//
// The kernel splits exactly: d/r = d/r erfc(r/sigma) + d/r erf(r/sigma),
// r = |d|_eps.  The short-range part decays like a Gaussian and is summed
// directly over the pairs closer than rc, found through the bounding boxes of
// clusters of samples sorted along a Hilbert curve.  The long-range part is smooth and is
// summed on a mesh:
//   1. every sample spreads a unit charge to 4 x 4 x 4 nodes with cubic
//      B-spline weights (64-bit fixed-point atomics: exact, order-free);
//   2. the charge mesh (M^3 nodes, zero-padded to L = 2M per axis) is
//      convolved with the long-range kernel by FP32 real FFTs (cuFFT);
//   3. every sample gathers the four convolved fields (force x, y, z and the
//      potential) from its 64 nodes with the same weights.
// The kernel spectra are built once per mesh and eps: the kernel, tapered to
// zero beyond every offset the mesh can have (a C-infinity step between
// radius sqrt(3) M h and 2 M h), is sampled on a 4M box, transformed (FP64),
// divided by the squared transform of the B-spline window (deconvolution),
// transformed back, cut to the offsets |m| < M and transformed on the L box.
// The taper keeps the deconvolution from amplifying a truncation edge (the
// free-space convolution idea of Vico, Greengard and Ferrando, 2016).
// The erfc of the short-range part is the rational approximation 7.1.26 of
// Abramowitz and Stegun (|error| <= 1.5e-7) times exp(-x^2).
#include <cuda_runtime.h>
#include <cufft.h>
#include <cub/device/device_radix_sort.cuh>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "kernels.h"
#include "ptx.cuh"

namespace sparkling {

namespace {

constexpr int kMeshThreads = 256;
constexpr double kFix = 4294967296.0;       // charge fixed point: round(w * 2^32)

int grid_for(int64_t n, int sms)
{
    const int64_t b = (n + kMeshThreads - 1) / kMeshThreads, cap = (int64_t)sms * 16;
    return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

// C-infinity step: 1 for t <= 0, 0 for t >= 1.
__device__ double taper(double t)
{
    if (t <= 0.0) return 1.0;
    if (t >= 1.0) return 0.0;
    const double a = exp(-1.0 / (1.0 - t)), b = exp(-1.0 / t);
    return a / (a + b);
}

// Component c (0..2 force, 3 potential) of the tapered long-range kernel at
// the offsets of the periodic Lb = 4M box (residue order), planes z0 ..
// z0 + nz - 1 of it: out[z - z0][y][x].
__global__ void fill_slab_kernel(double *out, int Lb, int z0, int nz, double h, double sigma,
                                 double eps2, double r1, double r2, int c)
{
    const int64_t total = (int64_t)nz * Lb * Lb;
    const double spi = sigma * 0.56418958354775628;   // sigma / sqrt(pi)
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int ix = (int)(e % Lb), iy = (int)((e / Lb) % Lb);
        const int iz = z0 + (int)(e / ((int64_t)Lb * Lb));
        const double x = (ix <= Lb / 2 ? ix : ix - Lb) * h;
        const double y = (iy <= Lb / 2 ? iy : iy - Lb) * h;
        const double z = (iz <= Lb / 2 ? iz : iz - Lb) * h;
        const double d2 = x * x + y * y + z * z;
        const double r = sqrt(d2 + eps2), q = r / sigma;
        const double chi = taper((sqrt(d2) - r1) / (r2 - r1));
        double v;
        if (c == 3) {
            v = r * erf(q) + spi * exp(-q * q);
        } else {
            const double e_over_r = r > 0.0 ? erf(q) / r : 2.0 * 0.56418958354775628 / sigma;
            v = (c == 0 ? x : (c == 1 ? y : z)) * e_over_r;
        }
        out[e] = v * chi;
    }
}

// One axis of the deconvolution: divide the spectrum of every 1-D line by
// sinc(f)^8, the squared transform of the cubic B-spline window along that
// axis (f = frequency index / Lb in cycles per sample).  Element e holds
// frequency (e / inner) % nf.
__global__ void deconvolve_axis_kernel(cufftDoubleComplex *k, int64_t n, int64_t inner, int nf,
                                       int Lb)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int f = (int)((e / inner) % nf);
        if (f == 0) continue;
        const double t = 3.14159265358979323846 * f / Lb;
        const double s = sin(t) / t, s2 = s * s, s4 = s2 * s2;
        const double w = s4 * s4;
        k[e].x /= w;
        k[e].y /= w;
    }
}

// Offset index of the L = 2M box (residue order; index M unused) -> index
// of the Lb box, or -1 for the unused index.
__device__ __forceinline__ int small_to_big(int i, int M, int Lb)
{
    if (i == M) return -1;
    const int m = i < M ? i : i - 2 * M;
    return (m + Lb) % Lb;
}

// Pass 1 (x): src[zz][y][x] (x over Lb) -> a1[z0 + zz][y][xs] (xs over 2M).
__global__ void keep_x_kernel(double *a1, const double *src, int z0, int nz, int Lb, int M)
{
    const int L = 2 * M;
    const int64_t total = (int64_t)nz * Lb * L;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int xs = (int)(e % L);
        const int64_t row = e / L;                       // zz * Lb + y
        const int bx = small_to_big(xs, M, Lb);
        a1[((int64_t)z0 * Lb) * L + e] = bx < 0 ? 0.0 : src[row * Lb + bx];
    }
}

// Pass 2 (y): plane src[y][x] (y over Lb, x over 2M) -> a2[z][ys][x].
__global__ void keep_y_kernel(double *a2, const double *src, int z, int Lb, int M)
{
    const int L = 2 * M;
    const int64_t total = (int64_t)L * L;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int x = (int)(e % L), ys = (int)(e / L);
        const int by = small_to_big(ys, M, Lb);
        a2[(int64_t)z * L * L + e] = by < 0 ? 0.0 : src[(int64_t)by * L + x];
    }
}

// Pass 3 (z): plane src[z][x] (z over Lb, x over 2M) for row ys -> the
// float L box out[zs][ys][x], scaled.
__global__ void keep_z_kernel(float *out, const double *src, int ys, int Lb, int M, double scale)
{
    const int L = 2 * M;
    const int64_t total = (int64_t)L * L;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int x = (int)(e % L), zs = (int)(e / L);
        const int bz = small_to_big(zs, M, Lb);
        out[((int64_t)zs * L + ys) * L + x] =
            bz < 0 ? 0.f : (float)(src[(int64_t)bz * L + x] * scale);
    }
}

// Cubic B-spline weights of the 4 nodes first .. first + 3 around mesh
// coordinate u (first = floor(u) - 1); u in double, weights in float.
__device__ __forceinline__ void bspline_weights(double u, int &first, float w[4])
{
    const double fl = floor(u);
    first = (int)fl - 1;
    const float f = (float)(u - fl), g = 1.f - f, f2 = f * f, f3 = f2 * f;
    w[0] = g * g * g * (1.f / 6.f);
    w[1] = (3.f * f3 - 6.f * f2 + 4.f) * (1.f / 6.f);
    w[2] = (-3.f * f3 + 3.f * f2 + 3.f * f + 1.f) * (1.f / 6.f);
    w[3] = f3 * (1.f / 6.f);
}

struct NodeWeights {
    int first[3];
    float w[3][4];
    bool ok;
};

__device__ __forceinline__ NodeWeights node_weights(float4 p, double x0, double inv_h, int M)
{
    NodeWeights nw;
    const double u[3] = {((double)p.x - x0) * inv_h, ((double)p.y - x0) * inv_h,
                         ((double)p.z - x0) * inv_h};
    nw.ok = true;
    for (int a = 0; a < 3; ++a) {
        const bool in = u[a] >= 1.0 && u[a] < (double)(M - 2);
        nw.ok = nw.ok && in;
        bspline_weights(in ? u[a] : 1.0, nw.first[a], nw.w[a]);
    }
    return nw;
}

// Unit charges of the samples (in curve order) on the M^3 charge mesh (fixed
// point: the order of the additions does not matter).
__global__ void spread_kernel(const float4 *__restrict__ pos, int64_t N, unsigned long long *Q,
                              double x0, double inv_h, int M, int *status)
{
    int bad = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N;
         i += (int64_t)gridDim.x * blockDim.x) {
        const NodeWeights nw = node_weights(pos[i], x0, inv_h, M);
        if (!nw.ok) {
            bad = 1;
            continue;
        }
        for (int c = 0; c < 4; ++c)
            for (int b = 0; b < 4; ++b) {
                const float wzy = nw.w[2][c] * nw.w[1][b];
                unsigned long long *row =
                    Q + ((int64_t)(nw.first[2] + c) * M + (nw.first[1] + b)) * M + nw.first[0];
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    const long long v = __double2ll_rn((double)(wzy * nw.w[0][a]) * kFix);
                    if (v) atomicAdd(row + a, (unsigned long long)v);
                }
            }
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(status, kDevRange);
}

// Fixed-point charges -> the zero-padded real L^3 box.
__global__ void charges_to_box_kernel(const unsigned long long *__restrict__ Q, float *box, int M,
                                      int L)
{
    const int64_t total = (int64_t)L * L * L;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int ix = (int)(e % L), iy = (int)((e / L) % L), iz = (int)(e / ((int64_t)L * L));
        float v = 0.f;
        if (ix < M && iy < M && iz < M)
            v = (float)((double)(long long)Q[((int64_t)iz * M + iy) * M + ix] * (1.0 / kFix));
        box[e] = v;
    }
}

// out = a * b (complex), n elements.
__global__ void spectrum_product_kernel(cufftComplex *out, const cufftComplex *__restrict__ a,
                                        const cufftComplex *__restrict__ b, int64_t n)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const cufftComplex x = a[e], y = b[e];
        out[e] = make_cuFloatComplex(x.x * y.x - x.y * y.y, x.x * y.y + x.y * y.x);
    }
}

// Long-range sums gathered from the convolved fields (L^3 boxes; node n of
// the mesh is box index n) -- the force x, y, z fields, or the potential
// field alone for the energy -- plus the short-range fixed-point sums
// ([3][N] or [1][N]): out = S + L.
// Thread k takes the k-th sample of the curve order (neighbours read the same
// nodes) and writes it at its own index idx[k].
template <bool ENERGY>
__global__ void gather_kernel(const float4 *__restrict__ pos, const int *__restrict__ idx,
                              int64_t N, const float *__restrict__ phi, int64_t box, int L, double x0,
                              double inv_h, int M, const unsigned long long *__restrict__ shortr,
                              dacc4 *out)
{
    constexpr int NC = ENERGY ? 1 : 3;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N;
         i += (int64_t)gridDim.x * blockDim.x) {
        const NodeWeights nw = node_weights(pos[i], x0, inv_h, M);
        float acc[NC];
#pragma unroll
        for (int k = 0; k < NC; ++k) acc[k] = 0.f;
        if (nw.ok) {
            for (int c = 0; c < 4; ++c)
                for (int b = 0; b < 4; ++b) {
                    const float wzy = nw.w[2][c] * nw.w[1][b];
                    const int64_t row = ((int64_t)(nw.first[2] + c) * L + (nw.first[1] + b)) * L +
                                        nw.first[0];
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        const float w = wzy * nw.w[0][a];
#pragma unroll
                        for (int k = 0; k < NC; ++k)
                            acc[k] = fmaf(w, __ldg(phi + k * box + row + a), acc[k]);
                    }
                }
        }
        dacc4 r;
        if (ENERGY) {
            r.x = r.y = r.z = 0.0;
            r.w = (double)(long long)shortr[i] * (1.0 / kFix) + (double)acc[0];
        } else {
            r.x = (double)(long long)shortr[i] * (1.0 / kFix) + (double)acc[0];
            r.y = (double)(long long)shortr[N + i] * (1.0 / kFix) + (double)acc[NC > 1 ? 1 : 0];
            r.z = (double)(long long)shortr[2 * N + i] * (1.0 / kFix) + (double)acc[NC > 2 ? 2 : 0];
            r.w = 0.0;
        }
        out[idx[i]] = r;
    }
}

// ---- short-range part ------------------------------------------------------
//
// The samples are sorted along a Hilbert curve (10 bits an axis; a Morton curve
// jumps, and the boxes of samples on both sides of a jump are large).  A
// cluster is 32 consecutive samples; clusters, runs of 32 clusters and runs of 32 of those
// keep their bounding boxes (levels 0, 1, 2).  Where samples crowd -- the
// centre, which every shot crosses -- their clusters are small, so the boxes
// follow the density by themselves.
//
// A warp holds a group of two clusters, one target of each a lane, and finds
// the clusters behind it in the order with a box within rc of the group's, 32
// tests at a time through the levels.  Two near clusters at a time, a source
// of each a lane, meet the group: the sources and their sums rotate one lane a
// step, so every unordered pair is evaluated once and counts for both samples
// (the pair term is odd).  The two sources of a lane share 64-bit registers
// (paired FP32).  Inside the group every ordered pair is evaluated.  A cluster
// near one half of the group only meets that half.
//
// Bound: the FP32 and SFU pipes together (22 lane operations and three SFU
// results an unordered pair evaluated, of which one in 3.4 is in range at 1e7
// samples on 256 cells and one in 1.4 at 1e6 on 128); 65536 samples on 64 cells:
// ncu has the FMA pipe 57 % and the SFU 49 % busy, the warps of an SM moving
// through the same step in phase.  Measured against the cell list before it
// (directed pairs, cells of rc/3, every source of 49 neighbour rows tested against
// 64 targets): 1e7 samples, 256 cells 176 -> 71 ms; 1e6 samples on spokes, 128
// cells 250 -> 80 ms.  On the way, 1e7 / 1e6 samples: directed with the sources
// culled against the boxes 124 / 152 ms, symmetric pairs 133 / 90, Hilbert instead
// of Morton order 82 / 77 ms; with four targets a lane 85 ms (larger boxes, half
// the shuffles).

constexpr int kCluster = 32;
constexpr float kFar = 1e17f;

// Spread the low 10 bits of v to every third bit.
__device__ __forceinline__ unsigned int spread3(unsigned int v)
{
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000ffu;
    v = (v | (v << 8)) & 0x0300f00fu;
    v = (v | (v << 4)) & 0x030c30c3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}

__device__ __forceinline__ unsigned int grid_coord(float x, float x0, float inv)
{
    const int c = (int)floorf((x - x0) * inv);
    return (unsigned int)(c < 0 ? 0 : (c > 1023 ? 1023 : c));
}

// Index of a cell on the Hilbert curve of the 1024^3 grid, by the exchange and
// inversion of axes bit by bit (Skilling, "Programming the Hilbert curve", 2004).
__device__ __forceinline__ unsigned int hilbert_key(unsigned int x, unsigned int y, unsigned int z)
{
    unsigned int a[3] = {x, y, z};
#pragma unroll
    for (int bit = 9; bit > 0; --bit) {
        const unsigned int low = (1u << bit) - 1u;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const unsigned int set = 0u - ((a[c] >> bit) & 1u);       // all ones where the bit is set
            const unsigned int swap = (a[0] ^ a[c]) & low & ~set;     // exchange with axis 0, or
            a[0] ^= swap | (low & set);                               // invert axis 0
            a[c] ^= swap;
        }
    }
    a[1] ^= a[0];                                                     // Gray code
    a[2] ^= a[1];
    unsigned int flip = 0u;
#pragma unroll
    for (int bit = 9; bit > 0; --bit) flip ^= (0u - ((a[2] >> bit) & 1u)) & ((1u << bit) - 1u);
    return spread3(a[0] ^ flip) << 2 | spread3(a[1] ^ flip) << 1 | spread3(a[2] ^ flip);
}

__global__ void curve_keys_kernel(const float4 *__restrict__ pos, int64_t N, float x0, float inv,
                                  unsigned int *keys, int *vals)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float4 p = pos[i];
        keys[i] = hilbert_key(grid_coord(p.x, x0, inv), grid_coord(p.y, x0, inv),
                              grid_coord(p.z, x0, inv));
        vals[i] = (int)i;
    }
}

struct Box {
    float4 lo, hi;
};

__device__ __forceinline__ Box empty_box()
{
    const float inf = __int_as_float(0x7f800000);
    return {make_float4(inf, inf, inf, 0.f), make_float4(-inf, -inf, -inf, 0.f)};
}

// Union of the boxes of the lanes of each aligned group of W lanes.
template <int W> __device__ __forceinline__ void box_union(Box &b)
{
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) {
        b.lo.x = fminf(b.lo.x, __shfl_xor_sync(0xffffffffu, b.lo.x, o));
        b.lo.y = fminf(b.lo.y, __shfl_xor_sync(0xffffffffu, b.lo.y, o));
        b.lo.z = fminf(b.lo.z, __shfl_xor_sync(0xffffffffu, b.lo.z, o));
        b.hi.x = fmaxf(b.hi.x, __shfl_xor_sync(0xffffffffu, b.hi.x, o));
        b.hi.y = fmaxf(b.hi.y, __shfl_xor_sync(0xffffffffu, b.hi.y, o));
        b.hi.z = fmaxf(b.hi.z, __shfl_xor_sync(0xffffffffu, b.hi.z, o));
    }
}

// The samples' positions in sorted order and the boxes of their clusters (one
// warp a cluster).  Coordinates are multiplied by `unit`, a power of two (no
// rounding), which puts sigma into [1/2, 1).  A sample that is not a number or so
// far away that squares overflow -- the call reports it -- goes where it is near
// to no other and outside its cluster's box: it spoils no other sample's sums.
__global__ void sorted_clusters_kernel(const int *__restrict__ idx, const float4 *__restrict__ pos,
                                       int64_t N, int64_t n0, float unit, float4 *spos, Box *boxes)
{
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * blockDim.x / 32;
    for (int64_t c = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / 32; c < n0; c += warps) {
        const int64_t k = c * kCluster + lane;
        Box b = empty_box();
        if (k < N) {
            float4 p = pos[idx[k]];
            p.x *= unit; p.y *= unit; p.z *= unit;
            if (fabsf(p.x) < kFar && fabsf(p.y) < kFar && fabsf(p.z) < kFar) b.lo = b.hi = p;
            else p = make_float4(kFar, kFar, kFar, 0.f);
            spos[k] = p;
        }
        box_union<32>(b);
        if (lane == 0) boxes[c] = b;
    }
}

// Boxes of the runs of 32 boxes of the level below (n of them).
__global__ void parent_boxes_kernel(const Box *__restrict__ below, int64_t n, Box *boxes)
{
    const int lane = threadIdx.x & 31;
    const int64_t up = (n + 31) / 32, warps = (int64_t)gridDim.x * blockDim.x / 32;
    for (int64_t c = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / 32; c < up; c += warps) {
        const int64_t k = c * 32 + lane;
        Box b = k < n ? below[k] : empty_box();
        box_union<32>(b);
        if (lane == 0) boxes[c] = b;
    }
}

struct ShortArgs {
    const float4 *spos;
    const Box *boxes;            // levels 0, 1, 2 one after the other
    int64_t N, n0, n1, n2;
    int64_t groups;              // ceil(N / kGroup)
    int parts;                   // parts of the sources of one group (a power of two)
    unsigned long long *queue;
    float rc2, rc2_cull;         // cut-off, compared with d^2 + eps2; the same for boxes, rounded up
    float eps2;                  // eps^2, at least kEps2
    float p;                     // 0.3275911 / sigma
    float gauss;                 // -log2(e) / sigma^2
    float nspi;                  // -sigma / sqrt(pi)
    float to_fix;                // sums to fixed point: 2^32 (and the energy back to its unit)
    unsigned long long *acc;     // [NV][N] fixed-point sums, curve order
};

__device__ __forceinline__ float gap(float lo, float hi, float tlo, float thi)
{
    return fmaxf(fmaxf(lo - thi, tlo - hi), 0.f);
}

// Whether box b may hold a point within rc of the box t (never false where
// one does: rc2_cull is rc^2 rounded up by more than the test's rounding).
__device__ __forceinline__ bool box_near(const Box &b, const Box &t, float rc2_cull)
{
    const float gx = gap(b.lo.x, b.hi.x, t.lo.x, t.hi.x), gy = gap(b.lo.y, b.hi.y, t.lo.y, t.hi.y),
                gz = gap(b.lo.z, b.hi.z, t.lo.z, t.hi.z);
    return fmaf(gx, gx, fmaf(gy, gy, gz * gz)) <= rc2_cull;
}

constexpr int kShortThreads = 128;               // 4 warps, each takes its own items
constexpr int kT = 2;                            // targets a lane
constexpr int kGroup = 32 * kT;
constexpr int kFoldSteps = 64;                   // cluster pairs summed in FP32 (4096 sources a target)

struct ShortTargets {
    f2 x[kT], y[kT], z[kT];                      // each target in both halves
    f2 ax[kT], ay[kT], az[kT];                   // its sums over the two sources' halves
};

__device__ __forceinline__ void add_fix(unsigned long long *p, float v, float to_fix)
{
    const long long x = __float2ll_rn(v * to_fix);
    if (x) atomicAdd(p, (unsigned long long)x);
}

// The group's targets against two clusters of sources (q0, q1: the lane's).
// erfc(x) is a polynomial in t = 1/(1 + p x) times exp(-x^2): 22 FP32 lane
// operations and three SFU results a pair, which load the two pipes alike (a
// polynomial for log2 erfc needs two SFU results and 24 operations: 7 % slower).
// SYM: the sources' sums are added to their totals as well.
// Pairs of samples with |d| < rc only; the self pair adds nothing to the force
// and g_short(0) to the energy.
// T0, TN: the targets that take part (both halves of the group, or one).
template <bool ENERGY, bool SYM, int T0, int TN>
__device__ __forceinline__ void short_step(const ShortArgs &a, ShortTargets &T, float4 q0, float4 q1,
                                           int64_t k0, int64_t k1, bool ok0, bool ok1)
{
    const int lane = threadIdx.x & 31, from = (lane + 1) & 31;
    f2 SX = f2_pack(q0.x, q1.x), SY = f2_pack(q0.y, q1.y), SZ = f2_pack(q0.z, q1.z);
    f2 BX = f2_pack(0.f, 0.f), BY = BX, BZ = BX;
    // paired constants, kept in registers (as constant-bank operands of the
    // paired instructions they cost 10 %)
    auto both = [](float v) { return f2_pack(v, v); };
    const f2 E2 = both(a.eps2);
    const f2 ONE = both(1.f), P = both(a.p), GA = both(a.gauss), NSPI = both(a.nspi);
    const f2 C5 = both(1.061405429f), C4 = both(-1.453152027f), C3 = both(1.421413741f),
             C2 = both(-0.284496736f), C1 = both(0.254829592f);
    for (int step = 0; step < 32; ++step) {
#pragma unroll
        for (int t = T0; t < T0 + TN; ++t) {
            const f2 DX = f2_sub(T.x[t], SX), DY = f2_sub(T.y[t], SY), DZ = f2_sub(T.z[t], SZ);
            const f2 R2 = f2_fma(DX, DX, f2_fma(DY, DY, f2_fma(DZ, DZ, E2)));
            float r2a, r2b, ea, eb;
            f2_unpack(R2, r2a, r2b);
            const f2 RI = f2_pack(rsqrt_sfu(r2a), rsqrt_sfu(r2b));
            const f2 R = f2_mul(R2, RI);
            float da, db;
            f2_unpack(f2_fma(R, P, ONE), da, db);
            const f2 TT = f2_pack(rcp_sfu(da), rcp_sfu(db));
            f2_unpack(f2_mul(R2, GA), ea, eb);
            ea = r2a < a.rc2 ? ex2_sfu(ea) : 0.f;
            eb = r2b < a.rc2 ? ex2_sfu(eb) : 0.f;
            const f2 G = f2_pack(ea, eb);
            const f2 EC = f2_mul(f2_mul(TT, G), f2_fma(TT, f2_fma(TT, f2_fma(TT, f2_fma(TT, C5, C4),
                                                                          C3), C2), C1));
            if (ENERGY) {
                const f2 E = f2_fma(R, EC, f2_mul(NSPI, G));
                T.ax[t] = f2_add(T.ax[t], E);
                if (SYM) BX = f2_add(BX, E);
            } else {
                const f2 W = f2_mul(EC, RI);
                T.ax[t] = f2_fma(DX, W, T.ax[t]);
                T.ay[t] = f2_fma(DY, W, T.ay[t]);
                T.az[t] = f2_fma(DZ, W, T.az[t]);
                if (SYM) {
                    BX = f2_fma(DX, W, BX);
                    BY = f2_fma(DY, W, BY);
                    BZ = f2_fma(DZ, W, BZ);
                }
            }
        }
        // the sources and their sums move one lane down
        SX = __shfl_sync(0xffffffffu, SX, from);
        SY = __shfl_sync(0xffffffffu, SY, from);
        SZ = __shfl_sync(0xffffffffu, SZ, from);
        if (SYM) {
            BX = __shfl_sync(0xffffffffu, BX, from);
            if (!ENERGY) {
                BY = __shfl_sync(0xffffffffu, BY, from);
                BZ = __shfl_sync(0xffffffffu, BZ, from);
            }
        }
    }
    if (SYM) {                                   // back home after 32 steps; the force term is odd
        float u, v;
        f2_unpack(BX, u, v);
        if (ok0) add_fix(a.acc + k0, ENERGY ? u : -u, a.to_fix);
        if (ok1) add_fix(a.acc + k1, ENERGY ? v : -v, a.to_fix);
        if (!ENERGY) {
            f2_unpack(BY, u, v);
            if (ok0) add_fix(a.acc + a.N + k0, -u, a.to_fix);
            if (ok1) add_fix(a.acc + a.N + k1, -v, a.to_fix);
            f2_unpack(BZ, u, v);
            if (ok0) add_fix(a.acc + 2 * a.N + k0, -u, a.to_fix);
            if (ok1) add_fix(a.acc + 2 * a.N + k1, -v, a.to_fix);
        }
    }
}

// A lane of `todo` whose cluster is near the halves `want`, or any.
__device__ __forceinline__ int pick(unsigned int todo, int near, int want)
{
    const unsigned int same = __ballot_sync(0xffffffffu, near == want) & todo;
    return __ffs(same ? same : todo) - 1;
}

// Persistent warps take items (group, part) from a queue; part p of P takes
// every P-th near level-1 run, so that no item is long where samples crowd.
// FP32 sums go to 64-bit fixed-point totals (exact, order-free).
template <bool ENERGY>
__global__ void __launch_bounds__(kShortThreads, 5) short_items_kernel(const ShortArgs a)
{
    constexpr int NV = ENERGY ? 1 : 3;
    constexpr unsigned int kAll = 0xffffffffu;
    __shared__ Box halves[kShortThreads / 32][2];
    const int lane = threadIdx.x & 31;
    const Box *box0 = a.boxes, *box1 = box0 + a.n0, *box2 = box1 + a.n1;
    const unsigned long long total = (unsigned long long)a.groups * a.parts;
    // samples that do not exist: beyond every cut-off of the others
    const float4 no_target = make_float4(1e18f, 1e18f, 1e18f, 0.f);
    const float4 no_source = make_float4(-1e18f, -1e18f, -1e18f, 0.f);
    for (;;) {
        unsigned long long u = 0;
        if (lane == 0) u = atomicAdd(a.queue, 1ull);
        u = __shfl_sync(kAll, u, 0);
        if (u >= total) break;
        const int part = (int)(u / a.groups);
        const int64_t g = (int64_t)(u % a.groups), first = g * kGroup;
        ShortTargets T;
        Box half[2] = {empty_box(), empty_box()};
#pragma unroll
        for (int t = 0; t < kT; ++t) {
            Box &tb = half[t / (kT / 2)];
            const int64_t k = first + t * 32 + lane;
            const bool ok = k < a.N;
            const float4 p = ok ? a.spos[k] : no_target;
            T.x[t] = f2_pack(p.x, p.x);
            T.y[t] = f2_pack(p.y, p.y);
            T.z[t] = f2_pack(p.z, p.z);
            T.ax[t] = T.ay[t] = T.az[t] = f2_pack(0.f, 0.f);
            if (ok) {
                tb.lo = make_float4(fminf(tb.lo.x, p.x), fminf(tb.lo.y, p.y), fminf(tb.lo.z, p.z), 0.f);
                tb.hi = make_float4(fmaxf(tb.hi.x, p.x), fmaxf(tb.hi.y, p.y), fmaxf(tb.hi.z, p.z), 0.f);
            }
        }
        box_union<32>(half[0]);
        box_union<32>(half[1]);
        // the halves' boxes wait in shared memory; the group's stays at hand
        __syncwarp();
        if (lane == 0) {
            halves[threadIdx.x >> 5][0] = half[0];
            halves[threadIdx.x >> 5][1] = half[1];
        }
        __syncwarp();
        const Box *hb = halves[threadIdx.x >> 5];
        Box tb;
        tb.lo = make_float4(fminf(half[0].lo.x, half[1].lo.x), fminf(half[0].lo.y, half[1].lo.y),
                            fminf(half[0].lo.z, half[1].lo.z), 0.f);
        tb.hi = make_float4(fmaxf(half[0].hi.x, half[1].hi.x), fmaxf(half[0].hi.y, half[1].hi.y),
                            fmaxf(half[0].hi.z, half[1].hi.z), 0.f);
        int steps = 0;
        auto fold = [&]() {
#pragma unroll
            for (int t = 0; t < kT; ++t) {
                const int64_t k = first + t * 32 + lane;
                float u0, v0;
                f2_unpack(T.ax[t], u0, v0);
                if (k < a.N) add_fix(a.acc + k, u0 + v0, a.to_fix);
                if (NV > 1) {
                    f2_unpack(T.ay[t], u0, v0);
                    if (k < a.N) add_fix(a.acc + a.N + k, u0 + v0, a.to_fix);
                    f2_unpack(T.az[t], u0, v0);
                    if (k < a.N) add_fix(a.acc + 2 * a.N + k, u0 + v0, a.to_fix);
                }
                T.ax[t] = T.ay[t] = T.az[t] = f2_pack(0.f, 0.f);
            }
            steps = 0;
        };
        // the group's own pairs, directed (part 0)
        if (part == 0) {
            for (int h = 0; h < kT; h += 2) {
                const int64_t k0 = first + h * 32 + lane, k1 = k0 + 32;
                short_step<ENERGY, false, 0, kT>(a, T, k0 < a.N ? a.spos[k0] : no_source,
                                                 k1 < a.N ? a.spos[k1] : no_source, 0, 0, false,
                                                 false);
                ++steps;
            }
        }
        // the clusters behind the group, two at a time
        const int64_t behind = (g + 1) * kT;       // first cluster behind
        int64_t held = -1;                         // a near cluster waiting for a second one,
        int held_near = 0;                         // and the halves it is near to (bits)
        auto meet = [&](int64_t c0, int64_t c1, int near) {
            const int64_t k0 = c0 * kCluster + lane, k1 = c1 * kCluster + lane;
            const bool ok0 = k0 < a.N, ok1 = c1 >= 0 && k1 < a.N;
            const float4 q0 = ok0 ? a.spos[k0] : no_source, q1 = ok1 ? a.spos[k1] : no_source;
            if (near == 3)
                short_step<ENERGY, true, 0, kT>(a, T, q0, q1, k0, k1, ok0, ok1);
            else if (near == 1)
                short_step<ENERGY, true, 0, kT / 2>(a, T, q0, q1, k0, k1, ok0, ok1);
            else
                short_step<ENERGY, true, kT / 2, kT / 2>(a, T, q0, q1, k0, k1, ok0, ok1);
            if (++steps == kFoldSteps) fold();
        };
        int ordinal = 0;
        for (int64_t b2 = behind / 1024 / 32 * 32; b2 < a.n2; b2 += 32) {
            unsigned int m2 = __ballot_sync(kAll, b2 + lane < a.n2 && (b2 + lane + 1) * 1024 > behind &&
                                                      box_near(box2[b2 + lane], tb, a.rc2_cull));
            while (m2) {
                const int64_t b1 = (b2 + __ffs(m2) - 1) * 32;
                m2 &= m2 - 1;
                unsigned int m1 = __ballot_sync(kAll, b1 + lane < a.n1 && (b1 + lane + 1) * 32 > behind &&
                                                          box_near(box1[b1 + lane], tb, a.rc2_cull));
                while (m1) {
                    const int64_t b0 = (b1 + __ffs(m1) - 1) * 32;
                    m1 &= m1 - 1;
                    if ((ordinal++ & (a.parts - 1)) != part) continue;
                    int near = 0;
                    if (b0 + lane < a.n0 && b0 + lane >= behind) {
                        const Box b = box0[b0 + lane];
                        near = (box_near(b, hb[0], a.rc2_cull) ? 1 : 0) |
                               (box_near(b, hb[1], a.rc2_cull) ? 2 : 0);
                    }
                    // clusters near the same halves meet them together
                    unsigned int todo = __ballot_sync(kAll, near != 0);
                    while (todo) {
                        const int l = held < 0 ? __ffs(todo) - 1 : pick(todo, near, held_near);
                        todo &= ~(1u << l);
                        const int ln = __shfl_sync(kAll, near, l);
                        if (held < 0) {
                            held = b0 + l;
                            held_near = ln;
                        } else {
                            meet(held, b0 + l, held_near | ln);
                            held = -1;
                        }
                    }
                }
            }
        }
        if (held >= 0) meet(held, -1, held_near);
        if (steps > 0) fold();
    }
}

} // namespace

// ---- host side ---------------------------------------------------------------

namespace {

bool seven_smooth(int n)
{
    for (int p : {2, 3, 5, 7})
        while (n % p == 0) n /= p;
    return n == 1;
}

template <typename T> cudaError_t grow(T *&p, size_t &cap, size_t bytes)
{
    if (bytes <= cap) return cudaSuccess;
    cudaFree(p);
    p = nullptr;
    cap = 0;
    cudaError_t e = cudaMalloc(&p, bytes);
    if (e == cudaSuccess) cap = bytes;
    return e;
}

} // namespace

struct MeshState {
    MeshConfig cfg;          // the mesh the spectra were built for
    bool built = false;
    int M = 0, L = 0;
    double x0 = 0.0;
    cufftComplex *spectra = nullptr;   // 4 kernel spectra on the L box (scaled by 1/L^3)
    size_t spectra_cap = 0;
    cufftHandle r2c = 0, c2r = 0;
    bool plans = false;
    // evaluation buffers (grow with N)
    unsigned long long *Q = nullptr; size_t Q_cap = 0;
    float *box = nullptr; size_t box_cap = 0;           // charges, then 4 fields
    cufftComplex *qhat = nullptr; size_t qhat_cap = 0;
    cufftComplex *tmp = nullptr; size_t tmp_cap = 0;
    unsigned int *keys = nullptr; size_t keys_cap = 0;   // 2N keys
    int *vals = nullptr; size_t vals_cap = 0;            // 2N indices
    float4 *spos = nullptr; size_t spos_cap = 0;         // samples in curve order
    Box *boxes = nullptr; size_t boxes_cap = 0;          // levels 0, 1, 2
    unsigned long long *shortr = nullptr; size_t shortr_cap = 0;   // fixed point [3][N], curve order
    unsigned long long *queue = nullptr;                 // item queue
    int short_ctas[2] = {0, 0};                          // persistent CTAs (gradient, energy)
    void *cub = nullptr; size_t cub_cap = 0;
};

MeshState *mesh_state_create() { return new MeshState(); }

void mesh_state_destroy(MeshState *m)
{
    if (!m) return;
    if (m->plans) { cufftDestroy(m->r2c); cufftDestroy(m->c2r); }
    cudaFree(m->spectra); cudaFree(m->Q); cudaFree(m->box); cudaFree(m->qhat); cudaFree(m->tmp);
    cudaFree(m->keys); cudaFree(m->vals); cudaFree(m->spos); cudaFree(m->boxes);
    cudaFree(m->shortr); cudaFree(m->cub); cudaFree(m->queue);
    delete m;
}

int mesh_guard(int n_cells)
{
    int g = 4;
    while (!seven_smooth(n_cells + 2 * g)) ++g;
    return g;
}

bool mesh_matches(const MeshState *m, const MeshConfig &c)
{
    return m->built && m->cfg.n_cells == c.n_cells && m->cfg.lo == c.lo && m->cfg.hi == c.hi &&
           m->cfg.sigma == c.sigma && m->cfg.rc == c.rc && m->cfg.eps == c.eps;
}

// Kernel spectra and FFT plans of mesh c (blocking; allocates the 4M box for
// the duration of the call).
cudaError_t mesh_build(MeshState *m, const MeshConfig &c, int sms, cudaStream_t st,
                       const char **what)
{
    m->built = false;
    const int g = mesh_guard(c.n_cells);
    const int M = c.n_cells + 2 * g, L = 2 * M, Lb = 4 * M, nf = Lb / 2 + 1;
    const double h = (c.hi - c.lo) / c.n_cells;
    const int64_t nl = (int64_t)L * L * L, nlc = (int64_t)L * L * (L / 2 + 1);
    // The deconvolution divides by a product of one factor per axis, so it
    // runs as three passes of 1-D transforms over the Lb = 4M box, each
    // keeping only the offsets |m| < M of its axis: pass 1 (x) on slabs of
    // kSlab planes of the kernel generated on the fly, pass 2 (y) per z
    // plane, pass 3 (z) per y row.  Peak memory: a1 = Lb * Lb * 2M and
    // a2 = Lb * 2M * 2M doubles (the full box would be Lb^3).
    constexpr int kSlab = 8;
    double *a1 = nullptr, *a2 = nullptr, *rbuf = nullptr;
    cufftDoubleComplex *cbuf = nullptr;
    float *small = nullptr;
    void *work = nullptr;
    cufftHandle px_f = 0, px_i = 0, py_f = 0, py_i = 0, pz_f = 0, pz_i = 0, sfwd = 0;
    bool made[7] = {false, false, false, false, false, false, false};
    cufftHandle *handles[7] = {&px_f, &px_i, &py_f, &py_i, &pz_f, &pz_i, &sfwd};
    cudaError_t err = cudaSuccess;
    auto done = [&](cudaError_t e) {
        for (int k = 0; k < 7; ++k)
            if (made[k]) cufftDestroy(*handles[k]);
        cudaFree(a1); cudaFree(a2); cudaFree(rbuf); cudaFree(cbuf); cudaFree(small);
        cudaFree(work);
        return e;
    };
    *what = "mesh kernel buffers";
    const size_t rbuf_n = std::max((size_t)kSlab * Lb * Lb, (size_t)Lb * L);
    const size_t cbuf_n = std::max((size_t)kSlab * Lb * nf, (size_t)nf * L);
    if ((err = grow(m->spectra, m->spectra_cap, (size_t)4 * nlc * sizeof(cufftComplex))) ||
        (err = cudaMalloc(&a1, (size_t)Lb * Lb * L * sizeof(double))) ||
        (err = cudaMalloc(&a2, (size_t)Lb * L * L * sizeof(double))) ||
        (err = cudaMalloc(&rbuf, rbuf_n * sizeof(double))) ||
        (err = cudaMalloc(&cbuf, cbuf_n * sizeof(cufftDoubleComplex))) ||
        (err = cudaMalloc(&small, nl * sizeof(float))))
        return done(err);
    *what = "mesh cuFFT plans";
    // 1-D plans: n = Lb; x: contiguous lines; y, z: lines of stride L (x the batch)
    int n1[1] = {Lb}, nfe[1] = {nf};
    size_t ws[7] = {0, 0, 0, 0, 0, 0, 0};
    auto many = [&](int k, int istride, int idist, int ostride, int odist, int batch, cufftType t,
                    bool real_in) {
        if (cufftCreate(handles[k]) != CUFFT_SUCCESS) return false;
        made[k] = true;
        int *inem = real_in ? n1 : nfe, *onem = real_in ? nfe : n1;
        return cufftSetAutoAllocation(*handles[k], 0) == CUFFT_SUCCESS &&
               cufftMakePlanMany(*handles[k], 1, n1, inem, istride, idist, onem, ostride, odist,
                                 t, batch, &ws[k]) == CUFFT_SUCCESS;
    };
    if (!many(0, 1, Lb, 1, nf, kSlab * Lb, CUFFT_D2Z, true) ||
        !many(1, 1, nf, 1, Lb, kSlab * Lb, CUFFT_Z2D, false) ||
        !many(2, L, 1, L, 1, L, CUFFT_D2Z, true) || !many(3, L, 1, L, 1, L, CUFFT_Z2D, false) ||
        !many(4, L * L, 1, L, 1, L, CUFFT_D2Z, true) || !many(5, L, 1, L, 1, L, CUFFT_Z2D, false))
        return done(cudaErrorUnknown);
    if (cufftCreate(&sfwd) != CUFFT_SUCCESS) return done(cudaErrorUnknown);
    made[6] = true;
    if (cufftSetAutoAllocation(sfwd, 0) != CUFFT_SUCCESS ||
        cufftMakePlan3d(sfwd, L, L, L, CUFFT_R2C, &ws[6]) != CUFFT_SUCCESS)
        return done(cudaErrorUnknown);
    *what = "mesh cuFFT work area";
    size_t wmax = 256;
    for (int k = 0; k < 7; ++k) wmax = std::max(wmax, ws[k]);
    if ((err = cudaMalloc(&work, wmax))) return done(err);
    for (int k = 0; k < 7; ++k)
        if (cufftSetWorkArea(*handles[k], work) != CUFFT_SUCCESS ||
            cufftSetStream(*handles[k], st) != CUFFT_SUCCESS)
            return done(cudaErrorUnknown);
    *what = "mesh kernel spectra";
    const double r1 = std::sqrt(3.0) * M * h, r2 = 2.0 * M * h;
    const double scale = 1.0 / ((double)Lb * Lb * Lb * (double)nl);
    for (int comp = 0; comp < 4; ++comp) {
        // pass 1: x lines of up to kSlab planes at a time (the plan always
        // transforms kSlab planes; rows past the last plane are not kept)
        for (int z0 = 0; z0 < Lb; z0 += kSlab) {
            const int nzz = std::min(kSlab, Lb - z0);
            const int64_t nr = (int64_t)nzz * Lb * Lb;
            fill_slab_kernel<<<grid_for(nr, sms), kMeshThreads, 0, st>>>(
                rbuf, Lb, z0, nzz, h, c.sigma, c.eps * c.eps, r1, r2, comp);
            if (cufftExecD2Z(px_f, rbuf, cbuf) != CUFFT_SUCCESS) return done(cudaErrorUnknown);
            deconvolve_axis_kernel<<<grid_for((int64_t)kSlab * Lb * nf, sms), kMeshThreads, 0, st>>>(
                cbuf, (int64_t)kSlab * Lb * nf, 1, nf, Lb);
            if (cufftExecZ2D(px_i, cbuf, rbuf) != CUFFT_SUCCESS) return done(cudaErrorUnknown);
            keep_x_kernel<<<grid_for((int64_t)nzz * Lb * L, sms), kMeshThreads, 0, st>>>(
                a1, rbuf, z0, nzz, Lb, M);
        }
        // pass 2: y lines of every z plane of a1
        for (int z = 0; z < Lb; ++z) {
            if (cufftExecD2Z(py_f, a1 + (int64_t)z * Lb * L, cbuf) != CUFFT_SUCCESS)
                return done(cudaErrorUnknown);
            deconvolve_axis_kernel<<<grid_for((int64_t)nf * L, sms), kMeshThreads, 0, st>>>(
                cbuf, (int64_t)nf * L, L, nf, Lb);
            if (cufftExecZ2D(py_i, cbuf, rbuf) != CUFFT_SUCCESS) return done(cudaErrorUnknown);
            keep_y_kernel<<<grid_for((int64_t)L * L, sms), kMeshThreads, 0, st>>>(a2, rbuf, z, Lb, M);
        }
        // pass 3: z lines of every y row of a2, into the float L box
        for (int ys = 0; ys < L; ++ys) {
            if (cufftExecD2Z(pz_f, a2 + (int64_t)ys * L, cbuf) != CUFFT_SUCCESS)
                return done(cudaErrorUnknown);
            deconvolve_axis_kernel<<<grid_for((int64_t)nf * L, sms), kMeshThreads, 0, st>>>(
                cbuf, (int64_t)nf * L, L, nf, Lb);
            if (cufftExecZ2D(pz_i, cbuf, rbuf) != CUFFT_SUCCESS) return done(cudaErrorUnknown);
            keep_z_kernel<<<grid_for((int64_t)L * L, sms), kMeshThreads, 0, st>>>(small, rbuf, ys, Lb,
                                                                                  M, scale);
        }
        if ((err = cudaGetLastError())) return done(err);
        if (cufftExecR2C(sfwd, small, m->spectra + comp * nlc) != CUFFT_SUCCESS)
            return done(cudaErrorUnknown);
    }
    if ((err = cudaStreamSynchronize(st)) != cudaSuccess) return done(err);
    // evaluation plans on the L box
    *what = "mesh evaluation plans";
    if (m->plans) {
        cufftDestroy(m->r2c);
        cufftDestroy(m->c2r);
        m->plans = false;
    }
    if (cufftPlan3d(&m->r2c, L, L, L, CUFFT_R2C) != CUFFT_SUCCESS) return done(cudaErrorUnknown);
    if (cufftPlan3d(&m->c2r, L, L, L, CUFFT_C2R) != CUFFT_SUCCESS) {
        cufftDestroy(m->r2c);
        return done(cudaErrorUnknown);
    }
    m->plans = true;
    m->cfg = c;
    m->M = M;
    m->L = L;
    m->x0 = c.lo - g * h;
    m->built = true;
    *what = "";
    return done(cudaSuccess);
}

// Repulsion sums of the N packed samples into out[i] = (sum d/r, sum |d|_eps)
// over all j (directed, the self pair included as eps in the potential).
// Asynchronous: once the buffers have their size for N (the first call of a
// sample count allocates them), a call only enqueues work on `st` and can be
// captured.
// no_alloc (a call under stream capture): return cudaErrorStreamCaptureUnsupported
// instead of growing a buffer.
cudaError_t mesh_eval(MeshState *m, const float4 *pos, int64_t N, bool energy, dacc4 *out,
                      int *status, int sms, cudaStream_t st, const char **what, int *launches,
                      bool no_alloc)
{
    const MeshConfig &c = m->cfg;
    const int M = m->M, L = m->L;
    const int64_t nm = (int64_t)M * M * M, nl = (int64_t)L * L * L, nlc = (int64_t)L * L * (L / 2 + 1);
    const int nfield = energy ? 1 : 3;
    const int NV = energy ? 1 : 3;
    const int64_t n0 = (N + kCluster - 1) / kCluster, n1 = (n0 + 31) / 32, n2 = (n1 + 31) / 32;
    const double h = (c.hi - c.lo) / c.n_cells;
    cudaError_t err;
    *what = "mesh evaluation buffers";
    size_t sort_bytes = 0;
    constexpr int kKeyBits = 30;
    cub::DeviceRadixSort::SortPairs(nullptr, sort_bytes, m->keys, m->keys, m->vals, m->vals,
                                    (int)N, 0, kKeyBits, st);
    if (no_alloc &&
        (nm * sizeof(unsigned long long) > m->Q_cap ||
         (size_t)(nfield + 1) * nl * sizeof(float) > m->box_cap ||
         nlc * sizeof(cufftComplex) > m->qhat_cap || nlc * sizeof(cufftComplex) > m->tmp_cap ||
         (size_t)2 * N * sizeof(unsigned int) > m->keys_cap ||
         (size_t)2 * N * sizeof(int) > m->vals_cap || (size_t)N * sizeof(float4) > m->spos_cap ||
         (size_t)(n0 + n1 + n2) * sizeof(Box) > m->boxes_cap ||
         (size_t)N * 3 * sizeof(unsigned long long) > m->shortr_cap ||
         sort_bytes + 256 > m->cub_cap || !m->queue || !m->short_ctas[0]))
        return cudaErrorStreamCaptureUnsupported;

    if ((err = grow(m->Q, m->Q_cap, nm * sizeof(unsigned long long))) ||
        (err = grow(m->box, m->box_cap, (size_t)(nfield + 1) * nl * sizeof(float))) ||
        (err = grow(m->qhat, m->qhat_cap, nlc * sizeof(cufftComplex))) ||
        (err = grow(m->tmp, m->tmp_cap, nlc * sizeof(cufftComplex))) ||
        (err = grow(m->keys, m->keys_cap, (size_t)2 * N * sizeof(unsigned int))) ||
        (err = grow(m->vals, m->vals_cap, (size_t)2 * N * sizeof(int))) ||
        (err = grow(m->spos, m->spos_cap, (size_t)N * sizeof(float4))) ||
        (err = grow(m->boxes, m->boxes_cap, (size_t)(n0 + n1 + n2) * sizeof(Box))) ||
        (err = grow(m->shortr, m->shortr_cap, (size_t)N * 3 * sizeof(unsigned long long))) ||
        (err = grow(m->cub, m->cub_cap, sort_bytes + 256)))
        return err;
    if (!m->queue && (err = cudaMalloc(&m->queue, sizeof(unsigned long long)))) return err;
    if (!m->short_ctas[0]) {
        int a = 0, b = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, short_items_kernel<false>, kShortThreads, 0);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, short_items_kernel<true>, kShortThreads, 0);
        m->short_ctas[0] = sms * std::max(a, 1);
        m->short_ctas[1] = sms * std::max(b, 1);
    }
    if (cufftSetStream(m->r2c, st) != CUFFT_SUCCESS || cufftSetStream(m->c2r, st) != CUFFT_SUCCESS)
        return cudaErrorUnknown;
    *what = "mesh evaluation";
    const int gN = grid_for(N, sms);
    int nk = 0;
    // short-range part: samples sorted, boxes, pair sums
    curve_keys_kernel<<<gN, kMeshThreads, 0, st>>>(pos, N, (float)m->x0, (float)(1024.0 / (M * h)),
                                                    m->keys, m->vals);
    if ((err = cub::DeviceRadixSort::SortPairs(m->cub, sort_bytes, m->keys, m->keys + N, m->vals,
                                               m->vals + N, (int)N, 0, kKeyBits, st)))
        return err;
    const int *idx = m->vals + N;
    Box *box1 = m->boxes + n0, *box2 = box1 + n1;
    int exponent = 0;
    std::frexp(c.sigma, &exponent);                // sigma = f 2^exponent, f in [1/2, 1)
    const double unit = std::ldexp(1.0, -exponent), sigma = c.sigma * unit, eps = c.eps * unit;
    sorted_clusters_kernel<<<grid_for(n0 * 32, sms), kMeshThreads, 0, st>>>(
        idx, pos, N, n0, (float)unit, m->spos, m->boxes);
    parent_boxes_kernel<<<grid_for(n1 * 32, sms), kMeshThreads, 0, st>>>(m->boxes, n0, box1);
    parent_boxes_kernel<<<grid_for(n2 * 32, sms), kMeshThreads, 0, st>>>(box1, n1, box2);
    ShortArgs a{};
    a.spos = m->spos; a.boxes = m->boxes;
    a.N = N; a.n0 = n0; a.n1 = n1; a.n2 = n2;
    a.groups = (N + kGroup - 1) / kGroup;
    a.parts = 1;
    while (a.parts < 32 && a.groups * a.parts < ((int64_t)1 << 20)) a.parts *= 2;
    a.queue = m->queue;
    const double rc = c.rc * unit;
    a.eps2 = std::max((float)(eps * eps), kEps2);
    a.rc2 = (float)(rc * rc + eps * eps);
    a.rc2_cull = (float)(rc * rc * (1.0 + 1e-5));
    a.p = (float)(0.3275911 / sigma);
    a.gauss = (float)(-1.4426950408889634 / (sigma * sigma));
    a.nspi = (float)(-sigma * 0.56418958354775628);
    a.to_fix = (float)(4294967296.0 / (energy ? unit : 1.0));
    a.acc = m->shortr;
    if ((err = cudaMemsetAsync(m->queue, 0, sizeof(unsigned long long), st)) ||
        (err = cudaMemsetAsync(m->shortr, 0, (size_t)N * NV * sizeof(unsigned long long), st)))
        return err;
    const int64_t warps_needed = a.groups * a.parts;
    const int ctas = (int)std::min<int64_t>(m->short_ctas[energy ? 1 : 0], (warps_needed + 3) / 4);
    if (energy)
        short_items_kernel<true><<<ctas, kShortThreads, 0, st>>>(a);
    else
        short_items_kernel<false><<<ctas, kShortThreads, 0, st>>>(a);
    nk += 6;
    // long-range part
    if ((err = cudaMemsetAsync(m->Q, 0, nm * sizeof(unsigned long long), st))) return err;
    spread_kernel<<<gN, kMeshThreads, 0, st>>>(m->spos, N, m->Q, m->x0 * unit, 1.0 / (h * unit), M,
                                               status);
    charges_to_box_kernel<<<grid_for(nl, sms), kMeshThreads, 0, st>>>(m->Q, m->box, M, L);
    if (cufftExecR2C(m->r2c, m->box, m->qhat) != CUFFT_SUCCESS) return cudaErrorUnknown;
    for (int k = 0; k < nfield; ++k) {
        const int comp = energy ? 3 : k;
        spectrum_product_kernel<<<grid_for(nlc, sms), kMeshThreads, 0, st>>>(
            m->tmp, m->qhat, m->spectra + comp * nlc, nlc);
        if (cufftExecC2R(m->c2r, m->tmp, m->box + (1 + k) * nl) != CUFFT_SUCCESS)
            return cudaErrorUnknown;
    }
    if (energy)
        gather_kernel<true><<<gN, kMeshThreads, 0, st>>>(m->spos, idx, N, m->box + nl, nl, L,
                                                         m->x0 * unit, 1.0 / (h * unit), M,
                                                         m->shortr, out);
    else
        gather_kernel<false><<<gN, kMeshThreads, 0, st>>>(m->spos, idx, N, m->box + nl, nl, L,
                                                          m->x0 * unit, 1.0 / (h * unit), M,
                                                          m->shortr, out);
    nk += 3 + nfield + 1;
    *launches = nk;
    *what = "";
    return cudaGetLastError();
}

} // namespace sparkling
