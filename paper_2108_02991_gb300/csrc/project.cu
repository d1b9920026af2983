// Per-shot projection onto the gradient-amplitude / slew-rate / box / pin
// constraint set (paper eq. constraints, Sec. II-D, Suppl. Sec. I) by FISTA on
// the Fenchel dual of min 1/2 |s - k|^2, in FP64 (FP32 samples: two-float sums
// in the register form, project_reg.cuh):
//   D1 s[n] = s[n+1] - s[n]                 (n < Ns-1)
//   D2 s[n] = s[n+2] - 2 s[n+1] + s[n]      (n < Ns-2)
//   s(q)    = pin(clip_box(k - D1^T q1 - D2^T q2))
//   z       = y + tau D s(y),  tau = 1/20 (|D1|^2 <= 4, |D2|^2 <= 16)
//   q+      = z * max(0, 1 - tau*radius/|z|)        (row-wise, radius alpha/beta)
//   t+      = (1 + sqrt(1 + 4 t^2))/2,  y = q+ + ((t-1)/t+)(q+ - q)
// The output is s(q).  With a gradient G the shot is first stepped:
// k = K - eta G (eq. proj_grad_descent).
//
// Fixed iterations run in the register form (project_reg.cuh) up to 8192
// samples a shot.  What follows is the form with its state in memory, for
// converged mode, longer shots, more iterations than the momentum table holds,
// radii outside the two-float range (FP64 samples: with subnormal squares) and
// FP32 samples of a context that asked for FP64.  Outside the register form FP32
// samples may (an opt-in of the context) iterate in FP32 on the displacement
// s - k and the duals (project_shot_mixed), else in FP64.
//
// One CTA per shot (grid-stride over shots).  The 18 per-sample FP64 arrays
// (k, s, y1, y2, q1, q2; x, y, z each, structure of arrays so that a warp
// touches consecutive doubles) live in shared memory when they fit and in a
// per-CTA global scratch region otherwise; the code is the same through
// generic pointers.  Each iteration is two phases separated by barriers:
// S computes s from the duals, Z updates the duals from s.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <cmath>
#include <cstdint>

#include "kernels.h"
#include "project_dev.cuh"
#include "project_reg.cuh"
#include "ptx.cuh"

namespace sparkling {

namespace {

constexpr int kProjMaxThreads = 1024;
constexpr size_t kProjSmemMax = 200 * 1024;

template <typename KT>
__global__ void __launch_bounds__(kProjMaxThreads) project_kernel(const ProjArgs p)
{
    extern __shared__ __align__(16) double psm[];
    const int Ns = p.Ns;
    double *base = p.gstate ? p.gstate + (size_t)blockIdx.x * 18 * (size_t)Ns : psm;
    const Arrays A = carve(base, Ns);
    ShotParams sp;
    sp.Ns = Ns;
    sp.alpha = p.alpha; sp.beta = p.beta; sp.box = p.box; sp.tol = p.tol; sp.margin = p.margin;
    for (int c = 0; c < 3; ++c) sp.pin[c] = p.pin[c];
    sp.pin_index = p.pin_index; sp.n_iter = p.n_iter; sp.check_every = p.check_every;
    sp.viol = p.viol; sp.notconv = p.notconv;
    KT *K = static_cast<KT *>(p.K);
    for (int64_t shot = blockIdx.x; shot < p.Nc; shot += gridDim.x) {
        const int64_t off = shot * (int64_t)Ns;
        const double *G = p.G;
        const double eta = p.eta;
        auto loadk = [&](int m, double *kv) {
            for (int c = 0; c < 3; ++c) {
                kv[c] = (double)K[3 * (off + m) + c];
                if (G) kv[c] -= eta * G[3 * (off + m) + c];
            }
        };
        if (sizeof(KT) == 4 && p.tol <= 0.0 && p.mixed) {
            // FP32 output, fixed iterations, asked for: the mixed-precision form
            project_shot_mixed<KT>(carve_f(reinterpret_cast<float *>(base), Ns), K + 3 * off, sp,
                                   loadk);
            if (p.viol) record_violation<KT>(K + 3 * off, sp);
        } else {
            project_shot<KT>(A, K + 3 * off, sp, loadk);
        }
    }
}

// Threads a CTA of the register form may have: M = 1 takes 80 registers a
// thread, M = 2 takes 128.
constexpr __host__ __device__ int reg_max_threads(int M) { return M == 1 ? 768 : 512; }
constexpr int kRegMaxCtas = 8;                 // portable cluster size

// How the CTAs of one shot meet.
constexpr int kAlone = 0;        // one CTA
constexpr int kMeet = 1;         // edges through distributed shared memory, two cluster barriers an iteration
// A CTA also computes the samples of a halo of its neighbours, whose edge
// spoils two samples an iteration, and the halos' state is copied from their
// owners every (halo - 2) / 2 iterations: for shots that leave the GPU idle,
// where a cluster barrier (~0.5 us) in every iteration would cost as much as
// the iteration.
constexpr int kHalo = 2;
constexpr int kMaxHalo = 32;

// The slots and neighbours of the calling warp; zeroed, and every CTA of the
// cluster running, on return.
template <class R, int M, int CL> struct RegEdges {
    typedef typename VecOf<R>::type V;
    struct Shared {
        EdgeSlot<R> slots[reg_max_threads(M) / 32];
        V band[CL == kHalo ? 2 : 1][CL == kHalo ? 4 : 1][CL == kHalo ? kMaxHalo : 1];
    };
    Shared *sh;
    EdgeSlot<R> *mine, *to_right = nullptr, *to_left = nullptr;
    bool first, last;
    int C, rank, own, halo;

    __device__ RegEdges(Shared *s, const RegShape &shape) : sh(s), own(shape.own), halo(shape.halo)
    {
        namespace cg = cooperative_groups;
        const cg::cluster_group cl = cg::this_cluster();
        C = CL ? (int)cl.num_blocks() : 1;
        rank = CL ? (int)cl.block_rank() : 0;
        const int warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
        first = (CL != kMeet || rank == 0) && warp == 0;
        last = (CL != kMeet || rank == C - 1) && warp == warps - 1;
        mine = &s->slots[warp];
        if (warp < warps - 1) to_right = &s->slots[warp + 1];
        else if (CL == kMeet && !last) to_right = cl.map_shared_rank(&s->slots[0], rank + 1);
        if (warp > 0) to_left = &s->slots[warp - 1];
        else if (CL == kMeet && !first) to_left = cl.map_shared_rank(&s->slots[warps - 1], rank - 1);
        for (int q = threadIdx.x; q < warps * kSlotWords; q += blockDim.x)
            reinterpret_cast<double *>(s->slots)[q] = 0.0;
        cluster_sync();
    }
    __device__ __forceinline__ static void cta_sync()
    {
        if (blockDim.x == 32) __syncwarp();
        else __syncthreads();
    }
    __device__ __forceinline__ static void cluster_sync()
    {
        if (CL) cooperative_groups::this_cluster().sync();
        else cta_sync();
    }
    // First sample of the thread; kHalo: the CTA owns [rank * own, (rank + 1) * own)
    // and begins `halo` before them.
    __device__ int first_sample() const
    {
        if (CL == kHalo) return (rank ? rank * own - halo : 0) + (int)threadIdx.x * M;
        return (rank * (int)blockDim.x + (int)threadIdx.x) * M;
    }
    __device__ __forceinline__ bool owns(int m) const
    {
        return CL != kHalo || (m >= rank * own && m < (rank + 1) * own);
    }

    // Every (halo - 2) / 2 iterations: the owners' state of the halos' samples.
    // (Before the first one, too: no CTA may store its result over samples that a
    // neighbour has still to load for its halo.)
    __device__ __forceinline__ void refresh(int it, int m0, V *y1, V *y2, V *w1, V *w2)
    {
        if (CL != kHalo || (it + 1) % ((halo - 2) / 2) != 0) return;
        namespace cg = cooperative_groups;
        const cg::cluster_group cl = cg::this_cluster();
        const int lo = rank * own, hi = lo + own;
        // the samples that a neighbour's halo holds: band 0 our first ones, band 1 our last
#pragma unroll
        for (int j = 0; j < M; ++j) {
            const int m = m0 + j;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int i = e == 0 ? m - lo : m - (hi - halo);
                if (m >= lo && m < hi && i >= 0 && i < halo) {
                    sh->band[e][0][i] = y1[j];
                    sh->band[e][1][i] = y2[j];
                    sh->band[e][2][i] = w1[j];
                    sh->band[e][3][i] = w2[j];
                }
            }
        }
        cl.sync();
#pragma unroll
        for (int j = 0; j < M; ++j) {
            const int m = m0 + j;
            const bool before = m < lo, after = m >= hi && m < hi + halo && rank < C - 1;
            if (before || after) {
                const Shared *from = cl.map_shared_rank(sh, before ? rank - 1 : rank + 1);
                const V(*b)[kMaxHalo] = reinterpret_cast<const V(*)[kMaxHalo]>(from->band[before ? 1 : 0]);
                const int i = before ? m - (lo - halo) : m - hi;
                y1[j] = b[0][i];
                y2[j] = b[1][i];
                w1[j] = b[2][i];
                w2[j] = b[3][i];
            }
        }
        cl.sync();             // the bands may be written again
    }

    template <class LoadK, class Store>
    __device__ __forceinline__ void project(const RegShot &sh_, const MomentumTables &mom,
                                            LoadK loadk, Store store)
    {
        const int m0 = first_sample();
        project_registers<R, M>(
            sh_, mom, m0, mine, to_right, to_left, first, last,
            [] { if (CL == kMeet) cluster_sync(); else cta_sync(); },
            [&](int it, V *y1, V *y2, V *w1, V *w2) {
                refresh(it, m0, y1, y2, w1, w2);
            },
            loadk, [&](int m, const V &s) { if (owns(m)) store(m, s); });
        cluster_sync();        // the slots are free again (and no CTA leaves early)
    }
};

// One shot per cluster (CL) or CTA, grid-stride over shots; thread t of CTA
// rank r owns samples (r * blockDim + t) * M + [0, M).
template <class R, int M, typename KT, int CL>
__global__ void __launch_bounds__(reg_max_threads(M)) project_reg_kernel(const ProjArgs p,
                                                                         const RegShape shape)
{
    __shared__ typename RegEdges<R, M, CL>::Shared shared;
    RegEdges<R, M, CL> edges(&shared, shape);
    RegShot sh;
    // a lone sample has no rows: its projection is the clip (or the pin)
    sh.Ns = p.Ns; sh.n_iter = p.Ns > 1 ? p.n_iter : 0; sh.pin_index = p.pin_index;
    sh.alpha = p.alpha; sh.beta = p.beta; sh.box = p.box;
    for (int c = 0; c < 3; ++c) sh.pin[c] = p.pin[c];
    KT *K = static_cast<KT *>(p.K);
    const double *G = p.G;
    const double eta = p.eta;
    for (int64_t shot = blockIdx.x / edges.C; shot < p.Nc; shot += gridDim.x / edges.C) {
        const int64_t off = shot * (int64_t)p.Ns;
        edges.project(sh, p.mom,
            [&](int m, double *kv) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    kv[c] = (double)K[3 * (off + m) + c];
                    if (G) kv[c] -= eta * G[3 * (off + m) + c];
                }
            },
            [&](int m, const typename VecOf<R>::type &s) {
                KT o[3];
                v_values(s, o);
#pragma unroll
                for (int c = 0; c < 3; ++c) K[3 * (off + m) + c] = o[c];
            });
    }
}

// The shots of a batch's trajectories (FP32 samples), after the engine: the
// gradient is formed from the trajectory's slots and repulsion totals in the
// order of the engine's projection items.  A trajectory whose pair items did
// not all finish (a bounded wait ran out) is left as it is.
template <int M, int CL>
__global__ void __launch_bounds__(reg_max_threads(M)) project_batch_kernel(const EngineArgs e,
                                                                           int B, int64_t shots,
                                                                           int Ns,
                                                                           MomentumTables mom,
                                                                           const RegShape shape)
{
    __shared__ typename RegEdges<Df, M, CL>::Shared shared;
    RegEdges<Df, M, CL> edges(&shared, shape);
    for (int64_t shot = blockIdx.x / edges.C; shot < shots; shot += gridDim.x / edges.C) {
        int lo = 0, hi = B - 1;                   // the largest t with off_t <= shot * Ns
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (e.traj[mid].off <= shot * Ns) lo = mid;
            else hi = mid - 1;
        }
        const EngineTraj &tr = e.traj[lo];
        if (e.done[lo] < (unsigned int)tr.n_pair_items) continue;   // the whole cluster alike
        RegShot sh;
        sh.Ns = Ns; sh.n_iter = Ns > 1 ? tr.n_iter : 0; sh.pin_index = tr.pin_index;
        sh.alpha = tr.alpha; sh.beta = tr.beta; sh.box = tr.box;
        for (int c = 0; c < 3; ++c) sh.pin[c] = tr.pin[c];
        float *K = static_cast<float *>(e.K) + 3 * shot * (int64_t)Ns;
        const int64_t first = shot * Ns - tr.off;               // local sample index
        const dacc4 *part = e.part + tr.part_off;
        const double invN = 1.0 / (double)tr.N, eta = tr.eta;
        const int slots_n = tr.slots, ach = tr.a_chunks;
        edges.project(sh, mom,
            [&](int m, double *kv) {
                const int64_t i = first + m, tile = i / kTile, l = i - tile * kTile;
                const dacc4 *p = part + tile * slots_n * kTile + l;
                double g[3] = {0.0, 0.0, 0.0}, r[3] = {0.0, 0.0, 0.0};
                for (int s = 0; s < slots_n; ++s) {
                    const dacc4 v = p[(int64_t)s * kTile];
                    if (s < ach) { g[0] += v.x; g[1] += v.y; g[2] += v.z; }
                    else { r[0] += v.x; r[1] += v.y; r[2] += v.z; }
                }
                if (e.racc) {
                    const unsigned long long *q = e.racc + 3 * (tr.off + i);
                    for (int c = 0; c < 3; ++c) r[c] = (double)(long long)q[c] / kFixScale;
                }
                for (int c = 0; c < 3; ++c) kv[c] = (double)K[3 * m + c] - eta * (g[c] - r[c] * invN);
            },
            [&](int m, const VecDf &s) {
                float o[3];
                v_values(s, o);
#pragma unroll
                for (int c = 0; c < 3; ++c) K[3 * m + c] = o[c];
            });
    }
}

// Violations of the result: the maxima are taken over all samples, so a block
// reduces once.  Shots of 256 samples and more are taken block by block; of
// shorter ones a block holds many, a thread a sample.
template <typename KT>
__global__ void __launch_bounds__(256) violation_kernel(const ProjArgs p)
{
    ShotParams sp;
    sp.Ns = p.Ns;
    sp.alpha = p.alpha; sp.beta = p.beta; sp.box = p.box; sp.tol = 0.0; sp.margin = 0.0;
    for (int c = 0; c < 3; ++c) sp.pin[c] = p.pin[c];
    sp.pin_index = p.pin_index; sp.n_iter = p.n_iter; sp.check_every = 0;
    sp.viol = p.viol; sp.notconv = nullptr;
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    const KT *K = static_cast<const KT *>(p.K);
    if (p.Ns >= (int)blockDim.x) {
        for (int64_t shot = blockIdx.x; shot < p.Nc; shot += gridDim.x)
            for (int n = threadIdx.x; n < p.Ns; n += blockDim.x)
                sample_violation<KT>(K + 3 * shot * p.Ns, n, sp, v);
    } else {
        const unsigned int first = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
        const int dshot = (int)(step / (unsigned int)p.Ns), dn = (int)(step % (unsigned int)p.Ns);
        int64_t shot = first / (unsigned int)p.Ns;
        int n = (int)(first % (unsigned int)p.Ns);
        while (shot < p.Nc) {
            sample_violation<KT>(K + 3 * shot * p.Ns, n, sp, v);
            shot += dshot;
            n += dn;
            if (n >= p.Ns) { n -= p.Ns; ++shot; }
        }
    }
    reduce_violation(v, sp);
}

template <int CL> void *reg_fn(int dtype, int M)
{
    if (dtype == 0)
        return M == 1 ? reinterpret_cast<void *>(project_reg_kernel<Df, 1, float, CL>)
                      : reinterpret_cast<void *>(project_reg_kernel<Df, 2, float, CL>);
    return M == 1 ? reinterpret_cast<void *>(project_reg_kernel<double, 1, double, CL>)
                  : reinterpret_cast<void *>(project_reg_kernel<double, 2, double, CL>);
}

} // namespace

bool project_reg_applies(int dtype, int Ns, double alpha, double beta, double box, double tol,
                         const double *pin, int pin_index, int n_iter)
{
    if (tol > 0.0 || n_iter > kMomentumMax || Ns > kRegMaxCtas * 2 * reg_max_threads(2)) return false;
    // radii whose squares are normal numbers (a row's square above them is, too)
    if (dtype != 0) return alpha >= 1e-150 && beta >= 1e-150;
    // two-float form: radii and box whose squares and low parts stay normal
    constexpr double lo = 1.0 / (1ll << 40), hi = (double)(1ll << 40);
    auto radius_ok = [&](double r) { return std::isinf(r) || (r >= lo && r <= hi); };
    if (!radius_ok(alpha) || !radius_ok(beta) || !(box >= lo && box <= hi)) return false;
    for (int c = 0; c < 3; ++c)
        if (pin_index >= 0 && !(std::fabs(pin[c]) <= hi)) return false;
    return true;
}

namespace {

// Shape of one shot over C CTAs with halos (at least 8 samples, 3 iterations
// between copies); false where it does not fit.
bool reg_halo_shape(int Ns, int M, int C, RegShape &s)
{
    const int sides = C == 2 ? 1 : 2;            // of two CTAs each has one neighbour
    s.per_thread = M;
    s.ctas = C;
    s.own = (Ns + C - 1) / C;
    s.threads = ((s.own + 8 * sides + M - 1) / M + 31) / 32 * 32;
    s.halo = (s.threads * M - s.own) / sides;
    s.halo = s.halo < kMaxHalo ? s.halo : kMaxHalo;
    s.halo = s.halo < s.own ? s.halo : s.own;
    // every CTA owns samples, and the last one holds what its neighbour needs
    return s.threads <= reg_max_threads(M) && s.halo >= 8 && Ns - (C - 1) * s.own >= s.halo;
}

// Time of 100 iterations (us) where an SM has `load` CTAs: a chain's latency,
// or the issue of the SM's warps (FP64: of its FP64 pipe); ~0.5 us a cluster
// barrier, of which a shape with halos has two a copy.  Fitted to shots of
// 64 .. 2560 samples, load 1.
double reg_time(bool fp64, const RegShape &s, double load = 1.0)
{
    const double w = load * (s.threads / 32);
    const bool one = s.per_thread == 1;
    const double chain = fp64 ? (one ? 310.0 : 550.0) : one ? 88.0 : 108.0;
    const double warp = fp64 ? (one ? 72.0 : 122.0) : one ? 14.0 : 19.0;
    const double barriers = s.halo ? 300.0 / ((s.halo - 2) / 2) : s.ctas > 1 ? 90.0 : 0.0;
    return (w * warp > chain ? w * warp : chain) + barriers;
}

} // namespace

// Shape rule.  Two floats (FP32 samples): issue-bound, so M = 2 (the fewest
// instructions a sample), and CTAs of at most 256 threads -- two on an SM
// cover each other's barriers: 4096 shots of 2560 samples take 21.9 ms as 5
// CTAs of 256 threads (before x and y were paired: 24.5 ms, and 30.1 ms as 3 of
// 448).  Shots of up to 128 samples are bound by the latency of one warp's
// chain: M = 1 (32 x 64: 86 against 107 us, then too).
// FP64: bound by the FP64 pipe, which every warp of an SM shares.  M = 1 costs
// ~10 % more operations but pads less and has the shorter chain: the times
// above decide, with the CTAs that fall to an SM (37 x 129: 379 against 531 us;
// 300 x 700: 2.80 against 2.53 ms; 20000 x 32, half a warp at M = 2: 7.6
// against 15.0 ms; 300 x 96: 428 against 561 us).  One CTA up to 1024 samples (a cluster barrier
// costs ~0.4 us: 300 x 700 as 2 CTAs takes 2.79 ms), else at most 256 threads.
// Few shots (`halos`; every CTA with an SM to itself): more, smaller CTAs a
// shot with halos, as the times above say.  FP64 8 x 1000 1891 -> 410 us, 20 x
// 500 985 -> 338, 37 x 129 381 -> 315; FP32 1 x 512 164 -> 120, 8 x 2560 238 -> 184.
RegShape project_reg_shape(int dtype, int64_t Nc, int Ns, int sms, bool halos)
{
    RegShape s;
    const bool fp64 = dtype != 0;
    const int one = fp64 ? 1024 : 512;            // samples a single CTA takes
    s.ctas = Ns <= one ? 1 : (Ns + 511) / 512;
    if (s.ctas > kRegMaxCtas) s.ctas = kRegMaxCtas;
    auto with = [&](int M) {
        RegShape t = s;
        t.per_thread = M;
        const int per = s.ctas * M;
        t.threads = ((Ns + per - 1) / per + 31) / 32 * 32;
        return t;
    };
    if (fp64 && s.ctas == 1 && Ns <= reg_max_threads(1)) {
        const double load = (double)((Nc + sms - 1) / sms);
        s = reg_time(true, with(1), load) <= reg_time(true, with(2), load) ? with(1) : with(2);
    } else {
        s = with(!fp64 && Ns <= 128 ? 1 : 2);
    }
    if (!halos) return s;
    double best = 0.95 * reg_time(fp64, s);
    for (int M = 1; M <= 2; ++M)
        for (int C = 2; C <= kRegMaxCtas && Nc * C <= sms; ++C) {
            RegShape h;
            if (!reg_halo_shape(Ns, M, C, h)) continue;
            const double t = reg_time(fp64, h);
            if (t < best) {
                best = t;
                s = h;
            }
        }
    return s;
}

namespace {

cudaError_t launch_reg(void *fn, const RegShape &s, int64_t shots, void **args, cudaStream_t st)
{
    cudaLaunchConfig_t cfg{};
    const int64_t most = ((int64_t)1 << 20) / s.ctas;
    cfg.gridDim = dim3((unsigned)((shots < most ? shots : most) * s.ctas));
    cfg.blockDim = dim3((unsigned)s.threads);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)s.ctas;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = s.ctas > 1 ? 1 : 0;
    return cudaLaunchKernelExC(&cfg, fn, args);
}

} // namespace

cudaError_t launch_project_batch(const EngineArgs &e, int32_t B, int64_t shots, int Ns,
                                 const MomentumTables &mom, const RegShape &s, cudaStream_t st)
{
    void *fn = s.ctas > 1 ? (s.per_thread == 1 ? reinterpret_cast<void *>(project_batch_kernel<1, kMeet>)
                                               : reinterpret_cast<void *>(project_batch_kernel<2, kMeet>))
                          : (s.per_thread == 1 ? reinterpret_cast<void *>(project_batch_kernel<1, kAlone>)
                                               : reinterpret_cast<void *>(project_batch_kernel<2, kAlone>));
    int b = B;
    MomentumTables m = mom;
    void *args[] = {const_cast<EngineArgs *>(&e), &b, &shots, &Ns, &m, const_cast<RegShape *>(&s)};
    return launch_reg(fn, s, shots, args, st);
}

cudaError_t launch_project_reg(const ProjArgs &p, int dtype, const RegShape &s, int sms,
                               cudaStream_t st)
{
    void *fn = s.halo ? reg_fn<kHalo>(dtype, s.per_thread)
               : s.ctas > 1 ? reg_fn<kMeet>(dtype, s.per_thread) : reg_fn<kAlone>(dtype, s.per_thread);
    void *args[] = {const_cast<ProjArgs *>(&p), const_cast<RegShape *>(&s)};
    cudaError_t e = launch_reg(fn, s, p.Nc, args, st);
    if (e != cudaSuccess || !p.viol) return e;
    // a block an SM (a sample takes ~4 us of FP64 latency); more, for the width,
    // only with two samples a thread, as a block's reduction costs about one
    const int64_t total = p.Nc * p.Ns, one = (total + 255) / 256, two = (total + 511) / 512;
    int64_t g = two < (int64_t)sms * 4 ? two : (int64_t)sms * 4;
    if (g < sms) g = one < sms ? one : sms;
    if (p.Ns >= 256) g = p.Nc < (int64_t)sms * 8 ? p.Nc : (int64_t)sms * 8;
    if (dtype == 0) violation_kernel<float><<<(unsigned)g, 256, 0, st>>>(p);
    else violation_kernel<double><<<(unsigned)g, 256, 0, st>>>(p);
    return cudaGetLastError();
}

size_t project_state_bytes(int Ns) { return (size_t)18 * Ns * sizeof(double); }

bool project_state_in_smem(int Ns) { return project_state_bytes(Ns) <= kProjSmemMax; }

int project_block(int Ns)
{
    int b = ((Ns + 31) / 32) * 32;
    if (b > kProjMaxThreads) b = kProjMaxThreads;
    if (b < 32) b = 32;
    return b;
}

int project_ctas_per_sm(int dtype, int Ns)
{
    void *fn = dtype == 0 ? reinterpret_cast<void *>(project_kernel<float>)
                          : reinterpret_cast<void *>(project_kernel<double>);
    const size_t smem = project_state_in_smem(Ns) ? project_state_bytes(Ns) : 0;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kProjSmemMax) !=
        cudaSuccess)
        return 0;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, project_block(Ns), smem) != cudaSuccess)
        return 0;
    return n;
}

cudaError_t launch_project(const ProjArgs &p, int dtype, int grid, cudaStream_t st)
{
    void *fn = dtype == 0 ? reinterpret_cast<void *>(project_kernel<float>)
                          : reinterpret_cast<void *>(project_kernel<double>);
    const size_t smem = p.gstate ? 0 : project_state_bytes(p.Ns);
    void *args[] = {const_cast<ProjArgs *>(&p)};
    return cudaLaunchKernel(fn, dim3((unsigned)grid), dim3(project_block(p.Ns)), args, smem, st);
}

} // namespace sparkling
