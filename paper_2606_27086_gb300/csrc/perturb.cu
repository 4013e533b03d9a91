// Perturbation phase of Algorithm 1 (nonascending subgradient steps with the
// power-law step size beta = gamma * alpha^l of Sec. 2.1.2) and the objective
// evaluations it needs: isotropic TV (Eq. (TV)) with the Combettes/Penfold
// subgradient, anisotropic TV, and the linear mean dose f = c.x (Sec. 2.3.3).
//
// One thread-block cluster owns one right-hand side.  Every trial needs a
// global decision f(z) <= f(y); the cluster makes it without the host: each
// CTA reduces its FP64 partial in a fixed order, the partials are exchanged
// through distributed shared memory after a hardware cluster barrier, and
// every CTA sums them in the same order -- so all CTAs take the same decision
// and the run is bitwise reproducible.  The trial loop is bounded by
// max_trials, so the kernel always ends.
#include <algorithm>
#include <type_traits>

#include <cooperative_groups.h>

#include "check.cuh"
#include "common.cuh"

namespace cg = cooperative_groups;

namespace suppy {

cudaError_t read_check_word_perturb(int* out3) { return take_check_words(out3); }

namespace {

// Strided view of right-hand side b of an n x B row-major array.  Reads go
// through L2 only (ld.global.cg): other CTAs of the cluster rewrite these
// vectors between the passes of one launch, and L2 is the coherence point.
struct Vec {
    float* p;
    int B;
    __device__ __forceinline__ float operator()(int j) const { return __ldcg(p + (size_t)j * B); }
};

// z = y - s * g, the trial point, computed identically wherever it is used.
__device__ __forceinline__ float trial(float y, float g, float s) { return __fmaf_rn(-s, g, y); }

// Trial step beta / ||g|| with beta = gamma alpha^l (Sec. 2.1.2).  The
// exponent is split in FP64, alpha^l = 2^(l log2 alpha) = 2^k 2^f with k an
// integer and f in [0, 1), and the rest is FP32, so the relative error stays
// at a few FP32 ulps for any l.  (FP64 on GB300 costs tens of cycles per
// dependent operation; an FP64 pow() takes microseconds, on the critical
// path of every trial.)
__device__ __forceinline__ float trial_scale(double gamma, double log2_alpha, long long ell,
                                             float inv_gnorm) {
    const double e = (double)ell * log2_alpha;
    const double k = floor(e);
    const float f = (float)(e - k);
    return (float)gamma * ldexpf(exp2f(f), (int)k) * inv_gnorm;
}

// Adaptive step of Nikazad et al. (Sec. 2.1.2): the reference value of a
// phase that starts at f_start -- fixed, or the lowest phase-start objective
// so far, this one included -- and beta / ||g|| = (f - f_ref) / ||g||^2, the
// subgradient projection onto the level set of f's linearisation.
__device__ __forceinline__ double adaptive_ref(const PerturbArgs& a, bool has_ref, double st_ref,
                                               double f_start) {
    if (a.adaptive == 2) return a.f_ref;
    return has_ref ? fmin(st_ref, f_start) : f_start;
}

__device__ __forceinline__ float adaptive_scale(double fy, double f_ref, double gg) {
    return fy > f_ref ? (float)((fy - f_ref) / gg) : 0.f;
}

// Objectives whose value is a sum of per-element terms (no stencil): the
// linear mean dose c.x, ||x||_1 and ||x||_2^2.
__device__ __forceinline__ bool elementwise(int obj) {
    return obj == SUPPY_OBJ_LINEAR || obj == SUPPY_OBJ_L1 || obj == SUPPY_OBJ_L2;
}

// Term and (sub)gradient of ||x||_1 (sign, 0 at 0) and ||x||_2^2 (2x).
__device__ __forceinline__ float norm_term(int obj, float v) {
    return obj == SUPPY_OBJ_L1 ? fabsf(v) : v * v;
}
__device__ __forceinline__ float norm_grad(int obj, float v) {
    if (obj == SUPPY_OBJ_L1) return (v > 0.f) ? 1.f : ((v < 0.f) ? -1.f : 0.f);
    return 2.f * v;
}

// Objective term owned by pixel p (FP64 result; TV terms are FP32 then widened).
template <class Y>
__device__ __forceinline__ double obj_term(int obj, int p, int H, int W, const double* c64,
                                           const Y& y) {
    if (obj == SUPPY_OBJ_LINEAR) return c64[p] * (double)y(p);
    if (obj == SUPPY_OBJ_L1 || obj == SUPPY_OBJ_L2) return (double)norm_term(obj, y(p));
    const int i = p / W, j = p - i * W;
    const float y0 = y(p);
    if (obj == SUPPY_OBJ_TV_ISO) {
        if (i < H - 1 && j < W - 1) {
            const float dx = y(p + W) - y0, dy = y(p + 1) - y0;
            return (double)sqrtf(dx * dx + dy * dy);
        }
        return 0.0;
    }
    float t = 0.f;   // anisotropic
    if (i < H - 1) t += fabsf(y(p + W) - y0);
    if (j < W - 1) t += fabsf(y(p + 1) - y0);
    return (double)t;
}

__device__ __forceinline__ float sgnf(float v) { return (v > 0.f) ? 1.f : ((v < 0.f) ? -1.f : 0.f); }

// Subgradient component at pixel p (gather form of the term-wise derivatives).
template <class Y>
__device__ __forceinline__ float subgrad(int obj, int p, int H, int W, const float* c32,
                                         const Y& y) {
    if (obj == SUPPY_OBJ_LINEAR) return c32[p];
    if (obj == SUPPY_OBJ_L1 || obj == SUPPY_OBJ_L2) return norm_grad(obj, y(p));
    const int i = p / W, j = p - i * W;
    const float y0 = y(p);
    float g = 0.f;
    if (obj == SUPPY_OBJ_TV_ISO) {
        // term (i, j): d/dX[i,j] = -(dx + dy) / phi
        if (i < H - 1 && j < W - 1) {
            const float dx = y(p + W) - y0, dy = y(p + 1) - y0;
            const float phi = sqrtf(dx * dx + dy * dy);
            if (phi > 0.f) g -= (dx + dy) / phi;
        }
        // term (i-1, j): d/dX[i,j] = dx' / phi'  (X[i,j] is its X[i'+1,j])
        if (i > 0 && j < W - 1) {
            const float ym = y(p - W);
            const float dx = y0 - ym, dy = y(p - W + 1) - ym;
            const float phi = sqrtf(dx * dx + dy * dy);
            if (phi > 0.f) g += dx / phi;
        }
        // term (i, j-1): d/dX[i,j] = dy'' / phi''  (X[i,j] is its X[i,j'+1])
        if (j > 0 && i < H - 1) {
            const float yl = y(p - 1);
            const float dx = y(p + W - 1) - yl, dy = y0 - yl;
            const float phi = sqrtf(dx * dx + dy * dy);
            if (phi > 0.f) g += dy / phi;
        }
        return g;
    }
    if (i < H - 1) g -= sgnf(y(p + W) - y0);
    if (i > 0) g += sgnf(y0 - y(p - W));
    if (j < W - 1) g -= sgnf(y(p + 1) - y0);
    if (j > 0) g += sgnf(y0 - y(p - 1));
    return g;
}

// dx^2 + dy^2 with one rounding order wherever a TV term is formed, so that
// equal images give equal objective values.
__device__ __forceinline__ float sq2(float dx, float dy) { return __fmaf_rn(dx, dx, __fmul_rn(dy, dy)); }

// Per-thread compensated FP32 sum (Kahan), handed to the CTA and cluster
// reductions as a float-float value.  FP64 arithmetic is scarce on GB300: one
// FP64 add per pixel and pass would cost more than the stencil itself.
struct KSum {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float v) {
        const float y = v - c;
        const float t = s + y;
        c = (t - s) - y;
        s = t;
    }
};

// Float-float value hi + lo (about 44 significant bits): CTA-level sums of the
// per-thread compensated FP32 sums stay in FP32 arithmetic, and FP64 is used
// only for the grid-level sum of the CTA partials.
struct FF {
    float hi, lo;
};

__device__ __forceinline__ FF ff_add(FF a, FF b) {
    const float s = a.hi + b.hi;
    const float bb = s - a.hi;
    const float e = (a.hi - (s - bb)) + (b.hi - bb) + (a.lo + b.lo);
    const float hi = s + e;
    return FF{hi, e - (hi - s)};
}

__device__ __forceinline__ FF ff_of(const KSum& k) { return FF{k.s, -k.c}; }

// An FP64 value as float-float (used for the FP64 per-element sums of the
// linear objective).
__device__ __forceinline__ FF ff_of(double v) {
    const float hi = (float)v;
    return FF{hi, (float)(v - (double)hi)};
}

// Deterministic cluster-wide sum of two values: float-float over the lanes
// and then the warps of each CTA (FP32 arithmetic), then one thread per CTA
// sums the cluster's CTA values in FP64 in rank order.  Every thread gets the
// same result, read from shared memory.  FP64 stays with one thread per CTA:
// it is scarce on GB300.
__device__ double2 cluster_sum2(FF a, FF b, FF* swf, double2* scta, double2* sres,
                                cg::cluster_group& cluster) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a = ff_add(a, FF{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)});
        b = ff_add(b, FF{__shfl_xor_sync(0xffffffffu, b.hi, o), __shfl_xor_sync(0xffffffffu, b.lo, o)});
    }
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
        swf[2 * wid] = a;
        swf[2 * wid + 1] = b;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        FF sa{0.f, 0.f}, sb{0.f, 0.f};
        for (int w = 0; w < kPerturbThreads / 32; ++w) {
            sa = ff_add(sa, swf[2 * w]);
            sb = ff_add(sb, swf[2 * w + 1]);
        }
        *scta = make_double2((double)sa.hi + (double)sa.lo, (double)sb.hi + (double)sb.lo);
    }
    cluster.sync();
    if (threadIdx.x == 0) {
        double2 t = make_double2(0.0, 0.0);
        const unsigned nr = cluster.num_blocks();
        for (unsigned r = 0; r < nr; ++r) {
            const double2 v = *cluster.map_shared_rank(scta, r);
            t.x += v.x;
            t.y += v.y;
        }
        *sres = t;
    }
    cluster.sync();   // every CTA has read scta; sres is visible to the CTA
    return *sres;
}

// Scalar decisions of a reduction step, taken by one thread after the
// subgradient pass and shared through shared memory: whether the step goes
// on, 1/||g|| and the adaptive step.
struct StepDecision {
    int go;
    float inv_gnorm, asc;
};

__device__ __forceinline__ StepDecision step_decision(const PerturbArgs& a, bool has_ref, double st_ref,
                                                      double gg, double fy, double f_start) {
    StepDecision d{0, 0.f, 0.f};
    if (a.record_only || gg == 0.0) return d;
    d.inv_gnorm = 1.0f / sqrtf((float)gg);
    if (a.adaptive) {
        const double f_ref = adaptive_ref(a, has_ref, st_ref, f_start);
        if (!(fy > f_ref)) return d;
        d.asc = adaptive_scale(fy, f_ref, gg);
    }
    d.go = 1;
    return d;
}

// Where a perturbation phase starts: the restart rule (Sec. 2.1.2: l <- r at
// the r-th restart) applied to the exponent and the restart state.
struct PhaseStart {
    long long ell;
    int restarts, last_restart_k;
};

__device__ __forceinline__ PhaseStart phase_start(const PerturbArgs& a, int b) {
    const RhsState& st = a.st[b];
    PhaseStart ps;
    ps.ell = st.ell;
    ps.restarts = st.restarts;
    ps.last_restart_k = st.last_restart_k;
    const int k = st.k;
    if (!a.record_only && a.restart_every > 0 && k > 0 && k % a.restart_every == 0 &&
        ps.last_restart_k != k) {
        ps.restarts += 1;
        ps.ell = ps.restarts;
        ps.last_restart_k = k;
    }
    return ps;
}

// Bookkeeping at the end of a phase: f at its start, exponent, restart
// state, counts of this phase and in total.
__device__ __forceinline__ void phase_end(const PerturbArgs& a, RhsState& st, const PhaseStart& ps,
                                          long long ell, int accepted, int trials, double f_start) {
    st.f_cur = f_start;
    st.f_valid = 1;
    if (a.record_only) return;
    if (a.adaptive == 1) {
        st.f_ref = adaptive_ref(a, st.has_ref != 0, st.f_ref, f_start);
        st.has_ref = 1;
    }
    st.ell = ell;
    st.restarts = ps.restarts;
    st.last_restart_k = ps.last_restart_k;
    st.accepted_last = accepted;
    st.trials_last = trials;
    st.accepted_total += accepted;
    st.trials_total += trials;
}

__global__ void __launch_bounds__(kPerturbThreads) k_perturb(const PerturbArgs a) {
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ FF swf[2 * (kPerturbThreads / 32)];
    __shared__ double2 scta, sres;
    __shared__ StepDecision dec;
    __shared__ float sc_s;
    const int ncl = (int)cluster.num_blocks();
    const int b = blockIdx.x / ncl;             // right-hand side of this cluster
    RhsState& st = a.st[b];
    if (st.stopped) return;                     // uniform over the cluster
    const int rank = (int)cluster.block_rank();
    const int tid = rank * kPerturbThreads + threadIdx.x;
    const int nthr = ncl * kPerturbThreads;
    const int n = a.n, H = a.H, W = a.W, obj = a.obj;
    const bool lin = (obj == SUPPY_OBJ_LINEAR);
    Vec y{a.x + b, a.B};
    Vec g{a.g + b, a.B};

    const PhaseStart ps = phase_start(a, b);
    // read before the first barrier: rank 0 rewrites it at the phase's end
    const bool has_ref = st.has_ref != 0;
    const double st_ref = st.f_ref;
    long long ell = ps.ell;
    int accepted = 0, trials = 0;
    double f_start = 0.0;   // thread 0 of each CTA
    bool have_f = false;
    for (int s = 0; s < (a.record_only ? 1 : a.n_red); ++s) {
        // pass G: subgradient, ||g||^2 and f(y) (the linear objective's terms
        // in FP64, the others compensated FP32)
        KSum kg, kf;
        double fl = 0.0;
        for (int p = tid; p < n; p += nthr) {
            const double t = obj_term(obj, p, H, W, a.c64, y);
            if (lin) fl += t;
            else kf.add((float)t);
            if (!a.record_only) {
                const float gp = subgrad(obj, p, H, W, a.c32, y);
                __stcg(g.p + (size_t)p * a.B, gp);
                kg.add(gp * gp);
            }
        }
        const double2 r = cluster_sum2(ff_of(kg), lin ? ff_of(fl) : ff_of(kf), swf, &scta, &sres,
                                       cluster);
        const double fy = r.y;
        if (threadIdx.x == 0) {
            if (!have_f) {
                f_start = fy;
                have_f = true;
            }
            dec = step_decision(a, has_ref, st_ref, r.x, fy, f_start);
        }
        __syncthreads();
        if (!dec.go) break;
        const float inv_gnorm = dec.inv_gnorm, asc = dec.asc;
        bool ok = false;
        const int jmax = a.adaptive ? 1 : a.max_trials;
        for (int j = 0; j < jmax; ++j) {
            if (threadIdx.x == 0)
                sc_s = a.adaptive ? asc : trial_scale(a.gamma, a.log2_alpha, ell, inv_gnorm);
            __syncthreads();
            const float sc = sc_s;
            if (!a.adaptive) ell += 1;
            trials += 1;
            Vec yy = y;
            Vec gv = g;
            auto z = [yy, gv, sc](int q) { return trial(yy(q), gv(q), sc); };
            KSum kz;
            double fzl = 0.0;
            for (int p = tid; p < n; p += nthr) {
                const double t = obj_term(obj, p, H, W, a.c64, z);
                if (lin) fzl += t;
                else kz.add((float)t);
            }
            const double fz =
                cluster_sum2(lin ? ff_of(fzl) : ff_of(kz), FF{0.f, 0.f}, swf, &scta, &sres, cluster).x;
            if (fz <= fy) {
                for (int p = tid; p < n; p += nthr) {
                    const size_t o = (size_t)p * a.B;
                    __stcg(y.p + o, trial(__ldcg(y.p + o), __ldcg(g.p + o), sc));
                }
                cluster.sync();
                accepted += 1;
                ok = true;
                break;
            }
        }
        if (!ok) break;
    }
    if (rank == 0 && threadIdx.x == 0) phase_end(a, st, ps, ell, accepted, trials, f_start);
}

// ------------------------------------------------------ stencil helpers ----
template <class Y>
__device__ __forceinline__ float tv_term(int obj, int i, int j, int H, int W, const Y& y) {
    const float y0 = y(i, j);
    if (obj == SUPPY_OBJ_TV_ISO) {
        if (i < H - 1 && j < W - 1) {
            const float dx = y(i + 1, j) - y0, dy = y(i, j + 1) - y0;
            return sqrtf(sq2(dx, dy));
        }
        return 0.f;
    }
    float t = 0.f;
    if (i < H - 1) t += fabsf(y(i + 1, j) - y0);
    if (j < W - 1) t += fabsf(y(i, j + 1) - y0);
    return t;
}

template <class Y>
__device__ __forceinline__ float tv_subgrad(int obj, int i, int j, int H, int W, const Y& y) {
    const float y0 = y(i, j);
    float g = 0.f;
    if (obj == SUPPY_OBJ_TV_ISO) {
        // each term contributes (its partial derivative) * 1/phi, phi = 0 -> 0
        if (i < H - 1 && j < W - 1) {
            const float dx = y(i + 1, j) - y0, dy = y(i, j + 1) - y0;
            const float q = sq2(dx, dy);
            if (q > 0.f) g -= (dx + dy) * rsqrtf(q);
        }
        if (i > 0 && j < W - 1) {
            const float ym = y(i - 1, j);
            const float dx = y0 - ym, dy = y(i - 1, j + 1) - ym;
            const float q = sq2(dx, dy);
            if (q > 0.f) g += dx * rsqrtf(q);
        }
        if (j > 0 && i < H - 1) {
            const float yl = y(i, j - 1);
            const float dx = y(i + 1, j - 1) - yl, dy = y0 - yl;
            const float q = sq2(dx, dy);
            if (q > 0.f) g += dy * rsqrtf(q);
        }
        return g;
    }
    if (i < H - 1) g -= sgnf(y(i + 1, j) - y0);
    if (i > 0) g += sgnf(y0 - y(i - 1, j));
    if (j < W - 1) g -= sgnf(y(i, j + 1) - y0);
    if (j > 0) g += sgnf(y0 - y(i, j - 1));
    return g;
}

// Row and column of element q of a strided loop over a row-major image (or
// band) of width W, advanced without a division per element: q grows by
// stride = si W + sj.
struct StrideWalk {
    int i, j, si, sj, W;
    __device__ StrideWalk(int q0, int stride, int w) : W(w) {
        i = q0 / w;
        j = q0 - i * w;
        si = stride / w;
        sj = stride - si * w;
    }
    __device__ __forceinline__ void next() {
        i += si;
        j += sj;
        if (j >= W) {
            j -= W;
            ++i;
        }
    }
};

// The values a TV term of pixel (i, j) reads at every trial point z = y - s g:
// y and g at (i, j), (i + 1, j) and (i, j + 1), loaded once per pixel.
struct TvNbr {
    float y0, g0, yd, gd, yr, gr;
    bool down, right;
};

__device__ __forceinline__ TvNbr tv_nbr(int i, int j, int H, int W, const float* y, const float* g,
                                        int B) {
    const size_t p = (size_t)i * W + j;
    TvNbr t;
    t.down = i < H - 1;
    t.right = j < W - 1;
    t.y0 = y[p * B];
    t.g0 = g[p * B];
    t.yd = t.down ? y[(p + W) * B] : 0.f;
    t.gd = t.down ? g[(p + W) * B] : 0.f;
    t.yr = t.right ? y[(p + 1) * B] : 0.f;
    t.gr = t.right ? g[(p + 1) * B] : 0.f;
    return t;
}

// TV term at the trial point with step s (computed as in the cluster kernels).
__device__ __forceinline__ float tv_trial_term(int obj, const TvNbr& t, float s) {
    const float z0 = trial(t.y0, t.g0, s);
    if (obj == SUPPY_OBJ_TV_ISO) {
        if (t.down && t.right) {
            const float dx = trial(t.yd, t.gd, s) - z0;
            const float dy = trial(t.yr, t.gr, s) - z0;
            return sqrtf(sq2(dx, dy));
        }
        return 0.f;
    }
    float v = 0.f;
    if (t.down) v += fabsf(trial(t.yd, t.gd, s) - z0);
    if (t.right) v += fabsf(trial(t.yr, t.gr, s) - z0);
    return v;
}

// -------------------------------------------------- tile-resident phase ----
// Same algorithm as k_perturb with every CTA's share of the image held in
// shared memory for the whole phase: the image is cut into a TR x TC grid of
// rectangles (element-wise objectives: into ranges), one per CTA, and a CTA
// loads its rectangle of y with a halo once, computes the subgradient on it
// (and on the one row and column the trial terms reach into), and evaluates
// the trial points from shared memory.  HBM / L2 see one read and one write of
// x per phase.  The CTAs of a right-hand side meet only in the sums that the
// decisions need, and every CTA takes the same decisions from the same FP64
// sums.  Two forms:
//  * GRID false: one thread-block cluster per right-hand side; the CTA sums
//    travel to every CTA's shared memory before one cluster barrier;
//  * GRID true: the whole GPU (a cooperative launch) for one right-hand side
//    after the other; the CTA sums go through L2 and one counter.
// The phase is bound by the latency of its two reductions and of the loads, so
// what was taken out is serial work: all loads of a thread in flight together,
// warps reduce in parallel, one barrier a reduction, no second copy of the
// image in L2.  Measured (GB300, isotropic TV, one step): cluster form, 64x64
// 22.4 -> 9.5 us, 128x128 22.6 -> 10.0 us; whole GPU, 512x512 25.1 -> 15.6 us,
// 1024x1024 45.9 -> 24.0 us; 16 images of 256x512 77.7 -> 61.6 us (before: image
// bands read element by element through the neighbours' shared memory, sums
// by one thread per CTA, and in the whole-GPU form y and g re-read from L2
// with a barrier of 5 us around a last CTA's reduction).
constexpr int kFirstTrials = 1;   // trial points of a step's first pass (the first usually passes)
constexpr int kMaxCluster = 16;

__device__ __forceinline__ FF ff_warp(FF a) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        a = ff_add(a, FF{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)});
    return a;
}

// q / d for q d < 2^32 and d >= 2, m = ceil(2^32 / d).
__device__ __forceinline__ int div_by(int q, unsigned m) { return (int)__umulhi((unsigned)q, m); }

template <bool GRID, int NT>
struct PhaseSums {
    FF* sw;                      // NT / 32 x kWideTrials warp sums
    FF* peer;                    // cluster: 2 x kMaxCluster x kWideTrials CTA sums, written by every CTA
    double* part;                // grid: 2 x tiles x kWideTrials CTA sums
    unsigned long long* bar;     // grid: arrivals; [1] their count when the launch began
    unsigned long long target;   // grid, thread 0: arrivals at the next barrier's end
    int* err;
    long long limit;
    int* flag;                   // shared
    int rank, tiles, par;

    // Every CTA's writes before are visible to every CTA after; false on
    // timeout (whole CTA alike).
    __device__ bool barrier() {
        if constexpr (!GRID) {
            if (tiles > 1) cg::this_cluster().sync();
            else __syncthreads();
            return true;
        } else {
            __syncthreads();
            if (threadIdx.x == 0) {
                int ok = 1;
                target += (unsigned long long)tiles;
                // release: the CTA's writes ordered before by the barrier above
                asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(bar), "l"(1ULL) : "memory");
                const long long t0 = clock64();
                for (int k = 0;; ++k) {
                    unsigned long long v;
                    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(bar) : "memory");
                    if (v >= target) break;
                    if (clock64() - t0 > limit || ((k & 63) == 63 && *(volatile int*)err)) {
                        atomicExch(err, 2);
                        ok = 0;
                        break;
                    }
                }
                *flag = ok;
            }
            __syncthreads();
            return *flag != 0;
        }
    }

    // Sums of NV values over every thread of the right-hand side's CTAs, in a
    // fixed order: float-float over lanes, then warps, FP64 over the CTAs.
    // Warp k's `out` is the sum of value k.
    template <int NV>
    __device__ bool sum(FF (&v)[NV], double& out) {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        constexpr int NW = NT / 32;
        static_assert(NV <= NW && NV <= kWideTrials && NW <= 32, "one warp a value, one lane a warp sum");
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            v[k] = ff_warp(v[k]);
            if (lane == 0) sw[warp * kWideTrials + k] = v[k];
        }
        __syncthreads();
        FF s{0.f, 0.f};
        if (warp < NV) {
            if (lane < NW) s = sw[lane * kWideTrials + warp];
            s = ff_warp(s);
        }
        if (!GRID && tiles == 1) {
            out = (double)s.hi + (double)s.lo;
            return true;
        }
        if (warp < NV) {
            if constexpr (GRID) {
                if (lane == 0)
                    __stcg(part + ((size_t)par * tiles + rank) * kWideTrials + warp, (double)s.hi + (double)s.lo);
            } else if (lane < tiles) {
                FF* dst = cg::this_cluster().map_shared_rank(peer, lane);
                dst[(par * kMaxCluster + rank) * kWideTrials + warp] = s;
            }
        }
        const bool ok = barrier();
        if (ok && warp < NV) {
            double t = 0.0;
            if constexpr (GRID) {
                // five loads in flight: one round trip for up to 160 CTAs
                for (int c = lane; c < tiles; c += 160) {
                    double p[5];
#pragma unroll
                    for (int u = 0; u < 5; ++u)
                        p[u] = c + 32 * u < tiles
                                   ? __ldcg(part + ((size_t)par * tiles + c + 32 * u) * kWideTrials + warp)
                                   : 0.0;
                    t += ((p[0] + p[1]) + (p[2] + p[3])) + p[4];
                }
                out = warp_sum(t);
            } else {
                if (lane < tiles) {
                    const FF p = peer[(par * kMaxCluster + lane) * kWideTrials + warp];
                    t = (double)p.hi + (double)p.lo;
                }
                for (int o = tiles >> 1; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                out = t;   // tiles is a power of two
            }
        }
        // the next sum uses the other buffer; this one is written again only
        // after the barrier of that sum, which every CTA reaches after reading
        par ^= 1;
        return ok;
    }
};

// KIND 0 isotropic TV, 1 anisotropic TV, 2 element-wise objectives.
template <int KIND, bool GRID, int NT>
__global__ void __launch_bounds__(NT) k_phase(const PerturbArgs a) {
    extern __shared__ float smem[];
    __shared__ FF sw[(NT / 32) * kWideTrials];
    __shared__ FF peer[GRID ? 1 : 2 * kMaxCluster * kWideTrials];
    __shared__ double gy_s[2];              // ||g||^2, f(y)
    __shared__ float pow_s[kWideTrials];    // gamma alpha^(l + j)
    __shared__ int pass_s[kWideTrials];     // trial j passed
    __shared__ StepDecision dec;
    __shared__ int flag;
    // the row pass after it starts to stream its strips as SMs come free
    grid_trigger();
    const int tiles = a.TR * a.TC;
    const int tile = GRID ? (int)blockIdx.x : (int)(blockIdx.x % tiles);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n = a.n, B = a.B, obj = a.obj;
    const int H = KIND == 2 ? 1 : a.H, W = KIND == 2 ? n : a.W;
    // the first xh rows (xw columns) of rectangles are one pixel larger
    const int ti = (int)((unsigned)tile / (unsigned)a.TC), tj = tile - ti * a.TC;
    int h = a.th + (ti < a.xh ? 1 : 0), w = a.tw + (tj < a.xw ? 1 : 0);
    const int r0 = ti * a.th + min(ti, a.xh), c0 = tj * a.tw + min(tj, a.xw);
    if (!CHECKED(h <= a.tmh && w <= a.tmw && r0 + h <= H && c0 + w <= W && (long long)H * W == n &&
                     (!a.pA || (KIND != 2 && W <= a.pWp)),
                 401, tile))
        h = w = 0;
    const int own = h * w;
    const bool lin = KIND == 2 && obj == SUPPY_OBJ_LINEAR;
    // y with a halo of one pixel up / left and two down / right (the
    // subgradient is needed one pixel down / right of the rectangle)
    const int P = KIND == 2 ? w : w + 3, PG = KIND == 2 ? w : w + 1;
    float* ys = smem;
    float* gs = smem + (KIND == 2 ? a.tmw : (a.tmh + 3) * (a.tmw + 3));
    const int ylen = KIND == 2 ? own : (h + 3) * P, glen = KIND == 2 ? own : (h + 1) * PG;
    const unsigned mP = tj < a.xw ? a.mP1 : a.mP0, mG = tj < a.xw ? a.mG1 : a.mG0;
    PhaseSums<GRID, NT> sums{sw, peer, a.part, reinterpret_cast<unsigned long long*>(a.ticket), 0ULL, a.err,
                             a.wait_cycles, &flag, tile, tiles, 0};
    if (GRID && tid == 0) sums.target = __ldcg(sums.bar + 1);
    for (int b = GRID ? 0 : (int)(blockIdx.x / tiles); b < (GRID ? B : (int)(blockIdx.x / tiles) + 1); ++b) {
        RhsState& st = a.st[b];
        // the state as the phase finds it: its end is written while slower CTAs
        // may still decide
        const int stopped = st.stopped;
        const PhaseStart ps = phase_start(a, b);
        const bool has_ref = st.has_ref != 0;
        const double st_ref = st.f_ref;
        float* X = a.x + b;
        // pixel of element q of the y tile, or -1 outside the image
        auto pixel = [&](int q) {
            if constexpr (KIND == 2) return c0 + q;
            const int qi = div_by(q, mP), i = r0 - 1 + qi, j = c0 - 1 + (q - qi * P);
            return (i >= 0 && i < H && j >= 0 && j < W) ? i * W + j : -1;
        };
        auto load = [&](bool halo_only) {
            for (int q0 = tid; q0 < ylen; q0 += 4 * NT) {
                float v[4];
                bool in[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int q = q0 + u * NT;
                    int p = q < ylen ? pixel(q) : -1;
                    if (halo_only && p >= 0) {
                        const int qi = div_by(q, mP), i = qi - 1, j = q - qi * P - 1;
                        if (i >= 0 && i < h && j >= 0 && j < w) p = -1;
                    }
                    in[u] = p >= 0;
                    v[u] = in[u] ? __ldcg(X + (size_t)p * B) : 0.f;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (in[u]) ys[q0 + u * NT] = v[u];
            }
        };
        // a CTA's shared memory may be written by its peers once it runs
        if (!GRID && tiles > 1) cg::this_cluster().barrier_arrive();
        load(false);
        if (!GRID && tiles > 1) cg::this_cluster().barrier_wait();
        if (stopped) continue;   // uniform over the right-hand side's CTAs
        if (lin)
            for (int q = tid; q < own; q += NT) gs[q] = a.c32[c0 + q];
        long long ell = ps.ell;
        if (tid < kWideTrials) pow_s[tid] = trial_scale(a.gamma, a.log2_alpha, ell + tid, 1.f);
        int accepted = 0, trials = 0;
        double f_start = 0.0;   // thread 0
        bool copied = false;
        __syncthreads();
        for (int s = 0; s < a.n_red; ++s) {
            // subgradient, ||g||^2 and f(y)
            KSum kg, kf;
            double fl = 0.0;
            for (int q = tid; q < glen; q += NT) {
                float g = 0.f, term = 0.f;
                if constexpr (KIND == 2) {
                    const float y = ys[q];
                    if (lin) {
                        g = gs[q];
                        fl += a.c64[c0 + q] * (double)y;
                    } else {
                        term = norm_term(obj, y);
                        g = norm_grad(obj, y);
                        gs[q] = g;
                    }
                    kf.add(term);
                    kg.add(g * g);
                } else {
                    const int qi = div_by(q, mG), qj = q - qi * PG, i = r0 + qi, j = c0 + qj;
                    if (i >= H || j >= W) continue;
                    const float* yp = ys + (qi + 1) * P + qj + 1;
                    const float y0 = yp[0];
                    const bool up = i > 0, left = j > 0, down = i < H - 1, right = j < W - 1;
                    if constexpr (KIND == 0) {
                        if (down && right) {
                            const float dx = yp[P] - y0, dy = yp[1] - y0, e = sq2(dx, dy);
                            term = sqrtf(e);
                            if (e > 0.f) g -= (dx + dy) * rsqrtf(e);
                        }
                        if (up && right) {
                            const float ym = yp[-P], dx = y0 - ym, dy = yp[1 - P] - ym, e = sq2(dx, dy);
                            if (e > 0.f) g += dx * rsqrtf(e);
                        }
                        if (left && down) {
                            const float yl = yp[-1], dx = yp[P - 1] - yl, dy = y0 - yl, e = sq2(dx, dy);
                            if (e > 0.f) g += dy * rsqrtf(e);
                        }
                    } else {
                        if (down) {
                            const float d = yp[P] - y0;
                            term += fabsf(d);
                            g -= sgnf(d);
                        }
                        if (up) g += sgnf(y0 - yp[-P]);
                        if (right) {
                            const float d = yp[1] - y0;
                            term += fabsf(d);
                            g -= sgnf(d);
                        }
                        if (left) g += sgnf(y0 - yp[-1]);
                    }
                    gs[q] = g;
                    if (qi < h && qj < w) {
                        kf.add(term);
                        kg.add(g * g);
                    }
                }
            }
            FF v2[2] = {ff_of(kg), lin ? ff_of(fl) : ff_of(kf)};
            double out = 0.0;
            if (!sums.sum(v2, out)) return;
            if (warp < 2 && lane == 0) gy_s[warp] = out;
            __syncthreads();
            const double fy = gy_s[1];
            if (tid == 0) {
                if (s == 0) f_start = fy;
                dec = step_decision(a, has_ref, st_ref, gy_s[0], fy, f_start);
            }
            __syncthreads();
            if (!dec.go) break;
            const float inv_gnorm = dec.inv_gnorm, asc = dec.asc;
            const int jmax = a.adaptive ? 1 : a.max_trials;
            bool ok = false;
            // f at N consecutive trial points; the first that passes, or -1,
            // or -2 when a wait gave up
            auto try_points = [&](auto NC, int cnt, const float* sj) -> int {
                constexpr int N = decltype(NC)::value;
                KSum kz[N];
                double fz[N];
#pragma unroll
                for (int k = 0; k < N; ++k) fz[k] = 0.0;
                // the same pixels in the same order as f(y): where a step leaves
                // y as it is, f(z) is f(y) to the last bit
                for (int q = tid; q < glen; q += NT) {
                    if constexpr (KIND == 2) {
                        const float y0 = ys[q], g0 = gs[q];
                        const double c = lin ? a.c64[c0 + q] : 0.0;
#pragma unroll
                        for (int k = 0; k < N; ++k) {
                            const float z = trial(y0, g0, sj[k]);
                            if (lin) fz[k] += c * (double)z;
                            else kz[k].add(norm_term(obj, z));
                        }
                    } else {
                        const int qi = div_by(q, mG), qj = q - qi * PG, i = r0 + qi, j = c0 + qj;
                        if (qi >= h || qj >= w) continue;
                        const float* yp = ys + (qi + 1) * P + qj + 1;
                        const float* gp = gs + q;
                        TvNbr t;
                        t.down = i < H - 1;
                        t.right = j < W - 1;
                        t.y0 = yp[0];
                        t.g0 = gp[0];
                        t.yd = yp[P];
                        t.gd = gp[PG];
                        t.yr = yp[1];
                        t.gr = gp[1];
#pragma unroll
                        for (int k = 0; k < N; ++k) kz[k].add(tv_trial_term(obj, t, sj[k]));
                    }
                }
                FF v[N];
#pragma unroll
                for (int k = 0; k < N; ++k) v[k] = lin ? ff_of(fz[k]) : ff_of(kz[k]);
                double o = 0.0;
                if (!sums.sum(v, o)) return -2;
                if (warp < N && lane == 0) pass_s[warp] = o <= fy;
                __syncthreads();
                int hit = -1;
#pragma unroll
                for (int k = N - 1; k >= 0; --k)
                    if (k < cnt && pass_s[k]) hit = k;
                return hit;
            };
            for (int jt = 0; jt < jmax && !ok;) {
                const int cnt = min(jt == 0 ? kFirstTrials : kWideTrials, jmax - jt);
                float sj[kWideTrials];
#pragma unroll
                for (int k = 0; k < kWideTrials; ++k) sj[k] = a.adaptive ? asc : pow_s[k] * inv_gnorm;
                const int hit = jt == 0 ? try_points(std::integral_constant<int, kFirstTrials>{}, cnt, sj)
                                        : try_points(std::integral_constant<int, kWideTrials>{}, cnt, sj);
                if (hit == -2) return;
                const int used = hit >= 0 ? hit + 1 : cnt;
                if (!a.adaptive) {
                    ell += used;
                    // every thread has its step sizes in registers (the sums'
                    // barriers lie between)
                    if (tid < kWideTrials && (hit < 0 || s + 1 < a.n_red)) pow_s[tid] = trial_scale(a.gamma, a.log2_alpha, ell + tid, 1.f);
                }
                trials += used;
                jt += used;
                if (hit >= 0) {
                    float sc = sj[0];
#pragma unroll
                    for (int k = 1; k < kWideTrials; ++k) sc = k == hit ? sj[k] : sc;
                    for (int q = tid; q < glen; q += NT) {
                        const int qi = KIND == 2 ? 0 : div_by(q, mG), qj = KIND == 2 ? q : q - qi * PG;
                        if (qi >= h || qj >= w) continue;
                        const int e = KIND == 2 ? q : (qi + 1) * P + qj + 1;
                        const float z = trial(ys[e], gs[q], sc);
                        ys[e] = z;
                        const int i = r0 + qi, j = c0 + qj;
                        X[(size_t)(i * W + j) * B] = z;
                        if (GRID && KIND != 2 && a.pA) {
                            a.pA[patch_pos(i, j, a.pWp, false)] = z;
                            a.pB[patch_pos(i, j, a.pWp, true)] = z;
                        }
                    }
                    copied = true;
                    accepted += 1;
                    ok = true;
                }
                __syncthreads();   // pow_s, pass_s
            }
            if (!ok) break;
            if (s + 1 < a.n_red && tiles > 1 && KIND != 2) {
                // the next step reads the neighbours' new y around the rectangle
                if (!sums.barrier()) return;
                load(true);
                __syncthreads();
            }
        }
        if (GRID && KIND != 2 && a.pA && !copied)
            // no step was taken: the patch copies of y as it stands
            for (int q = tid; q < glen; q += NT) {
                const int qi = div_by(q, mG), qj = q - qi * PG, i = r0 + qi, j = c0 + qj;
                if (qi >= h || qj >= w) continue;
                const float z = ys[(qi + 1) * P + qj + 1];
                a.pA[patch_pos(i, j, a.pWp, false)] = z;
                a.pB[patch_pos(i, j, a.pWp, true)] = z;
            }
        if (tile == 0 && tid == 0) phase_end(a, st, ps, ell, accepted, trials, f_start);
        if (GRID && b + 1 < B) __syncthreads();   // the tile is loaded anew
    }
    // the next launch counts on from here (this CTA has passed the last barrier)
    if (GRID && tile == 0 && tid == 0) __stcg(sums.bar + 1, sums.target);
}

// ------------------------------------------------ whole-GPU phase ----
// The perturbation phase of Algorithm 1 on the whole GPU, one right-hand side
// after the other, in a single cooperative launch (every CTA resident).  Each
// pass over the image -- the subgradient with ||g||^2 and f(y); f at up to
// kWideTrials consecutive trial points y - beta_j g/||g|| at once; the update
// y <- z_j -- takes a grid-stride share of the pixels per thread and ends in
// a grid barrier, inside which the last CTA to arrive sums the CTA partials
// in a fixed order; every CTA reads the same sums and takes the same
// decisions (the first j with f(z_j) <= f(y): exactly the trial the
// sequential loop accepts) without a further barrier.  y and g are read with plain coherent
// loads (other CTAs rewrite them between passes; the barrier's fences make
// those writes visible), never through the read-only path.  Element e of the
// n x B array is pixel e / B of right-hand side e % B.

// Last-CTA election: every CTA's partials are visible to the CTA that draws
// the last ticket; it resets the ticket for the next launch.
__device__ __forceinline__ bool last_cta(unsigned* ticket) {
    __shared__ bool is_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) is_last = (atomicAdd(ticket, 1u) == gridDim.x - 1);
    __syncthreads();
    if (is_last) __threadfence();
    return is_last;
}

// Fixed-order sum of part[c * stride + off] over the grid's CTAs by one warp.
__device__ __forceinline__ double warp_sum_parts(const double* part, int ncta, int stride,
                                                 int off) {
    const int lane = threadIdx.x & 31;
    double s = 0.0;
    for (int c = lane; c < ncta; c += 32) s += __ldcg(part + (size_t)c * stride + off);
    return warp_sum(s);
}

// Per-CTA sums of NV values per right-hand side, written as FP64 to
// part[(cta * B + b) * NV + v]: float-float sums over the lanes of each
// right-hand side, then over the warps in order.  sw holds 8 * NV * 32 values.
// Only the first nv values (uniform over the CTA) are reduced and written.
template <int NV, int NT = kWideThreads>
__device__ __forceinline__ void cta_partials(FF (&v)[NV], int B, FF* sw, double* part,
                                             int nv = NV) {
#pragma unroll
    for (int j = 0; j < NV; ++j)
        if (j < nv)
            for (int o = 16; o >= B && o > 0; o >>= 1) {
                const FF w{__shfl_xor_sync(0xffffffffu, v[j].hi, o),
                           __shfl_xor_sync(0xffffffffu, v[j].lo, o)};
                v[j] = ff_add(v[j], w);
            }
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane < B)
#pragma unroll
        for (int j = 0; j < NV; ++j)
            if (j < nv) sw[(wid * NV + j) * 32 + lane] = v[j];
    __syncthreads();
    for (int t = threadIdx.x; t < NV * B; t += NT) {
        const int b = t / NV, j = t - b * NV;
        if (j >= nv) continue;
        FF acc{0.f, 0.f};
        for (int w = 0; w < NT / 32; ++w) acc = ff_add(acc, sw[(w * NV + j) * 32 + b]);
        part[((size_t)blockIdx.x * B + b) * NV + j] = (double)acc.hi + (double)acc.lo;
    }
}

// The grid sums of the NV * B values, one warp per value, into res[b * NV + v]
// (shared memory).
template <int NV, int NT = kWideThreads>
__device__ __forceinline__ void grid_sums(const double* part, int B, double* res) {
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int t = wid; t < NV * B; t += NT / 32) {
        const double v = warp_sum_parts(part, gridDim.x, NV * B, t);
        if (lane == 0) res[t] = v;
    }
    __syncthreads();
}

// Grid barrier of a cooperative launch: bar[0] counts arrivals, bar[1] is the
// generation.  A CTA reads the generation before it arrives; the last to
// arrive first sums the NV CTA partials of the pass (one warp per value, a
// fixed order: the same FP64 sums whichever CTA arrives last) into gsum, then
// resets the count and advances the generation; the others wait, then read
// gsum into res (shared memory).  One CTA does the FP64 reduction: FP64 is
// scarce on GB300, and every CTA summing the partials itself took longer than
// the wait.  The wait is bounded: on timeout
// the CTA records error word 2 and every CTA leaves at its next barrier.  The
// budget is a launch argument (about two seconds of SM clock by default).
// The partials need no second buffer: they are read before the release, and
// written again only after it.
template <int NV>
__device__ __forceinline__ bool grid_barrier(unsigned* bar, int* err, const double* part,
                                             double* gsum, double* res, long long limit) {
    __shared__ int st_s;   // bit 0: ok, bit 1: this CTA arrived last
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile unsigned* gen = bar + 1;
        const unsigned g0 = *gen;
        __threadfence();
        int ok = 1, last = 0;
        if (atomicAdd(bar, 1u) == gridDim.x - 1) {
            last = 1;
            __threadfence();
        } else {
            const long long t0 = clock64();
            while (*gen == g0) {
                if (*(volatile int*)err || clock64() - t0 > limit) {
                    atomicExch(err, 2);
                    ok = 0;
                    break;
                }
                __nanosleep(32);
            }
            __threadfence();
        }
        st_s = ok | (last << 1);
    }
    __syncthreads();
    const int st = st_s;
    if (st & 2) {
        if constexpr (NV > 0) {
            grid_sums<NV, kPhaseThreads>(part, 1, res);
            if (threadIdx.x < NV) gsum[threadIdx.x] = res[threadIdx.x];
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            __threadfence();
            atomicExch(bar, 0u);
            __threadfence();
            atomicAdd(bar + 1, 1u);
        }
    } else {
        if constexpr (NV > 0)
            if (threadIdx.x < NV) res[threadIdx.x] = __ldcg(gsum + threadIdx.x);
    }
    __syncthreads();
    return (st & 1) && *(volatile int*)err == 0;
}

// Image of one right-hand side read with plain (coherent, L1-cached) loads:
// other CTAs rewrite it between passes, and the grid barrier's fences make
// their writes visible to these loads, which the read-only path (ld.global.nc)
// would not guarantee.
struct CohImage {
    const float* y;   // element 0 of the right-hand side
    int B, W;
    __device__ __forceinline__ float operator()(int i, int j) const {
        return y[((size_t)i * W + j) * B];
    }
};

__global__ void __launch_bounds__(kPhaseThreads, 1) k_wide_phase(const PerturbArgs a) {
    __shared__ FF sw[(kPhaseThreads / 32) * kWideTrials * 32];
    __shared__ double res[kWideTrials];
    __shared__ float sj_s[kWideTrials];
    __shared__ int dec_s[2];     // continue the step; the accepted trial (-1: none)
    __shared__ float dec_f[2];   // 1/||g||; the adaptive step
    const int B = a.B, n = a.n, H = a.H, W = a.W, obj = a.obj;
    const int tid = blockIdx.x * kPhaseThreads + threadIdx.x;
    const int stride = gridDim.x * kPhaseThreads;
    const bool lin = (obj == SUPPY_OBJ_LINEAR);
    const bool tv = !elementwise(obj);
    double* const part = a.part;
    double* const gsum = a.part + (size_t)gridDim.x * kWideTrials;
    for (int b = 0; b < B; ++b) {
        RhsState& st = a.st[b];
        if (st.stopped) continue;   // read by every CTA before the phase's first barrier
        const PhaseStart ps = phase_start(a, b);
        const bool has_ref = st.has_ref;
        const double st_ref = st.f_ref;
        long long ell = ps.ell;
        int accepted = 0, trials = 0;
        double f_start = 0.0;
        float* X = a.x + b;
        float* G = a.g + b;
        bool copied = false;   // the patch copies were written with the last update
        for (int s = 0; s < a.n_red; ++s) {
            // pass G: subgradient, ||g||^2 and f(y)
            KSum kg, kf;
            double fl = 0.0;
            StrideWalk px(tid, stride, tv ? W : 1);
            for (int p = tid; p < n; p += stride, px.next()) {
                float gp;
                if (lin) {
                    gp = a.c32[p];
                    fl += a.c64[p] * (double)X[(size_t)p * B];
                } else if (!tv) {
                    const float y0 = X[(size_t)p * B];
                    kf.add(norm_term(obj, y0));
                    gp = norm_grad(obj, y0);
                } else {
                    const CohImage yi{X, B, W};
                    kf.add(tv_term(obj, px.i, px.j, H, W, yi));
                    gp = tv_subgrad(obj, px.i, px.j, H, W, yi);
                }
                G[(size_t)p * B] = gp;
                kg.add(gp * gp);
            }
            {
                FF v[2] = {ff_of(kg), lin ? ff_of(fl) : ff_of(kf)};
                cta_partials<2, kPhaseThreads>(v, 1, sw, part);
            }
            if (!grid_barrier<2>(a.ticket, a.err, part, gsum, res, a.wait_cycles)) return;
            // the step's scalar decisions by one thread (FP64 is scarce on
            // GB300: not by every thread of the grid), shared through smem
            const double fy = res[1];
            if (threadIdx.x == 0) {
                const double gg = res[0];
                if (s == 0) f_start = fy;
                int go = gg != 0.0;
                float inv_gnorm = 0.f, asc = 0.f;
                if (go) {
                    inv_gnorm = 1.0f / sqrtf((float)gg);
                    if (a.adaptive) {
                        const double f_ref =
                            a.adaptive == 2 ? a.f_ref : (has_ref ? fmin(st_ref, f_start) : f_start);
                        if (!(fy > f_ref)) go = 0;
                        else asc = adaptive_scale(fy, f_ref, gg);
                    }
                }
                dec_s[0] = go;
                dec_f[0] = inv_gnorm;
                dec_f[1] = asc;
            }
            __syncthreads();
            if (!dec_s[0]) break;
            const float inv_gnorm = dec_f[0], asc = dec_f[1];
            const int jmax = a.adaptive ? 1 : a.max_trials;
            bool ok = false;
            for (int jt = 0; jt < jmax && !ok;) {
                // the first pass of a step tries kFirstTrials points (usually
                // the first is accepted once the exponent has settled), later
                // passes kWideTrials; the accepted trial is the same either way
                const int cnt = min(jt == 0 ? kFirstTrials : kWideTrials, jmax - jt);
                // the trial step sizes, one thread each
                if (threadIdx.x < kWideTrials)
                    sj_s[threadIdx.x] = a.adaptive
                                            ? asc
                                            : trial_scale(a.gamma, a.log2_alpha, ell + threadIdx.x,
                                                          inv_gnorm);
                __syncthreads();
                float sj[kWideTrials];
#pragma unroll
                for (int q = 0; q < kWideTrials; ++q) sj[q] = sj_s[q];
                // pass T: f at the cnt trial points (the slots past cnt are not read)
                KSum kz[kWideTrials];
                double fz[kWideTrials];
#pragma unroll
                for (int q = 0; q < kWideTrials; ++q) fz[q] = 0.0;
                StrideWalk px(tid, stride, tv ? W : 1);
                for (int p = tid; p < n; p += stride, px.next()) {
                    if (lin) {
                        const float y0 = X[(size_t)p * B], g0 = G[(size_t)p * B];
                        const double c = a.c64[p];
#pragma unroll
                        for (int q = 0; q < kWideTrials; ++q)
                            if (q < cnt) fz[q] += c * (double)trial(y0, g0, sj[q]);
                    } else if (!tv) {
                        const float y0 = X[(size_t)p * B], g0 = G[(size_t)p * B];
#pragma unroll
                        for (int q = 0; q < kWideTrials; ++q)
                            if (q < cnt) kz[q].add(norm_term(obj, trial(y0, g0, sj[q])));
                    } else {
                        const TvNbr t = tv_nbr(px.i, px.j, H, W, X, G, B);
#pragma unroll
                        for (int q = 0; q < kWideTrials; ++q)
                            if (q < cnt) kz[q].add(tv_trial_term(obj, t, sj[q]));
                    }
                }
                {
                    FF v[kWideTrials];
#pragma unroll
                    for (int q = 0; q < kWideTrials; ++q) v[q] = lin ? ff_of(fz[q]) : ff_of(kz[q]);
                    cta_partials<kWideTrials, kPhaseThreads>(v, 1, sw, part, cnt);
                }
                if (!grid_barrier<kWideTrials>(a.ticket, a.err, part, gsum, res, a.wait_cycles)) return;
                if (threadIdx.x == 0) {
                    int h = -1;
                    for (int q = 0; q < cnt; ++q)
                        if (res[q] <= fy) {
                            h = q;
                            break;
                        }
                    dec_s[1] = h;
                }
                __syncthreads();
                const int hit = dec_s[1];
                const int used = hit >= 0 ? hit + 1 : cnt;
                if (!a.adaptive) ell += used;
                trials += used;
                jt += used;
                if (hit >= 0) {
                    // pass U: y <- z_hit (and its patch copies, pixel by pixel)
                    const float sc = sj_s[hit];
                    if (a.pA) {
                        StrideWalk pw(tid, stride, W);
                        for (int p = tid; p < n; p += stride, pw.next()) {
                            const float v = trial(X[p], G[p], sc);
                            X[p] = v;
                            a.pA[patch_pos(pw.i, pw.j, a.pWp, false)] = v;
                            a.pB[patch_pos(pw.i, pw.j, a.pWp, true)] = v;
                        }
                        copied = true;
                    } else {
                        for (int p = tid; p < n; p += stride) {
                            const size_t o = (size_t)p * B;
                            X[o] = trial(X[o], G[o], sc);
                        }
                    }
                    accepted += 1;
                    ok = true;
                }
            }
            if (!ok) break;
            // the next reduction step reads the neighbours' new y
            if (s + 1 < a.n_red && !grid_barrier<0>(a.ticket, a.err, part, gsum, res, a.wait_cycles)) return;
        }
        if (a.pA && !copied) {
            // no step was taken: the copies of y as it stands (each thread its
            // own pixels, which no other thread writes in this launch)
            StrideWalk pw(tid, stride, W);
            for (int p = tid; p < n; p += stride, pw.next()) {
                const float v = X[p];
                a.pA[patch_pos(pw.i, pw.j, a.pWp, false)] = v;
                a.pB[patch_pos(pw.i, pw.j, a.pWp, true)] = v;
            }
        }
        if (blockIdx.x == 0 && threadIdx.x == 0) phase_end(a, st, ps, ell, accepted, trials, f_start);
    }
}

// ------------------------------------------------ variance stopping rule ----
// After an iteration: ||x - xprev||^2 and ||x||^2 per right-hand side
// (compensated FP32 per thread, float-float per CTA, FP64 over the grid),
// xprev <- x; the last CTA adds omega = ||x - xprev|| / ||x|| to the running
// sums of the state and stops a right-hand side once the sample variance of
// its omegas (k >= 2 of them) is below tol.
__global__ void __launch_bounds__(kWideThreads) k_variance(float* x, float* xprev, long long n,
                                                           int B, RhsState* st, double* part,
                                                           unsigned* ticket, double tol) {
    __shared__ FF sw[(kWideThreads / 32) * 2 * 32];
    __shared__ double res[2 * kMaxRhs];
    const long long nB = n * B;
    const long long tid = (long long)blockIdx.x * kWideThreads + threadIdx.x;
    const long long stride = (long long)gridDim.x * kWideThreads;
    const int b = (int)(tid & (B - 1));
    KSum kd, kx;
    if (!st[b].stopped)
        for (long long e = tid; e < nB; e += stride) {
            const float v = x[e], d = v - xprev[e];
            kd.add(d * d);
            kx.add(v * v);
            xprev[e] = v;
        }
    FF v[2] = {ff_of(kd), ff_of(kx)};
    cta_partials<2>(v, B, sw, part);
    if (!last_cta(ticket)) return;
    grid_sums<2>(part, B, res);
    if (threadIdx.x < B) {
        RhsState& s = st[threadIdx.x];
        if (!s.stopped) {
            const double D = res[2 * threadIdx.x], X = res[2 * threadIdx.x + 1];
            const double w = X > 0.0 ? sqrt(D / X) : 0.0;
            s.w_n += 1;
            s.w_s1 += w;
            s.w_s2 += w * w;
            if (s.w_n >= 2) {
                const double nn = (double)s.w_n;
                const double var = (s.w_s2 - s.w_s1 * s.w_s1 / nn) / (nn - 1.0);
                if (var < tol) s.stopped = 1;
            }
        }
    }
    if (threadIdx.x == 0) *ticket = 0u;
}

// Objective partials: CTA c writes f-partials of every right-hand side.
__global__ void __launch_bounds__(256) k_objective(const ObjArgs a) {
    __shared__ double sw[8];
    for (int b = 0; b < a.B; ++b) {
        Vec y{const_cast<float*>(a.x) + b, a.B};
        double f = 0.0;
        for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < a.n; p += gridDim.x * blockDim.x)
            f += obj_term(a.obj, p, a.H, a.W, a.c64, y);
        f = warp_sum(f);
        if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = f;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int w = 0; w < 8; ++w) s += sw[w];
            a.partial[(size_t)blockIdx.x * a.B + b] = s;
        }
        __syncthreads();
    }
}

}  // namespace

namespace {

// Shared memory of the tile-resident phase for rectangles of th x tw pixels.
size_t phase_smem(bool elem, int th, int tw) {
    if (elem) return sizeof(float) * 2 * (size_t)tw;
    return sizeof(float) * ((size_t)(th + 3) * (tw + 3) + (size_t)(th + 1) * (tw + 1));
}

constexpr size_t kPhaseSmem = 200 * 1024;

bool elem_obj(int obj) {
    return obj == SUPPY_OBJ_LINEAR || obj == SUPPY_OBJ_L1 || obj == SUPPY_OBJ_L2;
}

// The grid of at most `tiles` rectangles whose largest one, halo included, is
// smallest; false when it does not fit shared memory.
bool phase_tiles(int obj, int n, int H, int W, int tiles, bool exact, PhaseTiles* out) {
    PhaseTiles best;
    if (elem_obj(obj)) {
        if (tiles > n && exact) return false;
        best.TR = 1;
        best.TC = std::min(tiles, n);
        best.h = 1;
        best.w = (n + best.TC - 1) / best.TC;
        H = 1;
        W = n;
    } else {
        long long cost = -1;
        for (int r = 1; r <= std::min(tiles, H); ++r) {
            const int c = std::min(tiles / r, W);
            if (c < 1 || (exact && r * c != tiles)) continue;
            const int h = (H + r - 1) / r, w = (W + c - 1) / c;
            const long long k = (long long)(h + 3) * (w + 3);
            if (cost < 0 || k < cost) {
                cost = k;
                best = PhaseTiles{r, c, h, w};
            }
        }
        if (cost < 0) return false;
    }
    if (phase_smem(elem_obj(obj), best.h, best.w) > kPhaseSmem) return false;
    *out = best;
    return true;
}

// The rectangles as the kernel takes them: the size of the smaller ones, how
// many rows and columns of them are one pixel larger, and the factors that
// divide by the widths of their y (w + 3) and subgradient (w + 1) tiles.
void set_phase_tiles(PerturbArgs& a, const PhaseTiles& t) {
    const int H = elem_obj(a.obj) ? 1 : a.H, W = elem_obj(a.obj) ? a.n : a.W;
    a.TR = t.TR;
    a.TC = t.TC;
    a.tmh = t.h;
    a.tmw = t.w;
    a.th = H / t.TR;
    a.xh = H % t.TR;
    a.tw = W / t.TC;
    a.xw = W % t.TC;
    auto magic = [](int d) { return (unsigned)(((1ULL << 32) + d - 1) / d); };
    a.mP0 = magic(a.tw + 3);
    a.mP1 = magic(a.tw + 4);
    a.mG0 = magic(a.tw + 1);
    a.mG1 = magic(a.tw + 2);
}

using PhaseFn = void (*)(PerturbArgs);

PhaseFn phase_fn(int obj, bool grid, int threads) {
    const int kind = obj == SUPPY_OBJ_TV_ISO ? 0 : (obj == SUPPY_OBJ_TV_ANISO ? 1 : 2);
    if (!grid) return kind == 0 ? k_phase<0, false, 512> : (kind == 1 ? k_phase<1, false, 512> : k_phase<2, false, 512>);
    if (threads == 512)
        return kind == 0 ? k_phase<0, true, 512> : (kind == 1 ? k_phase<1, true, 512> : k_phase<2, true, 512>);
    return kind == 0 ? k_phase<0, true, 1024> : (kind == 1 ? k_phase<1, true, 1024> : k_phase<2, true, 1024>);
}

// Threads per CTA of the whole-GPU form: 1024 where 512 would take more than
// two pixels each.
int phase_threads(const PhaseTiles& t) { return (long long)t.h * t.w > 1024 ? 1024 : 512; }

}  // namespace

// CTAs per right-hand side of the cluster form: two pixels a thread for one
// right-hand side (64x64 and 128x128 images: 9.5-10 us, where one thread took
// eight pixels 22 us), eight for several, whose clusters share the GPU (16
// images of 256x512: 61.6 us in clusters of 16, 67.0 us in clusters of 8 with
// 1024 threads); at most 16 (one GPC).
int choose_perturb_cluster(int n, int B) {
    const long long per_cta = kPerturbThreads * (B == 1 ? 2 : 8);
    int cs = 1;
    while (cs < 16 && cs * per_cta < n) cs <<= 1;
    return cs;
}

int fit_perturb_cluster(int want, int obj, int n, int H, int W) {
    // more CTAs where their rectangles would not fit shared memory, then the
    // largest power of two for which a cluster can be resident
    PhaseTiles t;
    int most = want;
    while (most < 16 && !phase_tiles(obj, n, H, W, most, true, &t)) most <<= 1;
    for (int cs = most; cs >= 1; cs >>= 1) {
        const bool tiled = phase_tiles(obj, n, H, W, cs, true, &t);
        const size_t smem = tiled ? phase_smem(elem_obj(obj), t.h, t.w) : 0;
        auto kern = tiled ? phase_fn(obj, false, kPerturbThreads) : k_perturb;
        cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (smem) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(cs, 1, 1);
        cfg.blockDim = dim3(kPerturbThreads, 1, 1);
        cfg.dynamicSmemBytes = smem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = cs;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int nc = 0;
        if (cudaOccupancyMaxActiveClusters(&nc, kern, &cfg) == cudaSuccess && nc > 0) return cs;
        cudaGetLastError();
    }
    return 1;
}

cudaError_t launch_perturb(const PerturbArgs& args, int cluster, cudaStream_t s) {
    PerturbArgs a = args;
    PhaseTiles t;
    const bool tiled = !a.record_only && phase_tiles(a.obj, a.n, a.H, a.W, cluster, true, &t);
    size_t smem = 0;
    auto kern = k_perturb;
    if (tiled) {
        set_phase_tiles(a, t);
        smem = phase_smem(elem_obj(a.obj), t.h, t.w);
        kern = phase_fn(a.obj, false, kPerturbThreads);
    }
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    if (smem) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.B * cluster, 1, 1);
    cfg.blockDim = dim3(kPerturbThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

bool wide_phase_tiles(int obj, int n, int H, int W, int sms, PhaseTiles* out) {
    // a few hundred pixels a CTA at least: fewer CTAs meet sooner
    const int tiles = (int)std::max<long long>(1, std::min<long long>(sms, ((long long)n + 255) / 256));
    if (!phase_tiles(obj, n, H, W, tiles, false, out)) return false;
    const size_t smem = phase_smem(elem_obj(obj), out->h, out->w);
    auto kern = phase_fn(obj, true, phase_threads(*out));
    int nb = 0;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, phase_threads(*out), smem) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return nb >= 1;
}

cudaError_t launch_phase_tiles(const PerturbArgs& args, const PhaseTiles& t, cudaStream_t s) {
    PerturbArgs a = args;
    if (!a.ticket || !a.err || !a.part || (a.pA && elem_obj(a.obj))) return cudaErrorInvalidValue;
    set_phase_tiles(a, t);
    const size_t smem = phase_smem(elem_obj(a.obj), t.h, t.w);
    auto kern = phase_fn(a.obj, true, phase_threads(t));
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(t.TR * t.TC, 1, 1);
    cfg.blockDim = dim3(phase_threads(t), 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

// kWideTrials partials per CTA, two buffers (the tile-resident phase) or one
// and the grid sums
size_t wide_part_doubles(int grid) { return 2 * ((size_t)grid + 1) * kWideTrials; }

int wide_phase_blocks_per_sm() {
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_wide_phase, kPhaseThreads, 0) !=
        cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return nb;
}

cudaError_t launch_variance(float* x, float* xprev, long long n, int B, RhsState* st,
                            double* part, unsigned* ticket, double tol, int grid, cudaStream_t s) {
    k_variance<<<grid, kWideThreads, 0, s>>>(x, xprev, n, B, st, part, ticket, tol);
    return cudaGetLastError();
}

cudaError_t launch_perturb_wide(const PerturbArgs& a, int grid, cudaStream_t s) {
    if (!a.ticket || !a.err || !a.part || grid < 1 || (a.pA && elem_obj(a.obj))) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(kPhaseThreads, 1, 1);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_wide_phase, a);
}

cudaError_t launch_objective(const ObjArgs& a, int grid, double* out, cudaStream_t s) {
    k_objective<<<grid, 256, 0, s>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_reduce_pp(a.partial, grid, a.B, 1.0, 0, out, s);
}

}  // namespace suppy
