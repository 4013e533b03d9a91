// Split feasibility with dose-volume constraints: the CQ step of Sec. 2.1.1
// (the iteration printed after Eq. (Split)) over the dose-volume sets of
// Sec. 2.3.3,
//
//     x <- x + gamma sum_j w_j A_j^T (P_Qj(A_j x) - A_j x),
//
// in three launches: the doses d = A_q x (warp per row), the projections onto
// the DVC sets (one CTA per structure: radix selection of the K-th highest
// dose, equal doses ranked by row), and the correction gathered per column
// through the CSC copy of A_q (warps per column, deterministic) beside the
// fixed-order sum of the target-space proximity.
//
// Sets (reading of the paper's wording): an upper DVC (D_V <= d_ref) lets at
// most K = floor(V N) of the structure's N voxels exceed d_ref, a lower DVC
// (D_V >= d_ref) demands at least K = ceil(V N) voxels at or above d_ref.  The
// Euclidean projection keeps (upper) or raises to d_ref (lower) the K highest
// doses and lowers (upper) every other dose above d_ref to d_ref.
#include <cooperative_groups.h>

#include <algorithm>

#include "common.cuh"

namespace suppy {

namespace cg = cooperative_groups;

namespace {

constexpr int kDoseThreads = 256;
constexpr int kProjectThreads = 1024;
constexpr int kApplyThreads = 256;

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Order-preserving key of a float dose: larger dose, larger key; -0 and +0
// map to the same key (they are equal doses).
__device__ __forceinline__ uint32_t dose_key(float f) {
    if (f == 0.0f) f = 0.0f;
    const uint32_t b = __float_as_uint(f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// Entries e, e + step, ... of a lane, kBatch at once, and their sum with the
// gathered y: the loads of one batch run beside the gathers of another.
constexpr int kBatch = 6;
struct Batch {
    int c[kBatch];
    float v[kBatch];
    __device__ __forceinline__ void load(const int* __restrict__ idx, const float* __restrict__ val, int e,
                                         int step, int e1) {
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const bool ok = e + u * step < e1;
            c[u] = ok ? __ldg(idx + e + u * step) : -1;
            v[u] = ok ? __ldg(val + e + u * step) : 0.f;
        }
    }
    __device__ __forceinline__ float add(float s, const float* y, int stride) const {
        float g[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) g[u] = c[u] >= 0 ? y[(size_t)c[u] * stride] : 0.f;
#pragma unroll
        for (int u = 0; u < kBatch; ++u) s = fmaf(v[u], g[u], s);
        return s;
    }
};

// d_i = <a_i, x>: one warp per row, its rows consecutive, lanes strided over
// the row; the loads of the next row's first 192 entries are issued before
// this row's gathers of x (L1-resident) and the first row's before grid_wait;
// fixed combination order, warp tree.  The stream of A_q bounds it (70 MB on a
// radiotherapy plan of 55,360 rows: 5.2 TB/s while its CTAs run); a row at a
// time in a grid of 6920 CTAs took 19.1 us, this one 18.0.  Prefetching the
// matrix into L2 during the perturbation phase before it lost 4 us a CQ step.
__global__ void __launch_bounds__(kDoseThreads) k_dvc_dose(DvcArgs a) {
    grid_trigger();
    const int warp = (blockIdx.x * kDoseThreads + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int nw = (gridDim.x * kDoseThreads) >> 5;
    const int i0 = (int)((long long)a.mq * warp / nw), i1 = (int)((long long)a.mq * (warp + 1) / nw);
    Batch next;
    int e0 = 0, e1 = 0;
    if (i0 < i1) {
        e0 = a.rp[i0];
        e1 = a.rp[i0 + 1];
        next.load(a.col, a.val, e0 + lane, 32, e1);
    }
    grid_wait();
    if (a.st && a.st[0].stopped) return;
    for (int i = i0; i < i1; ++i) {
        const Batch cur = next;
        const int f0 = e0, f1 = e1;
        if (i + 1 < i1) {
            e0 = e1;
            e1 = a.rp[i + 2];
            next.load(a.col, a.val, e0 + lane, 32, e1);
        }
        float s = cur.add(0.f, a.x, a.B);
        for (int b = f0 + 32 * kBatch; b < f1; b += 32 * kBatch) {
            Batch more;
            more.load(a.col, a.val, b + lane, 32, f1);
            s = more.add(s, a.x, a.B);
        }
        s = warp_sum_f(s);
        if (lane == 0) a.dose[i] = s;
    }
}

// CTA-wide sum of one int per thread (all threads get the result).
__device__ __forceinline__ int cta_count(int v, int* red) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) red[wid] = v;
    __syncthreads();
    int t = 0;
    for (int w = 0; w < kProjectThreads / 32; ++w) t += red[w];
    return t;
}

// Float-float value hi + lo: the squared corrections are summed in FP32
// arithmetic with error-free transformations (FP64 throughput is far below
// FP32 on this part; FP64 appears only in the per-DVC total).
struct Ff {
    float hi, lo;
};

__device__ __forceinline__ Ff ff_add(Ff a, Ff b) {
    const float s = a.hi + b.hi;
    const float bb = s - a.hi;
    const float e = (a.hi - (s - bb)) + (b.hi - bb) + (a.lo + b.lo);
    const float hi = s + e;
    return Ff{hi, e - (hi - s)};
}

// d_ref - d as float-float (d_ref = ref_hi + ref_lo)
__device__ __forceinline__ Ff ff_diff(float ref_hi, float ref_lo, float d) {
    const float s = ref_hi - d;
    const float bb = s - ref_hi;
    const float t = (ref_hi - (s - bb)) + (-d - bb);
    const float lo = t + ref_lo;
    const float hi = s + lo;
    return Ff{hi, lo - (hi - s)};
}

__device__ __forceinline__ Ff ff_sq(Ff e) {
    const float p = e.hi * e.hi;
    float q = fmaf(e.hi, e.hi, -p);
    q = fmaf(2.f * e.hi, e.lo, q);
    const float hi = p + q;
    return Ff{hi, q - (hi - p)};
}

__device__ __forceinline__ Ff warp_ff(Ff v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const Ff w{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
        v = ff_add(v, w);
    }
    return v;
}

__device__ __forceinline__ float key_dose(uint32_t k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// Radix selection digits: four bytes of the 32-bit key, from the top (wider
// digits make the cluster-wide histogram exchange cost more than the rounds
// they save).
constexpr int kBins = 256;
constexpr int kRounds = 4;
__device__ __forceinline__ int digit_shift(int r) { return 24 - 8 * r; }
__device__ __forceinline__ uint32_t digit_mask(int) { return 0xffu; }

// One thread-block cluster per structure (kDvcCluster CTAs, each a
// contiguous chunk of the structure's rows): for each DVC of the structure in
// the given order, decide the set's projection of the structure's doses, add
// w_j (P_Qj(d) - d) to the corrections and write this CTA's part of
// ||P_Qj(d) - d||^2.  Per DVC: the first pass counts the doses beyond d_ref
// and builds the histogram of the top digit; up to three more passes refine the
// K-th highest key; the apply pass moves the doses.  Histograms are combined
// over the cluster through distributed shared memory after a cluster barrier
// (fixed rank order); they are double-buffered by round, so a CTA never
// clears a histogram that a slower CTA may still be reading.  SMEM: the
// chunk's keys are staged in shared memory once; otherwise every pass
// re-reads the doses.
template <bool SMEM>
__global__ void __launch_bounds__(kProjectThreads) k_dvc_project(DvcArgs a) {
    grid_trigger();
    grid_wait();
    if (a.st && a.st[0].stopped) return;          // uniform over the grid
    cg::cluster_group cl = cg::this_cluster();
    constexpr int CL = kDvcCluster;               // the launch's cluster size
    const int crank = (int)cl.block_rank();
    extern __shared__ uint32_t skey[];
    const int s = blockIdx.x / CL;
    const int r0 = a.sptr[s], N = a.sptr[s + 1] - r0;
    const int chunk = (N + CL - 1) / CL;
    const int c0 = min(N, crank * chunk), nloc = min(N, c0 + chunk) - c0;
    const int base_row = r0 + c0;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    __shared__ int hist[2][kBins];     // this CTA's histogram (double-buffered by round)
    __shared__ int ghist[kBins];       // the cluster's histogram
    __shared__ int red[kProjectThreads / 32];
    __shared__ Ff fred[kProjectThreads / 32];
    __shared__ uint32_t sh_prefix;
    __shared__ int sh_rank, sh_bin, sh_geq, sh_eqbase;
    __shared__ int slot_cnt[2];        // this CTA's count, double-buffered by DVC
    auto key_at = [&](int j) -> uint32_t {   // j in [0, nloc)
        if constexpr (SMEM) return skey[j];
        else return dose_key(a.dose[base_row + j]);
    };

    for (int j = tid; j < nloc; j += kProjectThreads) {
        a.corr[base_row + j] = 0.f;
        if constexpr (SMEM) skey[j] = dose_key(a.dose[base_row + j]);
    }
    int buf = 0;
    for (int q = a.sdvc[s], par = 0; q < a.sdvc[s + 1]; ++q, par ^= 1) {
        const DvcDesc dv = a.dvc[q];
        const bool upper = (dv.kind == 0);
        const int K = dv.K;
        const bool none_kept = (K == 0);
        uint32_t prefix = 0, mask = 0;
        int kk = K, eq_base = 0;
        bool feasible = false, need_order = false;
        for (int r = 0; r < kRounds; ++r, buf ^= 1) {
            const int shift = digit_shift(r);
            const uint32_t dm = digit_mask(r);
            int* h = hist[buf];
            for (int b = tid; b < kBins; b += kProjectThreads) h[b] = 0;
            __syncthreads();
            int cnt = 0;
            for (int base = 0; base < nloc; base += kProjectThreads) {
                const int j = base + tid;
                bool on = false;
                uint32_t bin = 0;
                if (j < nloc) {
                    const uint32_t key = key_at(j);
                    // first pass: also the doses beyond d_ref, compared with
                    // the FP64 d_ref exactly on keys (d > d_ref iff
                    // key > key_gt, d >= d_ref iff key >= key_ge)
                    if (r == 0) cnt += upper ? (key > dv.key_gt) : (key >= dv.key_ge);
                    on = (key & mask) == prefix;
                    bin = (key >> shift) & dm;
                }
                // warp-aggregated increments (many equal doses share a bin)
                const unsigned act = __ballot_sync(0xffffffffu, on);
                if (on) {
                    const unsigned peers = __match_any_sync(act, bin);
                    if ((int)(__ffs(peers) - 1) == lane) atomicAdd(&h[bin], __popc(peers));
                }
            }
            if (r == 0) {
                cnt = cta_count(cnt, red);
                if (tid == 0) slot_cnt[par] = cnt;
            }
            cl.sync();
            if (r == 0) {
                if (tid == 0) {
                    int v[CL];
#pragma unroll
                    for (int rr = 0; rr < CL; ++rr) v[rr] = *cl.map_shared_rank(slot_cnt + par, rr);
                    int t = 0;
#pragma unroll
                    for (int rr = 0; rr < CL; ++rr) t += v[rr];
                    sh_rank = t;
                }
                __syncthreads();
                const int total = sh_rank;
                feasible = upper ? (total <= K) : (total >= K);
                __syncthreads();
                if (feasible || none_kept) {
                    buf ^= 1;
                    break;
                }
            }
            for (int b = tid; b < kBins; b += kProjectThreads) {
                int v[CL];
#pragma unroll
                for (int rr = 0; rr < CL; ++rr) v[rr] = cl.map_shared_rank(h, rr)[b];
                int t = 0;
#pragma unroll
                for (int rr = 0; rr < CL; ++rr) t += v[rr];
                ghist[b] = t;
            }
            __syncthreads();
            if (wid == 0) {
                // bins from the top: lane L holds bins 255-8L .. 248-8L; the
                // lane whose range holds the kk-th highest key picks the bin
                // and the rank left inside it
                const int nb = (int)dm + 1, per = nb / 32;
                const int top = nb - 1 - per * lane;
                int tot = 0;
                for (int k = 0; k < per; ++k) tot += ghist[top - k];
                int incl = tot;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int v = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += v;
                }
                const int excl = incl - tot;
                if (excl < kk && kk <= incl) {
                    int above = excl, k = 0;
                    for (; k < per - 1; ++k) {
                        if (above + ghist[top - k] >= kk) break;
                        above += ghist[top - k];
                    }
                    sh_prefix = prefix | ((uint32_t)(top - k) << shift);
                    sh_rank = kk - above;
                    sh_bin = top - k;
                    sh_geq = ghist[top - k];
                }
            }
            __syncthreads();
            prefix = sh_prefix;
            kk = sh_rank;
            mask |= dm << shift;
            if (r == kRounds - 1) {
                // all keys equal to the threshold are kept unless rank falls
                // short of their number; then the ones in the chunks of lower
                // rank come first (their counts: the last round's bin of
                // those CTAs)
                need_order = kk < sh_geq;
                if (need_order && tid < 32) {
                    const int v = (lane < crank) ? cl.map_shared_rank(h, lane)[sh_bin] : 0;
                    int t = v;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                    if (lane == 0) sh_eqbase = t;
                }
                __syncthreads();
                eq_base = sh_eqbase;
            }
        }
        Ff acc{0.f, 0.f};
        if (!feasible) {
            const uint32_t thr = none_kept ? 0xffffffffu : prefix;
            const int rank = kk;
            // apply in row order; a running count ranks the keys equal to thr
            for (int base = 0; base < nloc; base += kProjectThreads) {
                const int j = base + tid;
                const bool in = j < nloc;
                const uint32_t key = in ? key_at(j) : 0u;
                const bool eq = in && !none_kept && key == thr;
                int before = eq_base, tile_total = 0;
                if (need_order) {
                    const unsigned bal = __ballot_sync(0xffffffffu, eq);
                    __syncthreads();
                    if (lane == 0) red[wid] = __popc(bal);
                    __syncthreads();
                    for (int w = 0; w < kProjectThreads / 32; ++w) {
                        const int rr = red[w];
                        before += (w < wid) ? rr : 0;
                        tile_total += rr;
                    }
                    before += __popc(bal & ((1u << lane) - 1u));
                }
                eq_base += tile_total;
                if (in) {
                    const bool kept = !none_kept && (key > thr || (eq && (!need_order || before < rank)));
                    const bool moves = upper ? (!kept && key > dv.key_gt) : (kept && key < dv.key_ge);
                    if (moves) {
                        const Ff e = ff_diff(dv.ref_hi, dv.ref_lo, key_dose(key));
                        a.corr[base_row + j] += dv.wf * e.hi;
                        acc = ff_add(acc, ff_sq(e));
                    }
                }
            }
        }
        // this CTA's sum of the squared corrections (warp tree, warps in
        // order); the chunks are added in rank order by k_dvc_total
        acc = warp_ff(acc);
        __syncthreads();
        if (lane == 0) fred[wid] = acc;
        __syncthreads();
        if (wid == 0) {
            const Ff t = warp_ff(fred[lane]);
            if (lane == 0) a.pd[(size_t)dv.orig * CL + crank] = (double)t.hi + (double)t.lo;
        }
    }
    cl.sync();    // no CTA leaves while another may still read its shared memory
}

// Target-space proximity: 1/2 w_j times each DVC's chunk sums (chunks in rank
// order), the DVCs in the caller's order; one thread.
__device__ __forceinline__ void dvc_total(const DvcArgs& a) {
    const double hw = 0.5 / (double)a.ndvc;
    double t = 0.0;
    for (int j = 0; j < a.ndvc; ++j) {
        double u = 0.0;
        for (int r = 0; r < kDvcCluster; ++r) u += __ldcg(a.pd + (size_t)j * kDvcCluster + r);
        t += hw * u;
    }
    a.target[0] = t;
}
__global__ void k_dvc_total(DvcArgs a) {
    grid_trigger();
    grid_wait();
    if (a.st && a.st[0].stopped) return;
    if (threadIdx.x == 0) dvc_total(a);
}

// x_j += gamma sum_i a_ij corr_i over the CSC copy: W warps per column (W
// chosen from the mean column length), lanes strided over the column, the
// first entries of the CTA's next columns loaded before this one's gathers of
// the corrections; per-warp sums added in warp order.  The last CTA sums the
// target-space proximity beside the others.  The stream of the CSC copy bounds
// it (70 MB on a radiotherapy plan of 6003 columns); a CTA and eight warps a
// column took 26.5 us there and the sum's own launch 4.9, this one 20.9 (eight
// warps 28.7: a barrier a column of 1455 entries; two warps the same as four).
template <int W>
__global__ void __launch_bounds__(kApplyThreads) k_dvc_apply(DvcArgs a) {
    constexpr int kGroups = kApplyThreads / (32 * W);
    constexpr int kStep = 32 * W;
    __shared__ float part[2][kApplyThreads / 32];
    grid_trigger();
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = wid / W, wg = wid % W;
    const int ctas = gridDim.x - 1;
    if ((int)blockIdx.x == ctas) {
        grid_wait();
        if (threadIdx.x == 0 && !(a.st && a.st[0].stopped)) dvc_total(a);
        return;
    }
    const int stride = ctas * kGroups, off = wg * 32 + lane;
    int j = blockIdx.x * kGroups + g;
    Batch next;
    int e0 = 0, e1 = 0;
    if (j < a.n) {
        e0 = a.cp[j];
        e1 = a.cp[j + 1];
    }
    next.load(a.crow, a.cval, e0 + off, kStep, e1);
    grid_wait();
    if (a.st && a.st[0].stopped) return;
    for (int j0 = blockIdx.x * kGroups, par = 0; j0 < a.n; j0 += stride, j += stride, par ^= 1) {
        const Batch cur = next;
        const int f0 = e0, f1 = e1;
        e0 = e1 = 0;
        if (j + stride < a.n) {
            e0 = a.cp[j + stride];
            e1 = a.cp[j + stride + 1];
        }
        next.load(a.crow, a.cval, e0 + off, kStep, e1);
        float sum = cur.add(0.f, a.corr, 1);
        for (int b = f0 + kBatch * kStep; b < f1; b += kBatch * kStep) {
            Batch more;
            more.load(a.crow, a.cval, b + off, kStep, f1);
            sum = more.add(sum, a.corr, 1);
        }
        const float ws = warp_sum_f(sum);
        if (lane == 0) part[par][wid] = ws;
        __syncthreads();   // the next column's sums go to the other half
        if (wg == 0 && lane == 0 && j < a.n && f1 > f0) {
            float t = 0.f;
#pragma unroll
            for (int w = 0; w < W; ++w) t += part[par][g * W + w];
            float* xj = a.xw + (size_t)j * a.B;
            *xj = *xj + a.gamma * t;
        }
    }
}

// ||A_s||_F^2 per structure (FP64, fixed order): CTA (s, c) sums chunk c of
// structure s's entries, then one thread per structure adds the chunks in
// order.
constexpr int kFrobChunks = 32;
__global__ void __launch_bounds__(kDoseThreads) k_dvc_frob(const int* rp, const float* val,
                                                           const int* sptr, double* part) {
    const int s = blockIdx.x / kFrobChunks, c = blockIdx.x % kFrobChunks;
    const long long e0 = rp[sptr[s]], e1 = rp[sptr[s + 1]];
    const long long len = (e1 - e0 + kFrobChunks - 1) / kFrobChunks;
    const long long b0 = e0 + (long long)c * len, b1 = min(e1, b0 + len);
    double acc = 0.0;
    for (long long e = b0 + threadIdx.x; e < b1; e += kDoseThreads) {
        const double v = (double)val[e];
        acc += v * v;
    }
    acc = warp_sum(acc);
    __shared__ double sw[kDoseThreads / 32];
    if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kDoseThreads / 32; ++w) t += sw[w];
        part[blockIdx.x] = t;
    }
}

__global__ void k_dvc_frob_sum(const double* part, int nstruct, double* out) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nstruct) return;
    double t = 0.0;
    for (int c = 0; c < kFrobChunks; ++c) t += part[(size_t)s * kFrobChunks + c];
    out[s] = t;
}

}  // namespace

// resident CTAs of a kernel on the device (the passes above run in one wave)
template <class F>
static int wave(F f, int threads) {
    int dev = 0, sms = 0, nb = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, f, threads, 0) != cudaSuccess)
        return 0;
    return sms * nb;
}

int dvc_dose_grid(int mq) {
    return (int)std::min<long long>(((long long)mq * 32 + kDoseThreads - 1) / kDoseThreads,
                                    wave(k_dvc_dose, kDoseThreads));
}

cudaError_t launch_dvc_dose(const DvcArgs& a, cudaStream_t s) {
    if (a.mq <= 0) return cudaSuccess;
    return launch_dependent(k_dvc_dose, a.dose_grid, kDoseThreads, 0, s, a);
}

size_t dvc_project_smem(int max_rows) {
    const size_t b = (size_t)((max_rows + kDvcCluster - 1) / kDvcCluster) * sizeof(uint32_t);
    return b <= kDvcSmemMax ? b : 0;
}

cudaError_t launch_dvc_project(const DvcArgs& a, cudaStream_t s, bool total) {
    if (a.nstruct > 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(a.nstruct * kDvcCluster, 1, 1);
        cfg.blockDim = dim3(kProjectThreads, 1, 1);
        cfg.dynamicSmemBytes = a.smem;
        cfg.stream = s;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = kDvcCluster;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
        cudaError_t e;
        if (a.smem > 0) {
            e = cudaFuncSetAttribute(k_dvc_project<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)a.smem);
            if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, k_dvc_project<true>, a);
        } else {
            e = cudaLaunchKernelEx(&cfg, k_dvc_project<false>, a);
        }
        if (e != cudaSuccess) return e;
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return total ? launch_dependent(k_dvc_total, 1, 32, 0, s, a) : cudaSuccess;
}

// Warps per column from the mean column length (eight lose at 1455 entries, see
// k_dvc_apply).
static int apply_warps(int n, long long nnz) {
    const long long mean = n > 0 ? nnz / n : 0;
    return mean >= 512 ? 4 : mean >= 256 ? 2 : 1;
}
template <class R, class F>
static R with_apply(int n, long long nnz, F f) {
    switch (apply_warps(n, nnz)) {
        case 4: return f(k_dvc_apply<4>);
        case 2: return f(k_dvc_apply<2>);
        default: return f(k_dvc_apply<1>);
    }
}

int dvc_apply_grid(int n, long long nnz) {
    const int groups = kApplyThreads / (32 * apply_warps(n, nnz));
    const int one = with_apply<int>(n, nnz, [](auto k) { return wave(k, kApplyThreads); }) - 1;
    return 1 + std::min((n + groups - 1) / groups, one);   // the last CTA sums the proximity
}

cudaError_t launch_dvc_apply(const DvcArgs& a, cudaStream_t s) {
    if (a.n <= 0) return cudaSuccess;
    return with_apply<cudaError_t>(a.n, a.nnz, [&](auto k) {
        return launch_dependent(k, a.apply_grid, kApplyThreads, 0, s, a);
    });
}

cudaError_t launch_dvc_frob(const int* rp, const float* val, const int* sptr, int nstruct,
                            double* part, double* out, cudaStream_t s) {
    if (nstruct <= 0) return cudaSuccess;
    k_dvc_frob<<<nstruct * kFrobChunks, kDoseThreads, 0, s>>>(rp, val, sptr, part);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_dvc_frob_sum<<<(nstruct + 127) / 128, 128, 0, s>>>(part, nstruct, out);
    return cudaGetLastError();
}

}  // namespace suppy
