// Strip-ordered streaming passes of the simultaneous projection sweep
// (Sec. 2.1.1, Eq. (3)) for one right-hand side.
//
// A strip is up to four consecutive items: rows of the CSR copy (row pass) or
// columns of the CSC copy (column pass) of A.  Its entries are stored as a
// sequence of packets of 128 slots, in the order the lanes of a warp take
// them: lanes 8r .. 8r+7 hold item r, and step s of a packet (s = 0..3) gives
// each item eight consecutive entries.  A packet's entries come from the same
// stretch of all four items (windows of at most 32 entries an item, cut where
// the sorted keys of the items agree), so that the four neighbouring rays of a
// CT or travel-time matrix are read side by side: one warp instruction covers
// a patch of 4 x 8 neighbouring pixels instead of a line of 32.  Sectors are
// what the gathers of x and the L2 reductions cost, and counted on CT 512x512
// (360 angles x 725 bins) in the patch numbering they fall from 41.6 M to
// 27.0 M a sweep; the padding of the windows costs 4.6% more slots.
//
// A packet is {four bases (int32, one an item), for the scatter the lanes'
// flags, 128 16-bit offsets, 128 values}: position = base of the item + offset, so an entry costs 6 bytes
// instead of 8 (FP32 values; nothing is rounded, a window ends where an
// offset would not fit) and a lane reads its four entries of a packet with
// one 4-byte, one 8-byte and one 16-byte shared-memory load.
//
// The passes are dependent launches: the strips are constants, so that the
// producer fills the ring while the kernel before still runs, and only the
// consumers wait for it (the launch, the first copies and the drain of 20 us
// block passes overlap: CT 128x128 in 10 blocks 112 -> 101 us an iteration,
// CT 512x512 in 36 blocks 764 -> 709).
//
// Each CTA (one per SM) owns a contiguous range of strips, balanced by their
// packets.  One producer warp streams whole strips into a shared-memory ring
// with bulk copies (cp.async.bulk) tracked by mbarriers, each strip in one
// contiguous piece; 24 consumer warps in groups of NW take the strips in
// turn, each warp a contiguous share of the strip's packets.  The dot
// products are summed over the eight lanes and then over the group's warps in
// a fixed order; the scatter reads the strip again from the ring.
//
// In the one-pass scatter, entries of neighbouring rows on the same pixel (18%
// of CT entries, most of a dose matrix's) are placed in the same slot of their
// items: the first item's lane adds the others' shares to its own (their
// values lie beside its own in the packet), so that a pixel is reduced once
// and no instruction reduces an address twice, which would split it.
//
// Measured (GB300, CT 512x512, 120.3 M entries, FP32; the streamed passes of
// stream.cu in their default shapes before): two-pass row pass 227 -> 152 us,
// column pass 196 -> 136 us (775 and 824 MB of DRAM, 5.1 and 6.0 TB/s of the 6.7
// copied), one-pass row pass 342 -> 207 us.  The scatter's L2 reductions (26.7 M
// sectors; 39 M before shared pixels were joined, 253 us) share the
// load/store pipe and the issue slots with the gathers: without them the
// one-pass row pass takes 127 us.
#include <algorithm>
#include <climits>

#include "check.cuh"
#include "common.cuh"
#include "tma.cuh"

namespace suppy {

cudaError_t read_check_word_strip(int* out3) { return take_check_words(out3); }

namespace {

using tma::bulk_g2s;
using tma::mbar_arrive;
using tma::mbar_arrive_expect_tx;
using tma::mbar_init;

constexpr int kConsumers = kStripThreads / 32 - 1;    // consumer warps (and one producer)
constexpr int kInFlight = kStripInFlight;             // strips in the ring: their barriers
constexpr int kPad = 0xffff;                          // offset of an empty slot
constexpr long long kDrainCycles = 4000000000LL;      // copies in flight get this long to land

template <typename VT>
struct Val4;
template <>
struct Val4<float> {
    static __device__ __forceinline__ float4 load(const unsigned char* p) {
        return *reinterpret_cast<const float4*>(p);
    }
};
template <>
struct Val4<__nv_bfloat16> {
    static __device__ __forceinline__ float4 load(const unsigned char* p) {
        const uint2 u = *reinterpret_cast<const uint2*>(p);
        return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u),
                           __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
    }
};
template <>
struct Val4<__half> {
    static __device__ __forceinline__ float4 load(const unsigned char* p) {
        const uint2 u = *reinterpret_cast<const uint2*>(p);
        const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&u.x));
        const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
        return make_float4(a.x, a.y, b.x, b.y);
    }
};

__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(tma::smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait: gives up (false) when `abort` is raised or `limit` cycles pass
// before the phase completes.
__device__ __forceinline__ bool bounded_wait(uint64_t* bar, uint32_t parity, volatile int* abort,
                                             long long limit) {
    if (mbar_test(bar, parity)) return true;
    const long long t0 = clock64();
    do {
        if (*abort || clock64() - t0 > limit) return false;
    } while (!tma::mbar_try_wait(bar, parity));
    return true;
}

// Barrier of a consumer group that also decides whether every thread is ok.
template <int NW>
__device__ __forceinline__ bool group_all(int grp, bool ok) {
    if constexpr (NW == 1) {
        return __all_sync(0xffffffffu, ok);
    } else {
        int r;
        asm volatile(
            "{\n\t.reg .pred p, q;\n\t"
            "setp.ne.s32 q, %3, 0;\n\t"
            "barrier.cta.red.and.pred p, %1, %2, q;\n\t"
            "selp.s32 %0, 1, 0, p;\n\t}"
            : "=r"(r)
            : "r"(grp + 1), "r"(NW * 32), "r"((int)ok)
            : "memory");
        return r != 0;
    }
}

template <typename VT, int KIND>
struct Packet {
    static constexpr int kBytes = strip_packet_bytes(sizeof(VT), KIND == 1);
    static constexpr int kIdx = KIND == 1 ? 80 : 16, kVal = kIdx + 256;   // after bases and flags
};

// x[base + o], 0 in an empty slot.  A coherent load: this kernel may have started
// before the one that writes x ended, so x is not read-only for its lifetime, as
// .nc would promise (same times either way).
__device__ __forceinline__ float gather(const float* x, int base, unsigned o) {
    float g;
    asm("{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %2, 65535;\n\t"
        "mov.f32 %0, 0f00000000;\n\t"
        "@p ld.global.f32 %0, [%1];\n\t}"
        : "=f"(g)
        : "l"(x + (base + (int)o)), "r"(o));
    return g;
}
// Sums a lane adds its products to.  Four keep the error of the two-pass sweep
// where the streamed passes have it (CT 257x257, DROP, distance from FP64
// 7.15e-8 streamed, 7.17e-8 with two, 7.10e-8 with four; same time); the
// scatter's row pass has no registers for them (512x512 1332 -> 1342 us a call)
// and is the more exact one as it is (1.21e-7 streamed, 1.14e-7).
template <int KIND>
constexpr int kSums = KIND == 1 ? 2 : 4;

// N packets from p: their loads, then their gathers together, then the
// products, so that they cost one gather latency.
template <typename VT, int KIND, int N>
__device__ __forceinline__ void dot_packets(const unsigned char* p, int lane, const float* __restrict__ x,
                                            long long x_len, float (&acc)[kSums<KIND>]) {
    int base[N];
    uint2 w[N];
    float4 v[N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const unsigned char* q = p + k * Packet<VT, KIND>::kBytes;
        base[k] = *reinterpret_cast<const int*>(q + 4 * (lane >> 3)) & 0x7fffffff;
        w[k] = *reinterpret_cast<const uint2*>(q + Packet<VT, KIND>::kIdx + 8 * lane);
        v[k] = Val4<VT>::load(q + Packet<VT, KIND>::kVal + lane * 4 * (int)sizeof(VT));
    }
    float g[N][4];
#pragma unroll
    for (int k = 0; k < N; ++k) {
        unsigned o[4] = {w[k].x & 0xffffu, w[k].x >> 16, w[k].y & 0xffffu, w[k].y >> 16};
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            if (!CHECKED(o[s] == kPad || (base[k] >= 0 && base[k] + (long long)o[s] < x_len), 501, base[k])) o[s] = kPad;
            g[k][s] = gather(x, base[k], o[s]);
        }
    }
#pragma unroll
    for (int k = 0; k < N; ++k) {
        acc[0] = fmaf(v[k].x, g[k][0], acc[0]);
        acc[1] = fmaf(v[k].y, g[k][1], acc[1]);
        acc[2 % kSums<KIND>] = fmaf(v[k].z, g[k][2], acc[2 % kSums<KIND>]);
        acc[3 % kSums<KIND>] = fmaf(v[k].w, g[k][3], acc[3 % kSums<KIND>]);
    }
}

// s += c u where bit `B` of f is set, as predicated instructions (the compiler
// makes a branch of each otherwise).
template <unsigned B>
__device__ __forceinline__ void fma_if(unsigned f, float c, float u, float& s) {
    asm("{\n\t.reg .pred p;\n\t.reg .u32 t;\n\t"
        "and.b32 t, %1, %4;\n\t"
        "setp.ne.u32 p, t, 0;\n\t"
        "@p fma.rn.f32 %0, %2, %3, %0;\n\t}"
        : "+f"(s)
        : "r"(f), "f"(c), "f"(u), "n"(B));
}

// L2 reduction of v into *p where bit B of f is clear.
template <unsigned B>
__device__ __forceinline__ void red_unless(unsigned f, float* p, float v) {
    asm volatile("{\n\t.reg .pred p;\n\t.reg .u32 t;\n\t"
                 "and.b32 t, %1, %3;\n\t"
                 "setp.eq.u32 p, t, 0;\n\t"
                 "@p red.relaxed.gpu.global.add.f32 [%0], %2;\n\t}" ::"l"(p),
                 "r"(f), "f"(v), "n"(B)
                 : "memory");
}

// The corrections of one packet (KIND 1).  The lane's flags: bits 0-3, entries
// it does not add (empty, or added by an earlier item's lane); bits 4-7, 8-11,
// 12-15, entries whose position the first, second and third item after its own
// hold in the same slot, which it adds with its own.  c0 .. c3: the
// coefficients of the lane's item and of those after it (0 past the strip).
template <typename VT>
__device__ __forceinline__ void scatter_packet(const unsigned char* sp, int lane, float c0, float c1, float c2,
                                               float c3, float* __restrict__ dst, long long dst_len) {
    using Pk = Packet<VT, 1>;
    constexpr int kItem = 8 * 4 * (int)sizeof(VT);   // bytes from one item's values to the next's
    const int word = *reinterpret_cast<const int*>(sp + 4 * (lane >> 3));
    const int base = word & 0x7fffffff;
    unsigned f = *reinterpret_cast<const unsigned short*>(sp + 16 + 2 * lane);
    const uint2 ix = *reinterpret_cast<const uint2*>(sp + Pk::kIdx + 8 * lane);
    const unsigned char* vp = sp + Pk::kVal + lane * 4 * (int)sizeof(VT);
    const float4 v = Val4<VT>::load(vp);
    // the next item's values (its own again for the last item: no flags)
    const float4 u = Val4<VT>::load(lane < 24 ? vp + kItem : vp);
    float s[4] = {c0 * v.x, c0 * v.y, c0 * v.z, c0 * v.w};
    fma_if<0x10u>(f, c1, u.x, s[0]);
    fma_if<0x20u>(f, c1, u.y, s[1]);
    fma_if<0x40u>(f, c1, u.z, s[2]);
    fma_if<0x80u>(f, c1, u.w, s[3]);
    if (word < 0) {   // uniform: the packet has positions of three or four items
        const float4 u2 = Val4<VT>::load(lane < 16 ? vp + 2 * kItem : vp);
        const float4 u3 = Val4<VT>::load(lane < 8 ? vp + 3 * kItem : vp);
        fma_if<0x100u>(f, c2, u2.x, s[0]);
        fma_if<0x200u>(f, c2, u2.y, s[1]);
        fma_if<0x400u>(f, c2, u2.z, s[2]);
        fma_if<0x800u>(f, c2, u2.w, s[3]);
        fma_if<0x1000u>(f, c3, u3.x, s[0]);
        fma_if<0x2000u>(f, c3, u3.y, s[1]);
        fma_if<0x4000u>(f, c3, u3.z, s[2]);
        fma_if<0x8000u>(f, c3, u3.w, s[3]);
    }
    // a row inside its slab adds nothing of its own
    if (c0 == 0.f) f |= ~(f >> 4) & 0xfu;
    const unsigned off[4] = {ix.x & 0xffffu, ix.x >> 16, ix.y & 0xffffu, ix.y >> 16};
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (!CHECKED(((f >> k) & 1u) || (base >= 0 && base + (long long)off[k] < dst_len), 502, base)) f |= 1u << k;
    float* const d = dst + base;
    red_unless<1u>(f, d + off[0], s[0]);
    red_unless<2u>(f, d + off[1], s[1]);
    red_unless<4u>(f, d + off[2], s[2]);
    red_unless<8u>(f, d + off[3], s[3]);
}

// KIND 0: row pass, coefficients out; 1: row pass with the scatter by L2
// reductions (COPIES: into kDeltaCopies accumulators); 2: column pass.
template <typename VT, int NW, int KIND, bool COPIES>
__global__ void __launch_bounds__(kStripThreads, 1) k_strip(const StripArgs a) {
    extern __shared__ __align__(128) unsigned char ring[];
    __shared__ __align__(8) uint64_t full[kInFlight], empty[kInFlight];
    __shared__ float part[2][kConsumers][4];
    __shared__ volatile int abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int s0 = a.cta[blockIdx.x], s1 = a.cta[blockIdx.x + 1];
    if (!CHECKED(s0 >= 0 && s0 <= s1 && s1 <= a.strips && ALIGNED16(ring) && ALIGNED16(a.blob), 503, blockIdx.x)) s0 = s1 = 0;
    constexpr int NG = kConsumers / NW;
    // a group waits for the fills of its own barriers only, in order: the wait
    // for one fill can never be taken for the fill before it
    static_assert(kInFlight % NG == 0, "a barrier's strips belong to one group");
    if (threadIdx.x == 0) {
        for (int k = 0; k < kInFlight; ++k) {
            mbar_init(&full[k], 1);
            mbar_init(&empty[k], NW);
        }
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (a.early) grid_trigger();
    // sums of the lanes that hold an item: the proximity terms (row pass), the
    // squares of the sums (column pass).  FP64, but for the coefficients' row
    // pass, which has nothing to hide FP64's 16 cycles of an SM a warp
    // instruction behind (EL on 71x48, 316 angles: 24.6 us with compensated FP32
    // sums, as in the streamed passes it stands in for, 25.4 with FP64 terms)
    double sq = 0.0;
    float ps = 0.f, pc = 0.f;
    bool stopped = false;
    int oldest = 0, issued = 0;   // producer: strips whose ring space came back, strips issued
    if (warp == 0) {
        uint64_t pol;
        if (a.keep) asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
        else pol = tma::policy_evict_first();
        // 32 strips at a time, one a lane: each goes out as soon as the strips
        // whose ring space it takes have come back (the places in the ring
        // were laid out with the records), so that a strip costs the producer
        // one wait and one copy
        int4 nxt = (s0 + lane < s1) ? a.meta[s0 + lane] : make_int4(0, 0, 0, 0);
        int back = 0, back_fill = 0;   // barriers of the oldest strip in the ring
        bool ok = true;
        for (int b = s0; ok && b < s1; b += 32) {
            const int4 m = nxt;
            nxt = (b + 32 + lane < s1) ? a.meta[b + 32 + lane] : make_int4(0, 0, 0, 0);
            const int q = b - s0 + lane;
            const int need = q - strip_live(m.w);
            uint32_t bytes = (uint32_t)((m.y & kStripPackets) * Packet<VT, KIND>::kBytes);
            if (!CHECKED(strip_at(m.w) + (long long)bytes <= a.ring &&
                             ((long long)(unsigned)m.x << 4) + bytes <= a.blob_bytes,
                         504, b + lane))
                bytes = 0;
            bool done = b + lane >= s1;
            for (;;) {
                if (!done && need <= oldest) {
                    uint64_t* bar = &full[q % kInFlight];
                    mbar_arrive_expect_tx(bar, bytes);
                    if (bytes)
                        bulk_g2s(ring + strip_at(m.w), a.blob + ((size_t)(unsigned)m.x << 4), bytes, bar, pol);
                    done = true;
                }
                issued = b - s0 + __popc(__ballot_sync(0xffffffffu, done && b + lane < s1));
                if (__all_sync(0xffffffffu, done)) break;
                // the ring is full, and nothing comes back before the kernel
                // ahead is over: it is waited for before a wait's budget starts
                grid_wait();
                ok = __all_sync(0xffffffffu, bounded_wait(&empty[back], back_fill, &abort_flag, a.wait_cycles));
                if (!ok) break;
                ++oldest;
                if (++back == kInFlight) {
                    back = 0;
                    back_fill ^= 1;
                }
            }
        }
        // the strips are constants: they stream in while the kernel before this
        // one ends.  A stopped system's consumers leave at once (abort_flag 2)
        grid_wait();
        if (lane == 0 && !ok && abort_flag != 2) {
            abort_flag = 1;
            atomicExch(a.err, 1);
        }
    } else {
        const int cw = warp - 1, grp = cw / NW, wi = cw % NW;
        const int r = lane >> 3;
        int par = 0, slot = grp, fill = 0;   // the strip's barriers, and which fill of them
        int4 nxt = (grp < s1 - s0) ? __ldg(a.meta + s0 + grp) : make_int4(0, 0, 0, 0);
        grid_wait();
        // a stopped system takes no step (and its row pass left no
        // coefficients): looked at after the first strip's sums, whose loads
        // need not wait for the flag's
        const int flag = KIND == 2 ? a.epi.st[0].stopped : (a.check_stop ? a.st[0].stopped : 0);
        for (int q = grp; q < s1 - s0; q += NG, par ^= 1) {
            int4 m = nxt;
            constexpr long long kBytes = Packet<VT, KIND>::kBytes;
            if (!CHECKED(strip_at(m.w) + (m.y & kStripPackets) * kBytes <= a.ring &&
                             m.z >= 0 && m.z + (31 - __clz((m.w & 15) | 1)) < a.items,
                         505, s0 + q))
                m = make_int4(0, 0, 0, 0);
            nxt = (q + NG < s1 - s0) ? __ldg(a.meta + s0 + q + NG) : make_int4(0, 0, 0, 0);
            const int npk = m.y & kStripPackets;
            const bool tall = (m.y & kStripTall) != 0;
            const int p0 = npk * wi / NW, p1 = npk * (wi + 1) / NW;
            const int item = m.z + r;
            const bool has = ((m.w >> r) & 1) != 0;   // a row with entries; a column of the strip
            const unsigned char* strip = ring + strip_at(m.w);
            // loads without a branch or a select behind them, which made the
            // strip's sums wait for them (about 500 cycles a strip); lanes
            // without an item repeat the strip's first
            const int from = has ? item : m.z;
            float li, ui, w, mul = 1.f;
            if constexpr (KIND != 2) {
                li = __ldg(a.l + from);
                ui = __ldg(a.u + from);
                w = __ldg(a.wr + from);
                const float* mp = a.coef_mul ? a.coef_mul : a.prox_mul;
                mul = __ldg((mp ? mp : a.wr) + from);
            } else if (wi == 0) {
                li = __ldg(a.lo + (a.box_len == 1 ? 0 : from));
                ui = __ldg(a.hi + (a.box_len == 1 ? 0 : from));
                w = a.xw[from];   // owned by this strip alone during the pass
                mul = __ldg((a.zc ? a.zc : a.lo) + (a.zc ? from : 0));
            }
            bool ok = bounded_wait(&full[slot], fill, &abort_flag, a.wait_cycles);
            float dot = 0.f;
            if (ok) {
                const float* xs = tall ? a.xT : a.x;
                float acc[kSums<KIND>] = {};
                int p = p0;
                const unsigned char* sp = strip + p0 * Packet<VT, KIND>::kBytes;
                for (; p + 4 <= p1; p += 4, sp += 4 * Packet<VT, KIND>::kBytes)
                    dot_packets<VT, KIND, 4>(sp, lane, xs, a.x_len, acc);
                if (p1 - p == 3) dot_packets<VT, KIND, 3>(sp, lane, xs, a.x_len, acc);
                else if (p1 - p == 2) dot_packets<VT, KIND, 2>(sp, lane, xs, a.x_len, acc);
                else if (p1 - p == 1) dot_packets<VT, KIND, 1>(sp, lane, xs, a.x_len, acc);
                dot = KIND == 1 ? acc[0] + acc[1] : (acc[0] + acc[1]) + (acc[2 % kSums<KIND>] + acc[3 % kSums<KIND>]);
            }
            if (KIND != 1) {
                // the strip is read once: its ring space goes back now
                __syncwarp();
                if (ok && lane == 0) mbar_arrive(&empty[slot]);
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
            if (NW > 1 && (lane & 7) == 0) part[par][cw][r] = dot;
            if (flag) break;
            ok = group_all<NW>(grp, ok);
            if (!ok) {
                abort_flag = 1;
                if (lane == 0) atomicExch(a.err, 1);
                break;
            }
            if constexpr (NW > 1) {
                // the other buffer takes the next strip's sums: a warp writes
                // this one again only after the group's next barrier
                dot = part[par][grp * NW][r];
#pragma unroll
                for (int k = 1; k < NW; ++k) dot += part[par][grp * NW + k][r];
            }
            if constexpr (KIND == 2) {
                if (has && wi == 0 && (lane & 7) == 0) {
                    const float s = a.zc ? dot * mul : dot;
                    if (a.delta_out) {
                        a.delta_out[item] = s;
                        if (a.norm) sq += (double)s * (double)s;
                    } else a.xw[item] = clampf(w + s, li, ui);
                }
            } else {
                const float d = clampf(dot, li, ui) - dot;
                const float coef = a.lam * w * d * (a.coef_mul ? mul : 1.f);
                if (has && wi == 0 && (lane & 7) == 0) {
                    if constexpr (KIND == 1) {
                        sq += (double)d * (double)d * (double)(a.prox_mul ? w * mul : w);
                    } else {
                        const float t = d * d * w * (a.prox_mul ? mul : 1.f);
                        const float y = t - pc, sum = ps + y;
                        pc = (sum - ps) - y;
                        ps = sum;
                    }
                    if (KIND == 0 && a.coef) a.coef[item] = coef;
                }
                if constexpr (KIND == 1) {
                    // an entry whose slot holds the same position in the item
                    // before is added by that item's lane (eight lanes back),
                    // which reads its value beside its own: one reduction a
                    // position, and none twice in one instruction
                    const float c0 = has ? coef : 0.f;
                    float c1 = __shfl_down_sync(0xffffffffu, c0, 8), c2 = __shfl_down_sync(0xffffffffu, c0, 16),
                          c3 = __shfl_down_sync(0xffffffffu, c0, 24);
                    if (__any_sync(0xffffffffu, c0 != 0.f)) {
                        float* dst = COPIES ? a.delta + (blockIdx.x % kDeltaCopies) * a.copy
                                            : (tall ? a.deltaT : a.delta);
                        const long long dst_len = COPIES ? a.copy : a.delta_len;
                        const unsigned char* sp = strip + p0 * Packet<VT, KIND>::kBytes;
                        for (int p = p0; p < p1; ++p, sp += Packet<VT, KIND>::kBytes)
                            scatter_packet<VT>(sp, lane, c0, c1, c2, c3, dst, dst_len);
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&empty[slot]);
                }
            }
            slot += NG;
            if (slot >= kInFlight) {
                slot -= kInFlight;
                fill ^= 1;
            }
        }
        stopped = flag != 0;
        if (stopped) abort_flag = 2;
    }
    // a small kernel after the pass starts once its CTAs are through; another
    // strip pass takes each SM as it comes free and fills its ring meanwhile
    if (!a.early) grid_trigger();
    // the values of the lanes that hold any, side by side for one warp's sum:
    // FP64 is scarce, and every warp summing its lanes, then a thread the warps,
    // held the end of each pass for 3950 cycles (1000 to 1600 so)
    __shared__ double sq_s[4 * NG];
    if (KIND == 0) sq = (double)ps - (double)pc;
    if (warp > 0 && (warp - 1) % NW == 0 && (lane & 7) == 0) sq_s[(warp - 1) / NW * 4 + (lane >> 3)] = sq;
    stopped = __syncthreads_or(stopped);
    if (abort_flag && threadIdx.x == 0) {
        // let the copies in flight land before the CTA leaves
        volatile int never = 0;
        for (int q = oldest; q < issued; ++q)
            tma::mbar_wait(&full[q % kInFlight], (q / kInFlight) & 1, &never, kDrainCycles);
    }
    if (KIND == 2 && a.norm && blockIdx.x == 0 && threadIdx.x == 0) *a.was_stopped = stopped;
    if (stopped) return;   // every thread has seen it: nothing of the launch is left out
    if (warp == 0 && (KIND != 2 || a.norm)) {
        double v = 0.0;
        for (int k = lane; k < 4 * NG; k += 32) v += sq_s[k];
        v = warp_sum(v);
        if (lane == 0) (KIND != 2 ? a.pp : a.norm)[blockIdx.x] = v;
    }
    if constexpr (KIND == 2) {
        __syncthreads();
        if (a.epi.last_seg && a.ticket) {
            // the last CTA to finish runs the sweep epilogue: every CTA of the
            // launch has read the stop flag by then, so the flag it may set is
            // seen by the next launch only
            __shared__ bool last;
            __threadfence();
            if (threadIdx.x == 0) last = atomicAdd(a.ticket, 1u) == gridDim.x - 1;
            __syncthreads();
            if (last) {
                __threadfence();
                sweep_epilogue(a.epi);
                if (threadIdx.x == 0) *a.ticket = 0u;
            }
        } else if (blockIdx.x == 0 && !a.epi.last_seg) {
            add_proximity(a.epi);
        }
    }
}

// ------------------------------------------------------------- building ----
// One CTA of four warps per strip, warp r for item r: the item's entries as
// keys in the order the strip walks them, then windows of at most 32 entries
// an item, each window one packet.  Keys: on an image grid the pixel in
// row-major order for strips whose rows run down the image and column-major
// order for the others (so that a ray's entries come in the order of its
// path), else the index itself.  A window ends at the smallest key that an
// item could not take (its 33rd entry, or one whose offset from the window's
// smallest position would not fit 16 bits): all items of the strip then stop
// at the same place.  FILL 0 counts the packets and writes the strip's
// record, FILL 1 writes the packets.
template <typename VT, int FILL>
__global__ void __launch_bounds__(128) k_strip_build(const StripBuild b) {
    extern __shared__ unsigned key_s[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned* raw = key_s + (size_t)warp * 2 * b.max_len;
    unsigned* key = raw + b.max_len;
    unsigned short* ord = reinterpret_cast<unsigned short*>(key_s + (size_t)8 * b.max_len) +
                          (size_t)warp * b.max_len;
    __shared__ int span_s[4][2], cnt_s[4], len_s[4];
    __shared__ unsigned lim_s[4];
    __shared__ int slot_s[4][32];   // positions by slot of the window (-1: none)
    __shared__ unsigned shared_s[4];   // slots shared with the item before
    const VT* val = static_cast<const VT*>(b.val);
    for (int t = blockIdx.x; t < b.nstrips; t += gridDim.x) {
        const int4 st = b.strips[t];   // first item in info, items, first item's number
        const int2 inf = warp < st.y ? b.info[st.x + warp] : make_int2(0, 0);
        const int len = inf.y;
        const int* idx = b.idx + inf.x;
        int r0 = INT_MAX, r1 = -1, c0 = INT_MAX, c1 = -1;
        if (b.W > 0)
            for (int e = lane; e < len; e += 32) {
                const int y = idx[e] / b.W, x = idx[e] - y * b.W;
                r0 = min(r0, y);
                r1 = max(r1, y);
                c0 = min(c0, x);
                c1 = max(c1, x);
            }
        r0 = __reduce_min_sync(0xffffffffu, r0);
        r1 = __reduce_max_sync(0xffffffffu, r1);
        c0 = __reduce_min_sync(0xffffffffu, c0);
        c1 = __reduce_max_sync(0xffffffffu, c1);
        if (lane == 0) {
            span_s[warp][0] = r1 < 0 ? 0 : r1 - r0;
            span_s[warp][1] = c1 < 0 ? 0 : c1 - c0;
            len_s[warp] = len;
        }
        __syncthreads();
        const bool tall = b.W > 0 && span_s[0][0] + span_s[1][0] + span_s[2][0] + span_s[3][0] >
                                         span_s[0][1] + span_s[1][1] + span_s[2][1] + span_s[3][1];
        bool sorted = true;
        for (int e = lane; e < len; e += 32) {
            const int c = idx[e];
            unsigned k = (unsigned)c;
            if (b.W > 0 && !tall) {
                const int y = c / b.W;
                k = (unsigned)((c - y * b.W) * b.H + y);
            }
            raw[e] = k;
        }
        __syncwarp();
        for (int e = lane; e + 1 < len; e += 32) sorted = sorted && raw[e] <= raw[e + 1];
        sorted = __all_sync(0xffffffffu, sorted);
        for (int e = lane; e < len; e += 32) {
            const unsigned k = raw[e];
            int rank = e;
            if (!sorted) {
                rank = 0;
                for (int f = 0; f < len; ++f) rank += raw[f] < k || (raw[f] == k && f < e);
            }
            key[rank] = k;
            ord[rank] = (unsigned short)e;
        }
        __syncwarp();
        int p = 0, npk = 0;
        unsigned char* out = FILL ? b.blob + ((size_t)(unsigned)b.meta[t].x << 4) : nullptr;
        const bool tall_pos = FILL ? (b.meta[t].y & kStripTall) != 0 : tall;
        for (;;) {
            const int left = len - p;
            if (!__syncthreads_or(left > 0)) break;
            int pos = 0, src = 0;
            if (lane < left) {
                src = inf.x + ord[p + lane];
                const int c = b.idx[src];
                pos = b.patch ? patch_index(c, b.recipW, b.W, b.Wp, tall_pos) : c;
            }
            // running extremes of the positions over the window
            int mn = lane < left ? pos : INT_MAX, mx = lane < left ? pos : INT_MIN;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int a0 = __shfl_up_sync(0xffffffffu, mn, o), a1 = __shfl_up_sync(0xffffffffu, mx, o);
                if (lane >= o) {
                    mn = min(mn, a0);
                    mx = max(mx, a1);
                }
            }
            const bool fits = lane < left && (long long)mx - mn < kPad;
            const int c = __popc(__ballot_sync(0xffffffffu, fits));   // a prefix of the lanes
            if (lane == 0) lim_s[warp] = p + c < len ? key[p + c] : 0xffffffffu;
            __syncthreads();
            const unsigned lim = min(min(lim_s[0], lim_s[1]), min(lim_s[2], lim_s[3]));
            int n = __popc(__ballot_sync(0xffffffffu, lane < c && key[p + lane] < lim));
            if (lane == 0) cnt_s[warp] = n;
            __syncthreads();
            // equal keys (repeated columns) may leave nothing below the limit
            if (cnt_s[0] + cnt_s[1] + cnt_s[2] + cnt_s[3] == 0) n = c;
            if constexpr (FILL) {
                const int base = n > 0 ? __shfl_sync(0xffffffffu, mn, n - 1) : 0;
                // the entry's slot of 32: in order, or -- for the scatter -- that
                // of the same position in the item before, the others in order
                // in the slots left
                int slot = lane;
                if (b.scatter) {
                    for (int i = 0; i < 4; ++i) {
                        if (warp == i) {
                            int m = -1;
                            if (i > 0 && lane < n)
                                for (int f = 0; f < 32; ++f)
                                    if (slot_s[i - 1][f] == pos) m = f;
                            // a position twice in one item keeps its first entry there
                            const unsigned same = __match_any_sync(0xffffffffu, m < 0 ? ~lane : m);
                            const bool forced = m >= 0 && (same & ((1u << lane) - 1u)) == 0;
                            const unsigned taken = __reduce_or_sync(0xffffffffu, forced ? 1u << m : 0u);
                            const unsigned rest = __ballot_sync(0xffffffffu, !forced);
                            slot = forced ? m : (int)__fns(~taken, 0, __popc(rest & ((1u << lane) - 1u)) + 1);
                            slot_s[i][lane] = -1;
                            if (lane == 0) shared_s[i] = taken;
                            __syncwarp();
                            if (lane < n) slot_s[i][slot] = pos;
                        }
                        __syncthreads();
                    }
                }
                unsigned char* q = out + (size_t)npk * strip_packet_bytes(sizeof(VT), b.scatter);
                const int kidx = b.scatter ? 80 : 16;
                if (lane == 0) reinterpret_cast<int*>(q)[warp] = base;
                if (b.scatter) {
                    // runs of shared slots: entry of slot j of this item
                    const unsigned n1 = warp < 3 ? shared_s[warp + 1] : 0u;
                    const unsigned n2 = warp < 2 ? n1 & shared_s[warp + 2] : 0u;
                    const unsigned n3 = warp < 1 ? n2 & shared_s[3] : 0u;
                    const bool chains = ((shared_s[1] & shared_s[2]) | (shared_s[2] & shared_s[3])) != 0;
                    if (lane == 0 && chains) reinterpret_cast<int*>(q)[warp] = base | INT_MIN;
                    if (lane < 8) {
                        unsigned f = 0;
                        for (int s = 0; s < 4; ++s) {
                            const int j = 8 * s + lane;
                            const bool skip = slot_s[warp][j] < 0 || ((shared_s[warp] >> j) & 1u);
                            f |= (skip ? 1u : 0u) << s | ((n1 >> j) & 1u) << (4 + s) | ((n2 >> j) & 1u) << (8 + s) |
                                 ((n3 >> j) & 1u) << (12 + s);
                        }
                        reinterpret_cast<unsigned short*>(q + 16)[warp * 8 + lane] = (unsigned short)f;
                    }
                }
                const int L = warp * 8 + (slot & 7), s = slot >> 3;
                reinterpret_cast<unsigned short*>(q + kidx)[L * 4 + s] =
                    lane < n ? (unsigned short)(pos - base) : (unsigned short)kPad;
                reinterpret_cast<VT*>(q + kidx + 256)[L * 4 + s] = lane < n ? val[src] : VT(0.f);
            }
            p += n;
            ++npk;
        }
        if (!FILL && threadIdx.x == 0) {
            int mask = 0;
            for (int r = 0; r < st.y; ++r)
                if (b.all_items || len_s[r] > 0) mask |= 1 << r;
            b.meta[t] = make_int4(0, npk | (tall ? kStripTall : 0), st.z, mask);
        }
        __syncthreads();
    }
}

using StripFn = void (*)(StripArgs);

template <typename VT, int KIND, bool COPIES = false>
StripFn pick_nw(int nw) {
    switch (nw) {
        case 1: return k_strip<VT, 1, KIND, COPIES>;
        case 2: return k_strip<VT, 2, KIND, COPIES>;
        case 4: return k_strip<VT, 4, KIND, COPIES>;
        default: return k_strip<VT, 8, KIND, COPIES>;
    }
}

template <typename VT>
StripFn pick_kind(int kind, int nw, bool copies) {
    if (kind == 0) return pick_nw<VT, 0>(nw);
    if (kind == 2) return pick_nw<VT, 2>(nw);
    return copies ? pick_nw<VT, 1, true>(nw) : pick_nw<VT, 1>(nw);
}

StripFn strip_fn(suppy_dtype dt, int kind, int nw, bool copies) {
    if (dt == SUPPY_F32) return pick_kind<float>(kind, nw, copies);
    if (dt == SUPPY_BF16) return pick_kind<__nv_bfloat16>(kind, nw, copies);
    return pick_kind<__half>(kind, nw, copies);
}

template <typename VT>
cudaError_t build(const StripBuild& b, int fill, int grid, cudaStream_t s) {
    const size_t smem = (size_t)b.max_len * 4 * (2 * sizeof(unsigned) + sizeof(unsigned short));
    auto f = fill ? k_strip_build<VT, 1> : k_strip_build<VT, 0>;
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    f<<<grid, 128, smem, s>>>(b);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_strip(const StripArgs& a, suppy_dtype dt, int kind, int nw, int grid, cudaStream_t s) {
    StripFn f = strip_fn(dt, kind, nw, a.copy > 0);
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, a.ring);
    if (e != cudaSuccess) return e;
    return launch_dependent(f, grid, kStripThreads, a.ring, s, a);
}

cudaError_t launch_strip_build(const StripBuild& b, suppy_dtype dt, int fill, cudaStream_t s) {
    if (b.nstrips < 1) return cudaSuccess;
    if (b.max_len < 1 || b.max_len > kStripMaxItem) return cudaErrorInvalidValue;
    const int grid = std::min(b.nstrips, 152 * 64);
    if (dt == SUPPY_F32) return build<float>(b, fill, grid, s);
    if (dt == SUPPY_BF16) return build<__nv_bfloat16>(b, fill, grid, s);
    return build<__half>(b, fill, grid, s);
}

}  // namespace suppy
