// Batched engine: many independent simulations (mesh handles) advanced by one
// persistent kernel, touching only tets that hold molecules.
//
// Realisations run in parallel are the embarrassingly parallel use of the
// method (Sec. I of arXiv:1512.03126).  Each thread-block cluster takes one
// simulation from a work queue (largest first) and runs its periods of
// Algorithm 1 itself, with cluster.sync() as the period barrier, so that no
// grid-wide synchronisation and no spin-wait is needed.  Per period the
// cluster visits the tets whose bit is set in that period's activity bitmap
// (tets that hold molecules or have a zero-order reaction on), runs the same
// per-tet work as the dense kernels (warp_step), and adds the
// molecules that stay or leave into the next count buffer with integer atomic
// adds — exact and independent of order, so the counts equal those of the
// dense gather.  A tet that keeps or receives molecules sets its bit in the
// next period's bitmap.  One simulation's active region is touched by one
// cluster only, which keeps it in those SMs' L1 and in L2.
//
// The random streams of a simulation are keyed by its own seed, period index
// and canonical tet ids, so its counts do not depend on what runs beside it.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <numeric>
#include <queue>
#include <type_traits>
#include <vector>

#include "rd_api_internal.h"
#include "rd_device.cuh"
#include "rd_internal.h"
#include "rd_period.cuh"
#include "rd_warp.cuh"

using namespace rdk;

namespace {

constexpr int kRunBlock = 512;

struct SlotDesc {
    DevMesh m;
    const uint4* thr;        // thresholds for tau
    const uint4* thr_last;   // thresholds for the shortened last period
    int32_t* N[2];           // count buffers [S][T]; the slice starts in N[0]
    uint32_t* bits[2];       // active-tet bitmaps, by period parity in the slice
    int32_t wshift;          // of 2^wshift words, at least as many as the cluster has warps
    int32_t sm;              // counts and bitmaps in the cluster's shared memory
    const uint4* packed;     // one species: {src, thr} per tet
    int32_t* N2;             // one species: counts of both parities interleaved
    uint64_t seed;
    uint32_t period0;        // global period index of local period 0
    int32_t P;               // periods to run in total
    int32_t q0, q1;          // this slice runs local periods q0 .. q1-1
    int32_t last_short;      // local period P-1 is shortened
    int32_t S;
    uint32_t zero_order;     // reactions of order 0 with k > 0
    double tau, tau_last;
    float tauf, tau_lastf;
};

// Fire-and-forget integer add to global memory (no value comes back, so the
// warp does not wait for the L2 round trip).
__device__ __forceinline__ void red_add(int32_t* p, int32_t v) {
    asm volatile("red.relaxed.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v));
}

// Device clock in nanoseconds (the global timer shared by all SMs).
__device__ __forceinline__ unsigned long long globaltimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Fire-and-forget OR into a global bitmap word.
__device__ __forceinline__ void red_or(uint32_t* p, uint32_t v) {
    asm volatile("red.relaxed.gpu.global.or.b32 [%0], %1;" ::"l"(p), "r"(v));
}

// The same into a word of a CTA of the cluster (shared::cluster address).
__device__ __forceinline__ uint32_t cta_address(uint32_t addr, uint32_t cta) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(cta));
    return r;
}
__device__ __forceinline__ void red_add_cluster(uint32_t addr, int32_t v) {
    asm volatile("red.relaxed.cluster.shared::cluster.add.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void red_or_cluster(uint32_t addr, uint32_t v) {
    asm volatile("red.relaxed.cluster.shared::cluster.or.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

constexpr int kWarps = kRunBlock / 32;
constexpr int kGroup = 8;                   // bitmap columns (32 words each) a warp loads at once
constexpr int kSmCols = 2;                  // of a simulation in shared memory: all of them
// A warp's list of tets to visit (a simulation in global memory): up to 31 left
// over, and what is appended at once.  The lists are where a simulation in
// shared memory has its counts.
constexpr int kListMost = 256;
constexpr size_t kListBytes = (size_t)kWarps * (32 + kListMost) * sizeof(int32_t);

// Dynamic shared memory of a warp, in words: the step's (rd_warp.cuh) and the
// bitmap words of its current batch.
__host__ __device__ inline int engine_warp_words(int S, bool react) { return warp_words(S, react) + 32 * kGroup; }

// A simulation of one species in the cluster's shared memory (kSm): a CTA
// keeps the words of its warps, wpc = W / kC of them, in both parities' bitmaps
// and a pair of counts (both parities) for each tet of these words, row by row
// (row i: the tets of bit i).  Bytes of one CTA:
__host__ __device__ inline size_t sm_bytes(int64_t T, int wshift, int kC) {
    const int64_t W = (int64_t)1 << wshift, wpc = W / kC, rows = (T + W - 1) / W;
    return (size_t)(rows * wpc * 8 + wpc * 8);
}

// Position of set bit number k (from 0) of w, by halves.
__device__ __forceinline__ int nth_set_bit(uint32_t w, int k) {
    int p = 0;
#pragma unroll
    for (int h = 16; h > 0; h >>= 1) {
        const int c = __popc(w & ((1u << h) - 1u));
        if (k >= c) {
            k -= c;
            p += h;
            w >>= h;
        }
    }
    return p;
}

// A simulation in the cluster's shared memory: tet t is bit t >> ws of word
// t mod 2^ws (one in global memory: bit t & 31 of word t >> 5).
__device__ __forceinline__ int tet_in_shared(int word, int bit, int ws) { return (bit << ws) | word; }

// Shared memory of the engine kernel.
__shared__ int32_t s_item;                          // work-item index (first CTA of the cluster)
__shared__ unsigned long long s_mass[3];            // [0] molecules of the simulation (all species) at the
                                                    // start of the period; [1], [2] net change by reactions
                                                    // in periods of even / odd parity (two's complement)
__shared__ SlotDesc s_desc;                         // the simulation's descriptor and chemistry
__shared__ ModelParams s_mp;
static_assert(sizeof(SlotDesc) + sizeof(ModelParams) + 64 <= 48u * 1024u - kDefaultShared, "static shared memory");
extern __shared__ __align__(16) int32_t s_warp[];   // [kWarps][engine_warp_words]; kSm: then bitmaps and counts

// Counts and bitmaps of one period and the next, in global memory: N[r] /
// N[r^1], or the two halves of the interleaved pairs.
template <bool kOne>
struct GlobalView {
    int32_t* cur;
    int32_t* next;
    uint32_t* bcur;
    uint32_t* bnext;
    int64_t T;
    static constexpr int stride = kOne ? 2 : 1;
    __device__ __forceinline__ GlobalView(const SlotDesc& d, int r)
        : bcur(d.bits[r]), bnext(d.bits[r ^ 1]), T(d.m.T) {
        cur = kOne ? d.N2 + r : d.N[r];
        next = kOne ? d.N2 + (r ^ 1) : d.N[r ^ 1];
    }
    __device__ __forceinline__ int32_t load(int s, int t) const { return __ldcg(cur + (s * T + t) * stride); }
    __device__ __forceinline__ void clear(int s, int t) const { cur[(s * T + t) * stride] = 0; }
    __device__ __forceinline__ void add(int s, int t, int32_t n) const { red_add(next + (s * T + t) * stride, n); }
    __device__ __forceinline__ void mark(int t) const { red_or(bnext + (t >> 5), 1u << (t & 31)); }
    __device__ __forceinline__ void send(int t, int32_t n, bool more) const {
        add(0, t, n);
        if (more) mark(t);
    }
    __device__ __forceinline__ void unvisit(int t) const { red_or(bcur + (t >> 5), 1u << (t & 31)); }
    // the tet's own CTA
    __device__ __forceinline__ void keep(int s, int t, int32_t n) const { add(s, t, n); }
    __device__ __forceinline__ void mark_own(int t) const { mark(t); }
};

// The same in the cluster's shared memory: load, clear, keep and mark_own are
// of tets of the calling CTA.
template <int kC>
struct ClusterView {
    int32_t* cnt;           // [rows][wpc][2] of this CTA
    uint32_t* bcur;
    uint32_t* bnext;
    uint32_t next_at, bnext_at;   // shared addresses of the next period's counts and bits
    int ws, wl, r;
    static constexpr int kShift = kC == 1 ? 0 : (kC == 2 ? 1 : (kC == 4 ? 2 : 3));
    __device__ __forceinline__ ClusterView(const SlotDesc& d, int r_, int32_t* data) : ws(d.wshift), wl(d.wshift - kShift), r(r_) {
        const int wpc = 1 << wl;
        uint32_t* bits = reinterpret_cast<uint32_t*>(data);
        bcur = bits + r * wpc;
        bnext = bits + (r ^ 1) * wpc;
        cnt = data + 2 * wpc;
        next_at = (uint32_t)__cvta_generic_to_shared(cnt + (r ^ 1));
        bnext_at = (uint32_t)__cvta_generic_to_shared(bnext);
    }
    __device__ __forceinline__ int slot(int t) const { return ((t >> ws) << wl) | (t & ((1 << wl) - 1)); }
    __device__ __forceinline__ int32_t load(int, int t) const { return cnt[2 * slot(t) + r]; }
    __device__ __forceinline__ void clear(int, int t) const { cnt[2 * slot(t) + r] = 0; }
    // one species: a leaver's add and bit together
    __device__ __forceinline__ void send(int t, int32_t n, bool more) const {
        const uint32_t word = (uint32_t)t & ((1u << ws) - 1u), loc = word & ((1u << wl) - 1u);
        const uint32_t row = (uint32_t)t >> ws;
        const uint32_t there = cta_address(bnext_at, word >> wl);
        red_add_cluster(there + (next_at - bnext_at) + 8u * ((row << wl) | loc), n);
        if (more) red_or_cluster(there + 4u * loc, 1u << row);
    }
    __device__ __forceinline__ void keep(int, int t, int32_t n) const { atomicAdd(cnt + 2 * slot(t) + (r ^ 1), n); }
    __device__ __forceinline__ void mark_own(int t) const { atomicOr(bnext + (t & ((1 << wl) - 1)), 1u << (t >> ws)); }
    __device__ __forceinline__ void unvisit(int t) const { atomicOr(bcur + (t & ((1 << wl) - 1)), 1u << (t >> ws)); }
};

// Leavers of a tet into the next period's counts (fire-and-forget integer
// adds).  An add that takes a count past 2^31-1 wraps it negative; as the
// simulation's molecule total is kept below 2^32 (checked every period), the
// next read of the count, or the check at the end of the slice, sees it
// negative and reports the overflow, exactly when the dense gather would.
template <class View, bool kOne>
struct Scatter {
    const View& c;
    bool more;            // a further period follows in this slice
    const int4* src;
    int t;
    int4 sr;
    bool have;
    uint32_t send;        // faces through which something leaves (several species)
    uint32_t bad;
    long long sent;       // molecules that leave

    __device__ __forceinline__ Scatter(const View& c_, bool more_, const int4* src_, int t_, int4 sr_, bool have_)
        : c(c_), more(more_), src(src_), t(t_), sr(sr_), have(have_), send(0), bad(0), sent(0) {}

    __device__ __forceinline__ void operator()(int sp, const int4& o) {
        if (!have) sr = __ldg(src + t);
        have = true;
        const int nbr[4] = {sr.x, sr.y, sr.z, sr.w}, n[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            if (n[f] <= 0) continue;
            if (nbr[f] < 0) { bad |= kErrNegative; continue; }
            if constexpr (kOne) {
                c.send(nbr[f] >> 2, n[f], more);
            } else {
                c.add(sp, nbr[f] >> 2, n[f]);
                send |= 1u << f;
            }
        }
        sent += (long long)o.x + o.y + o.z + o.w;
    }
};

// One round: the tets t of the live lanes through the step, what stays and what
// leaves into the next counts and bits.  Without kCalls a lane whose tet needs
// the double-precision samplers is left undone (its counts too) and *deferred
// set.
template <bool kOne, bool kReact, bool kCalls, class View>
__device__ __forceinline__ uint32_t engine_round(const SlotDesc& d, const ModelParams& mp, int S, const WarpMem& w,
                                                 const PeriodView& v, const View& c, bool more, int t, bool live,
                                                 uint32_t* err, unsigned long long* mass_delta, bool* deferred) {
    const int lane = threadIdx.x & 31;
    int4 sr = make_int4(-1, -1, -1, -1);
    uint4 pre = make_uint4(0u, 0u, 0u, 0u);
    long long held = 0;
    uint32_t bad = 0;
    Presence pr;
    const uint32_t mask = kReact && mp.has_mask && live ? __ldg(d.m.mask + t) : 0xffffffffu;
    if (kOne && live) {
        // the record and the count, loaded together
        sr = __ldg(reinterpret_cast<const int4*>(d.packed + 2 * (int64_t)t));
        pre = __ldg(v.thr + (int64_t)t * v.thr_stride);
    }
    if constexpr (kOne && !kReact && !kCalls) {
        // At most eight molecules in each tet: two Philox blocks of its own draw
        // them, and everything stays in registers (most rounds of a mesh with
        // more tets than molecules).  With this and one sum a batch a round takes
        // 584 instructions in all, 711 with warp_step and a sum a column: 64 cubes of
        // 20 to 40 cells, 100 periods from the 2,500th on, 2.42 -> 1.90 ms (2.22
        // before the warp step); the 512-cube ensemble 1.86 -> 1.43 s.
        const int32_t n = live ? c.load(0, t) : 0;
        if (!__any_sync(kAllLanes, n < 0 || n > 8)) {
            if (n == 0) return 0u;
            const uint32_t key = (uint32_t)key_of(d.m, t), k0 = (uint32_t)v.seed, k1 = (uint32_t)(v.seed >> 32);
            uint32_t a0 = 0, a1 = 0;
            for (int b = 0; 4 * b < n; ++b)
                count_block(rdd::philox_block((uint32_t)b, key, v.period, rdd::kPurposeDiffusion << 16, k0, k1),
                            min(4, n - 4 * b), pre, a0, a1);
            c.clear(0, t);
            const int nbr[4] = {sr.x, sr.y, sr.z, sr.w};
            const int o[4] = {(int)(a0 & 0xffffu), (int)(a0 >> 16), (int)(a1 & 0xffffu), (int)(a1 >> 16)};
#pragma unroll
            for (int f = 0; f < 4; ++f) {
                if (o[f] == 0) continue;
                if (nbr[f] < 0) bad |= kErrNegative;
                else c.send(nbr[f] >> 2, o[f], more);
            }
            const int32_t stay = n - (o[0] + o[1] + o[2] + o[3]);
            if (stay > 0) {
                c.keep(0, t, stay);
                if (more) c.mark_own(t);
            }
            return bad;
        }
    }
    if (live) {
        for (int s0 = 0; s0 < S; s0 += 4) {
            int32_t n[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (s0 + k < S) n[k] = c.load(s0 + k, t);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (s0 + k >= S) continue;
                if (n[k] < 0) {          // wrapped past 2^31-1 by the previous period's adds
                    bad |= kErrOverflow;
                    c.clear(s0 + k, t);
                    n[k] = 0;
                }
                w.N[32 * (s0 + k) + lane] = n[k];
                pr.add(s0 + k, n[k]);
                if (kReact) held += n[k];
            }
        }
    }
    const uint32_t had = pr.any;
    Scatter<View, kOne> scatter(c, more, d.m.src, t, sr, kOne);
    uint32_t dirty = 0;
    bad |= warp_step<kOne, kReact, false, kCalls, kOne>(d.m, mp, S, w, v, t, live, mask, pr, &dirty, deferred, err,
                                                        scatter, pre);
    bad |= scatter.bad;
    long long delta = 0;
    if (live && (kCalls || !*deferred)) {
        bool keep = pr.any != 0u;
        if (kReact && d.zero_order) keep = keep || (mask & d.zero_order) != 0u;
        if (kOne) {
            if (had) c.clear(0, t);
            if (pr.any) {
                const int32_t n = w.N[lane];
                c.keep(0, t, n);
                if (kReact) delta += n;
            }
        } else {
            for (uint32_t bits = had; bits; bits &= bits - 1u) c.clear(__ffs(bits) - 1, t);
            for (uint32_t bits = pr.any; bits; bits &= bits - 1u) {
                const int s = __ffs(bits) - 1;
                const int32_t n = w.N[32 * s + lane];
                c.keep(s, t, n);
                if (kReact) delta += n;
            }
        }
        if (kReact) delta += scatter.sent - held;
        if (more) {
            if (keep) c.mark_own(t);
            if constexpr (!kOne) {
                const int nbr[4] = {scatter.sr.x, scatter.sr.y, scatter.sr.z, scatter.sr.w};
#pragma unroll
                for (int f = 0; f < 4; ++f)
                    if ((scatter.send >> f) & 1u) c.mark(nbr[f] >> 2);
            }
        }
    }
    // net molecules made by reactions: all that stays and leaves minus what was
    // held
    if (kReact && delta != 0) atomicAdd(mass_delta, (unsigned long long)delta);
    return bad;
}

// What a period's passes of one warp share.
template <bool kOne, bool kReact, int kC, bool kSm>
struct WarpPeriod {
    using View = typename std::conditional<kSm, ClusterView<kC>, GlobalView<kOne>>::type;
    static constexpr int kW = kC * kWarps;
    static constexpr int kWShift = kC == 1 ? 4 : (kC == 2 ? 5 : (kC == 4 ? 6 : 7));
    static_assert((1 << kWShift) == kW, "warps of a cluster");
    int S, per;                // this warp's words: `per` of them
    int word0, used;           // global: the words that hold tets
    // Word number k of the warp.  Global bitmaps: runs of 4 words (128 tets, 16
    // bytes) dealt round-robin, so that a load takes 8 sectors instead of 32
    // (192 cubes of up to 384,000 tets, 0.1 s: 1.37 -> 0.83 s).
    __device__ __forceinline__ int word(int k) const {
        if (kSm) return word0 + k;
        return per >= 4 ? ((((k >> 2) << kWShift) + word0) << 2) | (k & 3) : (k << kWShift) + word0;
    }
    __device__ __forceinline__ bool has(int k) const { return k < per && (kSm || word(k) < used); }
    __device__ __forceinline__ uint32_t* at(int k) const { return kSm ? words + k : words + word(k); }
    WarpMem w;
    PeriodView v;
    View c;
    uint32_t* words;           // this warp's words of the period's bitmap
    uint32_t* wb;              // the current batch's
    int32_t* list;             // global bitmaps: tets to visit
    bool more;

    static __device__ __forceinline__ View view(const SlotDesc& d, int r, int S) {
        if constexpr (kSm) return View(d, r, s_warp + kWarps * engine_warp_words(S, kReact));
        else return View(d, r);
    }
    static __device__ __forceinline__ PeriodView period_view(const SlotDesc& d, int q) {
        const bool last = (q == d.P - 1) && d.last_short;
        // thresholds: packed beside the reverse-face record (stride 2) except in
        // a shortened last period
        return PeriodView{d.period0 + (uint32_t)q, last ? d.tau_last : d.tau, last ? d.tau_lastf : d.tauf, d.seed,
                          last ? d.thr_last : (kOne ? d.packed + 1 : d.thr), kOne && !last ? 2 : 1};
    }
    __device__ __forceinline__ WarpPeriod(const SlotDesc& d, int q)
        : S(kOne ? 1 : d.S), per((1 << d.wshift) >> kWShift),
          w(s_warp + (threadIdx.x >> 5) * engine_warp_words(S, kReact), S, kReact, s_mp.rx), v(period_view(d, q)),
          c(view(d, (q - d.q0) & 1, S)), more(q + 1 < d.q1) {
        const int warp = threadIdx.x >> 5;
        const int rank = kC > 1 ? (int)cooperative_groups::this_cluster().block_rank() : 0;
        word0 = (rank * kWarps + warp) * (kSm ? per : 1);
        used = (d.m.T + 31) >> 5;
        words = c.bcur + (kSm ? warp * per : 0);
        wb = reinterpret_cast<uint32_t*>(s_warp + warp * engine_warp_words(S, kReact) + warp_words(S, kReact));
        list = s_warp + kWarps * engine_warp_words(S, kReact) + warp * (32 + kListMost);
    }
};

// The warp's words of a batch: up to kGroup columns (32 words, one per lane)
// loaded at once and cleared for their next use.  Returns the lane's set bits.
template <bool kSm, class Period>
__device__ __forceinline__ int load_batch(const Period& p, int w0) {
    const int lane = threadIdx.x & 31;
    constexpr int kCols = kSm ? kSmCols : kGroup;
    uint32_t wds[kCols];
    int own = 0;
#pragma unroll
    for (int kk = 0; kk < kCols; ++kk) {
        const int i = w0 + kk * 32 + lane;
        wds[kk] = p.has(i) ? (kSm ? *p.at(i) : __ldcg(p.at(i))) : 0u;
    }
#pragma unroll
    for (int kk = 0; kk < kCols; ++kk) {
        if (wds[kk]) *p.at(w0 + kk * 32 + lane) = 0u;
        p.wb[kk * 32 + lane] = wds[kk];
        own += __popc(wds[kk]);
    }
    return own;
}

__device__ __forceinline__ int sum_to_lane(int x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int dd = 1; dd < 32; dd <<= 1) {
        const int y = __shfl_up_sync(kAllLanes, x, dd);
        if (lane >= dd) x += y;
    }
    return x;
}

// The tets of the set bits of the warp's words, in rounds of 32: visit(t, live)
// once a round.  Words are cleared when they are loaded.  Returns the number of
// set bits.
//
// In shared memory a simulation has two columns a warp at most: one prefix sum
// over the lanes' set bits lets each lane find a tet of its own (a search over
// the sums, the column, the bit in the word: a fixed 110 instructions a round).
//
// In global memory the lanes append their set bits to a list, and every 32 of
// them make a round, so that only a period's last one is not full.  One prefix
// sum serves a whole batch, and a lane goes through its words at its own pace.
template <bool kSm, class Period, class Visit>
__device__ __forceinline__ uint32_t visit_set_bits(const SlotDesc& d, const Period& p, Visit visit) {
    const int lane = threadIdx.x & 31;
    uint32_t done = 0;
    if constexpr (kSm) {
        for (int w0 = 0; w0 < p.per; w0 += 32 * kSmCols) {
            const int own = load_batch<true>(p, w0);
            const int inc = sum_to_lane(own);
            const int total = __shfl_sync(kAllLanes, inc, 31);
            done += (uint32_t)total;
            __syncwarp();
            for (int e0 = 0; e0 < total; e0 += 32) {
                // the lane's tet: the batch's set bit number e0 + lane
                const int e = e0 + lane;
                const bool live = e < total;
                int from = 0;
#pragma unroll
                for (int step = 16; step > 0; step >>= 1)
                    if (__shfl_sync(kAllLanes, inc, from + step - 1) <= e) from += step;
                int k = e - __shfl_sync(kAllLanes, inc - own, from);
                uint32_t word = p.wb[from];
                int col = 0;
#pragma unroll
                for (int kk = 1; kk < kSmCols; ++kk) {
                    const int c = __popc(word);
                    if (col == kk - 1 && k >= c) {
                        k -= c;
                        col = kk;
                        word = p.wb[kk * 32 + from];
                    }
                }
                const int i = w0 + col * 32 + from;
                visit(live ? tet_in_shared(p.word(i), nth_set_bit(word, k), d.wshift) : 0, live);
                __syncwarp();
            }
        }
    } else {
        int32_t* const list = p.list;
        int cnt = 0, own = 0, col = 0, w0 = -32 * kGroup, base = 0;
        uint32_t word = 0u;   // of the lane: bits left in the batch (own), in its current word
        for (;;) {
            while (cnt < 32) {
                if (!__any_sync(kAllLanes, own > 0)) {
                    w0 += 32 * kGroup;
                    if (w0 >= p.per) break;
                    own = load_batch<false>(p, w0);
                    word = 0u;
                    col = 0;
                    __syncwarp();
                    continue;
                }
                int n = own;
                int inc = sum_to_lane(n);
                int total = __shfl_sync(kAllLanes, inc, 31);
                if (total > kListMost) {   // as much as the list holds: eight bits of each lane
                    n = min(n, kListMost / 32);
                    inc = sum_to_lane(n);
                    total = __shfl_sync(kAllLanes, inc, 31);
                }
                own -= n;
                for (int at = cnt + inc - n; n > 0; --n) {
                    while (word == 0u) {
                        word = p.wb[col * 32 + lane];
                        base = p.word(w0 + col * 32 + lane) << 5;
                        ++col;
                    }
                    list[at++] = base + __ffs(word) - 1;
                    word &= word - 1u;
                }
                cnt += total;
                done += (uint32_t)total;
                __syncwarp();
            }
            if (cnt == 0) break;
            const int take = min(cnt, 32);
            cnt -= take;
            const bool live = lane < take;
            const int t = live ? list[cnt + lane] : 0;
            __syncwarp();
            visit(t, live);
            __syncwarp();
        }
    }
    return done;
}

// The warp's tets whose bits the rounds set back, with the double-precision
// samplers, 32 of them side by side (with a round for each bit of the lanes'
// own words, 24,576 tets of 5,000 molecules on 8 CTAs kept 6 lanes of 32 busy:
// 48 ms where this takes 17).
template <bool kOne, bool kReact, int kC, bool kSm>
__device__ __noinline__ uint32_t run_deferred(int q, uint32_t* err, unsigned long long* mass_delta) {
    const SlotDesc& d = s_desc;
    const WarpPeriod<kOne, kReact, kC, kSm> p(d, q);
    uint32_t bad = 0;
    visit_set_bits<kSm>(d, p, [&](int t, bool live) {
        bool none = false;
        bad |= engine_round<kOne, kReact, true>(d, s_mp, p.S, p.w, p.v, p.c, p.more, t, live, err, mass_delta, &none);
    });
    return bad;
}

// One period of a simulation for one warp: its tets in rounds of 32
// (engine_round).  In shared memory a bitmap word holds 32 tets a power of two
// apart, so that every word has its share of a compact cloud of molecules and of
// its crowded tets, and the words go to the cluster's kW warps in equal
// contiguous parts; in global memory a word holds 32 consecutive tets and
// words are dealt in runs of four (WarpPeriod::word).
//
// Out of line and free of calls, like run_deferred beside it: with the round
// in the kernel's own loop, what it keeps across the call of run_deferred
// (addresses and descriptor fields lifted out of the loops) sat in local
// memory, 110 loads a round.
struct PeriodResult {
    uint32_t bad, done, late;   // error bits, tets visited, whether some were deferred
};
template <bool kOne, bool kReact, int kC, bool kSm>
__device__ __noinline__ PeriodResult run_period(int q, uint32_t* err, unsigned long long* mass_delta) {
    const SlotDesc& d = s_desc;
    const WarpPeriod<kOne, kReact, kC, kSm> p(d, q);
    uint32_t bad = 0;
    bool late = false;              // some tet was deferred
    const uint32_t done = visit_set_bits<kSm>(d, p, [&](int t, bool live) {
        bool deferred = false;
        bad |= engine_round<kOne, kReact, false>(d, s_mp, p.S, p.w, p.v, p.c, p.more, t, live, err, mass_delta,
                                                 &deferred);
        if (__ballot_sync(kAllLanes, deferred)) {
            // back into the bitmap, for the pass after these rounds
            late = true;
            if (deferred) {
                p.c.unvisit(t);
            }
        }
    });
    if (late && !kSm) __threadfence();   // the bits set back are read by other lanes
    __syncwarp();
    return PeriodResult{bad, done, late ? 1u : 0u};
}

// One simulation per cluster of kC CTAs (kC = 1: per CTA).  The cluster's
// first CTA owns the work-item index; the others read it through distributed
// shared memory.  cluster.sync() (a hardware barrier) separates periods.
//
// The tets to visit in a period are the set bits of that period's bitmap
// (global memory, one bit per tet, one bitmap per period parity).  Each
// visited word is cleared for its next use; a tet that keeps or receives
// molecules sets its bit in the other parity's bitmap (an OR, which is
// idempotent, so no membership test and no list are needed).  At the end of
// a slice both bitmaps are zero.
//
// Count adds are fire-and-forget reductions.  A count that an add takes past
// 2^31-1 wraps negative and is reported when read (next period, or the check
// at the end of the slice); the molecule total of the simulation, tracked per
// period (each round adds what its reactions make or consume), is kept
// below 2^32 - 1 so that no count can wrap all the way round unseen.
// Where a simulation's descriptor says so (one species, a mesh whose counts
// fit, see sm_bytes) the counts and
// bitmaps are in the cluster's shared memory for the slice, and every add and
// OR goes to the owning CTA's.  In global memory a period of a 24^3-cell cube
// on 8 CTAs took 18,700 cycles of which a warp worked 8,500 (2,000 to load its
// words, 900 for the counts); the rest was the barrier's wait for the adds to
// reach L2.
template <int S_, bool kReact, int kC>
__global__ void __launch_bounds__(kRunBlock, 1)
k_engine_run(const SlotDesc* __restrict__ descs, const ModelParams* __restrict__ mps, const int32_t* __restrict__ order,
             int32_t n_items, int32_t* head, uint32_t* err, unsigned long long* processed,
             unsigned long long* times) {
    namespace cg = cooperative_groups;
    constexpr bool kOne = S_ == 1;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = kC > 1 ? (int)cluster.block_rank() : 0;
    int32_t* item = kC > 1 ? cluster.map_shared_rank(&s_item, 0) : &s_item;
    unsigned long long* mass = kC > 1 ? cluster.map_shared_rank(&s_mass[0], 0) : &s_mass[0];
    auto csync = [&]() {
        if (kC > 1) cluster.sync();
        else __syncthreads();
    };
    const int lane = threadIdx.x & 31;
    unsigned long long done = 0;
    for (;;) {
        csync();
        if (rank == 0 && threadIdx.x == 0) {
            *item = atomicAdd(head, 1);
            mass[0] = mass[1] = mass[2] = 0ull;
        }
        csync();
        const int32_t k = *item;
        // every CTA has read the item before the leader may overwrite it or
        // any CTA leaves (a CTA's shared memory must outlive remote reads)
        csync();
        if (k >= n_items) break;
        const int slot = order[k];
        if (times && rank == 0 && threadIdx.x == 0) {
            times[4 * slot] = globaltimer_ns();
            times[4 * slot + 2] = 0ull;
        }
        unsigned long long item_done = 0;
        {
            const uint32_t* from = reinterpret_cast<const uint32_t*>(descs + slot);
            for (int i = threadIdx.x; i < (int)(sizeof(SlotDesc) / 4); i += kRunBlock)
                reinterpret_cast<uint32_t*>(&s_desc)[i] = from[i];
            from = reinterpret_cast<const uint32_t*>(mps + slot);
            for (int i = threadIdx.x; i < (int)(sizeof(ModelParams) / 4); i += kRunBlock)
                reinterpret_cast<uint32_t*>(&s_mp)[i] = from[i];
        }
        __syncthreads();
        const SlotDesc& d = s_desc;
        const int T = d.m.T;
        const int S = kOne ? 1 : d.S;
        const int W = 1 << d.wshift;
        constexpr bool inter = kOne;   // interleaved counts
        const bool sm = kOne && d.sm != 0;
        uint32_t bad = 0;
        // initial bitmap: occupied tets and tets with a zero-order reaction on;
        // and the simulation's molecule total.  A lane a tet: in shared memory
        // word by word of this CTA, 32 tets W apart (a row of the counts at a
        // time), in global memory 32 consecutive tets a warp.
        unsigned long long mine = 0;
        const int wpc = W / kC;   // in shared memory: the words, and the tets, of this CTA
        int32_t* const data = s_warp + kWarps * engine_warp_words(S, kReact);
        auto look = [&](int t) {
            bool occ = false;
            if (kReact && d.zero_order) occ = ((s_mp.has_mask ? d.m.mask[t] : 0xffffffffu) & d.zero_order) != 0u;
            for (int s = 0; s < S; ++s) {
                const int32_t c = d.N[0][(int64_t)s * T + t];
                occ = occ || c > 0;
                mine += (uint32_t)max(c, 0);
                if (c < 0) bad |= kErrNegative;
                if (sm) reinterpret_cast<int2*>(data + 2 * wpc)[(t >> d.wshift) * wpc + (t & (wpc - 1))] = make_int2(c, 0);
                else if (inter) reinterpret_cast<int2*>(d.N2)[t] = make_int2(c, 0);
            }
            return occ;
        };
        if (sm) {
            for (int i = threadIdx.x; i < wpc; i += kRunBlock) {
                uint32_t word = 0;
                for (int bit = 0; bit < 32; ++bit) {
                    const int t = tet_in_shared(rank * wpc + i, bit, d.wshift);
                    if (t < T && look(t)) word |= 1u << bit;
                }
                reinterpret_cast<uint32_t*>(data)[i] = word;
                reinterpret_cast<uint32_t*>(data)[wpc + i] = 0u;
            }
        } else {
            for (int base = rank * kRunBlock; base < T; base += kC * kRunBlock) {
                const int t = base + threadIdx.x;
                const uint32_t word = __ballot_sync(kAllLanes, t < T && look(t));
                if (lane == 0 && t < T) d.bits[0][t >> 5] = word;
            }
        }
#pragma unroll
        for (int dd = 16; dd > 0; dd >>= 1) mine += __shfl_xor_sync(kAllLanes, mine, dd);
        if (lane == 0 && mine) atomicAdd(&mass[0], mine);
        // The molecule total after a period, kept below 2^32 - 1: then no
        // int32 count can wrap past 2^32 unseen (see Scatter).  Reactions
        // change it; each round adds their net change.
        auto account = [&](int q) {
            if (rank == 0 && threadIdx.x == 0) {
                unsigned long long* dq = &mass[1 + (q & 1)];
                mass[0] += *dq;
                *dq = 0ull;
                if ((long long)mass[0] >= 4294967295ll) atomicOr(err, kErrOverflow);
            }
        };
        for (int q = d.q0; q < d.q1; ++q) {
            csync();   // the previous period's adds and bits are complete
            if (q > d.q0) account(q - 1);
            unsigned long long* made = &mass[1 + (q & 1)];
            PeriodResult r;
            if (sm) {
                if constexpr (kOne) {
                    r = run_period<true, kReact, kC, true>(q, err, made);
                    if (r.late) bad |= run_deferred<true, kReact, kC, true>(q, err, made);
                }
            } else {
                r = run_period<kOne, kReact, kC, false>(q, err, made);
                if (r.late) bad |= run_deferred<kOne, kReact, kC, false>(q, err, made);
            }
            bad |= r.bad;
            item_done += r.done;
        }
        csync();   // every add of the slice is complete
        account(d.q1 - 1);
        // a count the last period's adds took past 2^31-1 reads negative
        {
            const int half = (d.q1 - d.q0) & 1;
            if (sm) {
                for (int i = threadIdx.x; i < wpc; i += kRunBlock)
                    for (int t = rank * wpc + i, bit = 0; t < T; t += W, ++bit) {
                        const int32_t c = data[2 * wpc + 2 * (bit * wpc + i) + half];
                        if (c < 0) bad |= kErrOverflow;
                        d.N[0][t] = c;
                    }
            }
            for (int t = rank * kRunBlock + threadIdx.x; !sm && t < T; t += kC * kRunBlock) {
                if (inter) {
                    // the slice's counts are in the pairs' half (q1 - q0) & 1;
                    // hand them back in N[0]
                    const int32_t c = __ldcg(d.N2 + 2 * (int64_t)t + half);
                    if (c < 0) bad |= kErrOverflow;
                    d.N[0][t] = c;
                } else {
                    for (int s = 0; s < S; ++s)
                        if (__ldcg(d.N[half] + (int64_t)s * T + t) < 0) bad |= kErrOverflow;
                }
            }
        }
        if (bad) atomicOr(err, bad);
        done += item_done;
        if (times) {
            if (lane == 0 && item_done) atomicAdd(times + 4 * slot + 2, item_done);
            if (rank == 0 && threadIdx.x == 0) times[4 * slot + 1] = globaltimer_ns();
        }
    }
    // entries processed: counted by lane 0 of each warp (warp-uniform)
    if (lane == 0 && done) atomicAdd(processed, done);
}

__global__ void k_pack(int32_t T, const int4* __restrict__ src, const uint4* __restrict__ thr, uint4* __restrict__ out) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    int4 s4 = src[t];
    out[2 * t] = make_uint4((uint32_t)s4.x, (uint32_t)s4.y, (uint32_t)s4.z, (uint32_t)s4.w);
    out[2 * t + 1] = thr[t];
}

void launch_pack(int32_t T, const int4* src, const uint4* thr, uint4* out, cudaStream_t st) {
    k_pack<<<(T + 255) / 256, 256, 0, st>>>(T, src, thr, out);
    note_launch();
}

// Arguments of one engine launch.  `clusters` is the number of simulations
// to keep in flight (0: as many clusters as fit on the GPU at once); the
// launch never asks for more clusters than fit, since a persistent cluster
// that cannot be resident would only start when another one has finished.
struct EngineLaunch {
    const SlotDesc* descs;
    const ModelParams* mps;
    const int32_t* order;
    int32_t n_items;
    int32_t* head;
    uint32_t* err;
    unsigned long long* processed;
    unsigned long long* times;
    cudaStream_t st;
    int sms;
    int clusters;
    int S;                // largest species count of the group's simulations
    size_t data = 0;      // bytes of counts and bitmaps in a CTA's shared memory (0: in global memory)
    int used = 0;         // clusters launched
    int max_active = 0;   // clusters resident at once (occupancy query)
    bool query_only = false;   // fill max_active, launch nothing
};

// What of a CTA's shared memory one species' counts and bitmaps may take: the rest
// of the SM's 256 KB caches the records of simulations that stay in global memory.
inline size_t sm_data_limit(bool react) {
    return 128 * 1024 - (sizeof(SlotDesc) + sizeof(ModelParams) + 256) -
           (size_t)kWarps * engine_warp_words(1, react) * sizeof(int32_t);
}

template <int SA, bool R, int C>
cudaError_t launch_cluster(EngineLaunch& L) {
    auto kern = k_engine_run<SA, R, C>;
    // the attribute covers every group of this kernel, whatever its species
    const size_t most = (size_t)kWarps * engine_warp_words(SA == 1 ? 1 : kMaxS, R) * sizeof(int32_t) +
                        (SA == 1 ? sm_data_limit(R) : kListBytes);
    const size_t dyn = (size_t)kWarps * engine_warp_words(L.S, R) * sizeof(int32_t) + L.data;
    const cudaError_t ce = allow_shared((const void*)kern, dyn, most);
    if (ce != cudaSuccess) return ce;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C, 1, 1);
    cfg.blockDim = dim3(kRunBlock, 1, 1);
    cfg.dynamicSmemBytes = dyn;
    cfg.stream = L.st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int fit = 0;
    if (C == 1) {
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kRunBlock, dyn) == cudaSuccess)
            fit = per_sm * L.sms;
    } else if (cudaOccupancyMaxActiveClusters(&fit, kern, &cfg) != cudaSuccess) {
        fit = 0;
    }
    cudaGetLastError();
    if (fit <= 0) fit = std::max(1, L.sms / C);
    L.max_active = fit;
    if (L.query_only) return cudaSuccess;
    int n = L.clusters > 0 ? std::min(L.clusters, fit) : fit;
    n = std::max(1, std::min(n, L.n_items));
    L.used = n;
    if (C == 1) {
        kern<<<n, kRunBlock, dyn, L.st>>>(L.descs, L.mps, L.order, L.n_items, L.head, L.err, L.processed,
                                          L.times);
        return cudaGetLastError();
    }
    cfg.gridDim = dim3(n * C, 1, 1);
    return cudaLaunchKernelEx(&cfg, kern, L.descs, L.mps, L.order, L.n_items, L.head, L.err, L.processed,
                              L.times);
}

template <int SA>
cudaError_t launch_run_sa(bool react, int cluster, EngineLaunch& L) {
    if (cluster >= 8) return react ? launch_cluster<SA, true, 8>(L) : launch_cluster<SA, false, 8>(L);
    if (cluster == 4) return react ? launch_cluster<SA, true, 4>(L) : launch_cluster<SA, false, 4>(L);
    if (cluster == 2) return react ? launch_cluster<SA, true, 2>(L) : launch_cluster<SA, false, 2>(L);
    return react ? launch_cluster<SA, true, 1>(L) : launch_cluster<SA, false, 1>(L);
}

// log2 of a bitmap's words: at least T / 32 and the warps of a cluster.
inline int words_shift(int64_t T, int cluster) {
    int s = 4;
    while ((1 << s) < cluster * kWarps || ((int64_t)32 << s) < T) ++s;
    return s;
}

// Kernel groups of a step: by species class (1, 2, up to 4, up to 8, more: it
// sets the shared memory of a warp), with and without reactions.
constexpr int kGroups = 10;
inline int group_of(int S, int R) {
    const int c = S <= 1 ? 0 : (S <= 2 ? 1 : (S <= 4 ? 2 : (S <= 8 ? 3 : 4)));
    return 2 * c + (R > 0 ? 1 : 0);
}
cudaError_t launch_group(int g, int cluster, EngineLaunch& L) {
    constexpr int most[5] = {1, 2, 4, 8, kMaxS};
    L.S = most[g >> 1];
    return g >> 1 ? launch_run_sa<0>((g & 1) != 0, cluster, L) : launch_run_sa<1>((g & 1) != 0, cluster, L);
}

// Bytes of a CTA's shared memory that a simulation's counts and bitmaps take,
// or 0 where they stay in global memory: one species, all its words in a
// warp's kSmCols columns, and room.
inline size_t sm_need(int64_t T, int S, int R, int cluster) {
    const int shift = words_shift(T, cluster);
    if (S != 1 || (1 << shift) > 32 * kSmCols * cluster * kWarps) return 0;
    const size_t b = sm_bytes(T, shift, cluster);
    return b <= sm_data_limit(R > 0) ? b : 0;
}

// Every instantiation of the engine kernel is launched once, with no work
// items, when the first engine is created on a device: each cluster takes an
// item index past the end and leaves, touching only the queue head (reset
// afterwards).  A step launches one kernel per species group on concurrent
// streams, and on the serving mix a step whose groups included kernels not
// launched before in the process ran the groups one after another (each
// started when the previous one ended) instead of side by side.
// head: int32[kGroups] of the engine being created (set to zero before, since a
// fresh allocation may hold anything and a negative index would be taken for
// an item, and left zero); err and
// processed: its error word and entry counter (not written: no item runs).
void warm_engine_kernels(int32_t* head, uint32_t* err, unsigned long long* processed, int sms) {
    static std::mutex mu;
    static std::vector<int> warmed;   // devices done
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return;
    }
    std::lock_guard<std::mutex> lock(mu);
    if (std::find(warmed.begin(), warmed.end(), dev) != warmed.end()) return;
    if (cudaMemsetAsync(head, 0, sizeof(int32_t) * kGroups, (cudaStream_t)0) != cudaSuccess) {
        cudaGetLastError();
        return;
    }
    EngineLaunch W{nullptr, nullptr, nullptr, 0, head, err, processed, nullptr, (cudaStream_t)0, sms, 1, 1};
    for (int g = 0; g < 4; ++g)   // every kernel: one species or several, with or without reactions
        for (int c = 1; c <= 8; c <<= 1) {
            if (launch_group(g, c, W) == cudaSuccess) note_launch();
            cudaGetLastError();   // a failure here shows again, and is reported, at a real launch
        }
    cudaMemsetAsync(head, 0, sizeof(int32_t) * kGroups, (cudaStream_t)0);
    cudaStreamSynchronize((cudaStream_t)0);
    cudaGetLastError();
    warmed.push_back(dev);
}

}  // namespace

struct rdsplit_engine {
    int32_t max_slots = 0;
    int64_t capacity = 0;
    cudaStream_t stream = 0;
    SlotDesc* d_desc = nullptr;
    ModelParams* d_mp = nullptr;
    int32_t* d_order = nullptr;
    int32_t* d_head = nullptr;
    uint32_t* err = nullptr;
    unsigned long long* processed = nullptr;  // (slot, tet) entries processed so far
    unsigned long long* d_times = nullptr;    // [max_slots][4] start, end (ns), entries of each slot's last slice
    int64_t launches = 0;                     // persistent launches issued
    int64_t steps = 0;                        // periods advanced, summed over step calls
    int32_t timing = 0;                       // time every launch with CUDA events
    cudaEvent_t ev[2] = {nullptr, nullptr};
    double timing_ms = 0.0;
    int64_t timing_n = 0;
    int sms = 1;
    int32_t concurrency = 0;                  // simulations in flight (0 = as many as fit)
    int32_t last_in_flight = 0;               // clusters of the last launch
    int32_t last_max_active = 0;              // clusters that fit at once in the last launch
    int64_t slice_work = 0;                   // tet-periods per simulation and step call (0: no limit)
    int32_t last_groups = 0;                  // kernel groups of the last launch
    cudaStream_t aux[kGroups] = {};                // one stream per kernel group
    cudaEvent_t ev_fork = nullptr;
    cudaEvent_t ev_join[kGroups] = {};
    int32_t cluster = 2;                      // CTAs per simulation (1, 2, 4 or 8)
    bool cluster_auto = false;                // chosen at each step for the simulations at hand
    std::vector<rdsplit_mesh_t> slot_mesh;    // null = free
    std::vector<SlotDesc> h_desc;
    std::vector<int32_t> slot_q;              // local periods done
    std::vector<double> slot_t_end;
    std::vector<int32_t> finished;            // slots finished and not yet reported
    int64_t active_tets = 0;

    ~rdsplit_engine() {
        for (cudaEvent_t x : ev)
            if (x) cudaEventDestroy(x);
        if (ev_fork) cudaEventDestroy(ev_fork);
        for (cudaEvent_t x : ev_join)
            if (x) cudaEventDestroy(x);
        for (cudaStream_t x : aux)
            if (x) cudaStreamDestroy(x);
        void* ps[] = {d_desc, d_mp, d_order, d_head, err, processed, d_times};
        for (void* p : ps) rdapi::dev_free(p);
    }
};

namespace {

int engine_err(rdsplit_engine* e, const char* where) {
    uint32_t v = 0;
    cudaError_t ce = cudaMemcpyAsync(&v, e->err, sizeof v, cudaMemcpyDeviceToHost, e->stream);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(e->stream);
    if (ce != cudaSuccess) {
        cudaGetLastError();
        return rdapi::fail(RDSPLIT_ECUDA, "%s: %s", where, cudaGetErrorString(ce));
    }
    if (v == 0) return RDSPLIT_OK;
    cudaMemsetAsync(e->err, 0, sizeof(uint32_t), e->stream);
    if (v & kErrOverflow) return rdapi::fail(RDSPLIT_EOVERFLOW, "%s: count overflow", where);
    if (v & kErrEventCap) return rdapi::fail(RDSPLIT_EOVERFLOW, "%s: SSA event cap exceeded", where);
    if (v & kErrNegative) return rdapi::fail(RDSPLIT_EINVAL, "%s: negative count", where);
    return rdapi::fail(RDSPLIT_ECUDA, "%s: device error bits 0x%x", where, v);
}

// Periods to reach t_end from t with Algorithm 1 (Step 1 aligns the last one)
// and the length of the last period.
void plan_periods(double t, double tau, double t_end, int64_t* P, double* tau_last, bool* last_short) {
    int64_t n = 0;
    *tau_last = tau;
    *last_short = false;
    while (t < t_end) {
        if (t + tau > t_end) {
            *tau_last = t_end - t;
            *last_short = true;
            t = t_end;
        } else {
            t = t + tau;
        }
        ++n;
    }
    *P = n;
}

// What a simulation costs a cluster of c CTAs, in arbitrary units: a period has
// a part that no CTA takes off (its serial chain and barrier) and one that they
// share (36, 22, 14 and 10 us were measured on 1, 2, 4 and 8 CTAs for 3,000
// occupied tets).
inline double slice_cost(const rdsplit_engine* e, int32_t s, int c) {
    const rdsplit_mesh* h = e->slot_mesh[s];
    return (double)(e->h_desc[s].q1 - e->h_desc[s].q0) * (0.25 + std::min(1.0, (double)h->T / 8192.0) * h->S / c);
}

// CTAs per simulation for a whole ensemble: the size whose schedule (longest
// first, each simulation to the cluster that is free first) ends soonest.  Its
// choice was the fastest of the four sizes for 512 cubes of 6 to 40 cells a side
// (2 CTAs: 1.42 s; 2.54, 1.63, 2.69 on 1, 4, 8), 40 cubes of 6 to 24 (8: 14 ms;
// 52, 37, 30 on 1, 2, 4), 24 of them with A/B/C (8: 5.0 ms; 26, 16, 9.0) and 152
// tubes of 960 tets (1: 5.7 ms; 9.4, 20, 43 on 2, 4, 8).
int choose_cluster(rdsplit_engine* e, const std::vector<int32_t>& items) {
    int best = 2;
    double best_end = HUGE_VAL;
    for (int c = 1; c <= 8; c <<= 1) {
        EngineLaunch Q{nullptr, nullptr, nullptr, 1, nullptr, nullptr, nullptr, nullptr, e->stream, e->sms, 0, 1};
        Q.query_only = true;
        std::vector<double> cost;
        for (int32_t s : items) cost.push_back(slice_cost(e, s, c));
        const rdsplit_mesh* first = e->slot_mesh[items[0]];
        if (launch_group(group_of(first->S, first->R), c, Q) != cudaSuccess) {
            cudaGetLastError();
            continue;
        }
        std::sort(cost.begin(), cost.end(), [](double a, double b) { return a > b; });
        std::priority_queue<double, std::vector<double>, std::greater<double>> free_at;
        for (int i = 0; i < Q.max_active; ++i) free_at.push(0.0);
        double end = 0.0;
        for (double w : cost) {
            const double t = free_at.top() + w;
            free_at.pop();
            free_at.push(t);
            end = std::max(end, t);
        }
        if (end < best_end) {
            best_end = end;
            best = c;
        }
    }
    return best;
}

void finish_slot(rdsplit_engine* e, int slot) {
    rdsplit_mesh* h = e->slot_mesh[slot];
    const SlotDesc& d = e->h_desc[slot];
    // a simulation added with t_end at or before its time ran no period and
    // keeps its time, as rdsplit_run would
    if (d.P > 0) h->t = e->slot_t_end[slot];
    h->period = (int64_t)d.period0 + d.P;
    e->active_tets -= h->T;
    e->slot_mesh[slot] = nullptr;
    e->finished.push_back(slot);
}

}  // namespace

extern "C" {

int rdsplit_engine_create(int32_t max_slots, int64_t max_active_tets, rdsplit_engine_t* out) {
    if (!out) return rdapi::fail(RDSPLIT_EINVAL, "rdsplit_engine_create: out is NULL");
    *out = nullptr;
    if (max_slots < 1 || max_slots > (1 << 20)) return rdapi::fail(RDSPLIT_EINVAL, "rdsplit_engine_create: bad max_slots");
    if (max_active_tets < 1) return rdapi::fail(RDSPLIT_EINVAL, "rdsplit_engine_create: max_active_tets must be >= 1");
    rdsplit_engine* e = new rdsplit_engine();
    e->max_slots = max_slots;
    e->capacity = max_active_tets;
    e->d_desc = (SlotDesc*)rdapi::dev_alloc(sizeof(SlotDesc) * max_slots);
    e->d_mp = (ModelParams*)rdapi::dev_alloc(sizeof(ModelParams) * max_slots);
    e->d_order = (int32_t*)rdapi::dev_alloc(sizeof(int32_t) * max_slots);
    e->d_head = (int32_t*)rdapi::dev_alloc(sizeof(int32_t) * kGroups);
    e->err = (uint32_t*)rdapi::dev_alloc(sizeof(uint32_t));
    e->processed = (unsigned long long*)rdapi::dev_alloc(sizeof(unsigned long long));
    e->d_times = (unsigned long long*)rdapi::dev_alloc(sizeof(unsigned long long) * 4 * max_slots);
    if (!e->d_desc || !e->d_mp || !e->d_order || !e->d_head || !e->err || !e->processed || !e->d_times) {
        delete e;
        return rdapi::fail(RDSPLIT_ENOMEM, "rdsplit_engine_create: device allocation failed");
    }
    e->slot_mesh.assign(max_slots, nullptr);
    e->h_desc.assign(max_slots, SlotDesc{});
    e->slot_q.assign(max_slots, 0);
    e->slot_t_end.assign(max_slots, 0.0);
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&e->sms, cudaDevAttrMultiProcessorCount, dev);
    warm_engine_kernels(e->d_head, e->err, e->processed, e->sms);
    if (cudaMemsetAsync(e->processed, 0, sizeof(unsigned long long), e->stream) != cudaSuccess ||
        cudaMemsetAsync(e->d_times, 0, sizeof(unsigned long long) * 4 * max_slots, e->stream) != cudaSuccess ||
        cudaMemsetAsync(e->err, 0, sizeof(uint32_t), e->stream) != cudaSuccess) {
        cudaGetLastError();
        delete e;
        return rdapi::fail(RDSPLIT_ECUDA, "rdsplit_engine_create: memset failed");
    }
    *out = e;
    return RDSPLIT_OK;
}

int rdsplit_engine_set_stream(rdsplit_engine_t e, void* stream) {
    if (!e) return rdapi::fail(RDSPLIT_EINVAL, "rdsplit_engine_set_stream: NULL engine");
    e->stream = (cudaStream_t)stream;
    return RDSPLIT_OK;
}

int rdsplit_engine_add(rdsplit_engine_t e, rdsplit_mesh_t h, double t_end, uint64_t seed, int32_t* slot_out) {
    const char* where = "rdsplit_engine_add";
    if (!e || !h) return rdapi::fail(RDSPLIT_EINVAL, "%s: NULL argument", where);
    if (!h->has_model) return rdapi::fail(RDSPLIT_ESTATE, "%s: the mesh has no model", where);
    if (std::isnan(t_end)) return rdapi::fail(RDSPLIT_EINVAL, "%s: t_end is NaN", where);
    for (int s = 0; s < e->max_slots; ++s)
        if (e->slot_mesh[s] == h) return rdapi::fail(RDSPLIT_EINVAL, "%s: mesh already in the engine", where);
    int slot = -1;
    for (int s = 0; s < e->max_slots; ++s)
        if (!e->slot_mesh[s]) { slot = s; break; }
    if (slot < 0) return rdapi::fail(RDSPLIT_ENOMEM, "%s: no free slot", where);
    if (e->active_tets + h->T > e->capacity)
        return rdapi::fail(RDSPLIT_ENOMEM, "%s: active-tet capacity %lld exceeded", where, (long long)e->capacity);
    int64_t P = 0;
    double tau_last = h->tau;
    bool last_short = false;
    plan_periods(h->t, h->tau, t_end, &P, &tau_last, &last_short);
    if (h->period + P > (int64_t)0xffffffffll) return rdapi::fail(RDSPLIT_EOVERFLOW, "%s: period index exceeds 2^32-1", where);
    if (P > 0x7fffffffll) return rdapi::fail(RDSPLIT_EINVAL, "%s: too many periods", where);
    const size_t T = (size_t)h->T;
    const size_t W = (size_t)1 << words_shift(h->T, 8);   // for any cluster size
    if (!h->bits[0]) {
        h->bits[0] = (uint32_t*)rdapi::dev_alloc(4 * W);
        h->bits[1] = (uint32_t*)rdapi::dev_alloc(4 * W);
        if (!h->bits[0] || !h->bits[1]) return rdapi::fail(RDSPLIT_ENOMEM, "%s: bitmap allocation failed", where);
    }
    cudaStream_t st = e->stream;
    cudaError_t ce = cudaMemsetAsync(h->bits[0], 0, 4 * W, st);
    if (ce == cudaSuccess) ce = cudaMemsetAsync(h->bits[1], 0, 4 * W, st);
    if (ce == cudaSuccess) ce = cudaMemsetAsync(h->rem, 0, sizeof(int32_t) * T * h->S, st);
    if (ce != cudaSuccess) {
        cudaGetLastError();
        return rdapi::fail(RDSPLIT_ECUDA, "%s: memset failed: %s", where, cudaGetErrorString(ce));
    }
    if (last_short) launch_thresholds(h->T, h->mp, h->g, h->G, tau_last, h->thr_last, st);
    // one species: packed per-tet records and interleaved counts (fewer cache
    // lines per active tet)
    const bool pack = h->S == 1;
    if (pack && !h->packed) {
        h->packed = (uint4*)rdapi::dev_alloc(32 * T);
        h->N2 = (int2*)rdapi::dev_alloc(8 * T);
        if (!h->packed || !h->N2) return rdapi::fail(RDSPLIT_ENOMEM, "%s: packed-record allocation failed", where);
    }
    if (pack) launch_pack(h->T, h->src, h->thr, h->packed, st);
    SlotDesc d{};
    d.m = h->dev_mesh();
    d.thr = h->thr;
    d.thr_last = last_short ? h->thr_last : h->thr;
    d.N[0] = h->cnt;
    d.N[1] = h->rem;
    d.bits[0] = h->bits[0];
    d.bits[1] = h->bits[1];
    d.wshift = 0;   // set at each step
    d.packed = pack ? h->packed : nullptr;
    d.N2 = pack ? reinterpret_cast<int32_t*>(h->N2) : nullptr;
    d.seed = seed;
    d.period0 = (uint32_t)h->period;
    d.P = (int32_t)P;
    d.q0 = d.q1 = 0;
    d.last_short = last_short ? 1 : 0;
    d.S = h->S;
    d.zero_order = 0;
    for (int r = 0; r < h->R; ++r)
        if (h->mp.order[r] == 0 && h->mp.k[r] > 0.0) d.zero_order |= 1u << r;
    d.tau = h->tau;
    d.tau_last = tau_last;
    d.tauf = (float)h->tau;
    d.tau_lastf = (float)tau_last;
    ce = cudaMemcpyAsync(e->d_mp + slot, &h->mp, sizeof(ModelParams), cudaMemcpyHostToDevice, st);
    if (ce != cudaSuccess) {
        cudaGetLastError();
        return rdapi::fail(RDSPLIT_ECUDA, "%s: model upload failed: %s", where, cudaGetErrorString(ce));
    }
    e->h_desc[slot] = d;
    e->slot_mesh[slot] = h;
    e->slot_q[slot] = 0;
    e->slot_t_end[slot] = t_end;
    e->active_tets += h->T;
    if (P == 0) finish_slot(e, slot);
    if (slot_out) *slot_out = slot;
    return RDSPLIT_OK;
}

// Advance every active simulation by up to n_steps periods in one persistent
// launch.  Finished handles receive their counts, time and period index;
// their slot ids are queued for rdsplit_engine_poll.
int rdsplit_engine_step(rdsplit_engine_t e, int64_t n_steps) {
    const char* where = "rdsplit_engine_step";
    if (!e) return rdapi::fail(RDSPLIT_EINVAL, "%s: NULL engine", where);
    if (n_steps <= 0) return RDSPLIT_OK;
    std::vector<int32_t> items;
    std::vector<double> work;
    int64_t max_adv = 0;
    for (int s = 0; s < e->max_slots; ++s) {
        rdsplit_mesh* h = e->slot_mesh[s];
        if (!h) continue;
        SlotDesc& d = e->h_desc[s];
        d.q0 = e->slot_q[s];
        // periods of this slice: n_steps, or fewer for a large simulation
        // when a work budget per slice is set (tets x periods), so that the
        // slices of one launch cost about the same
        int64_t n = n_steps;
        if (e->slice_work > 0) n = std::max<int64_t>(1, std::min<int64_t>(n_steps, e->slice_work / h->T));
        d.q1 = (int32_t)std::min<int64_t>((int64_t)d.P, (int64_t)d.q0 + n);
        if (d.q1 <= d.q0) continue;
        items.push_back(s);
        work.push_back((double)(d.q1 - d.q0) * (double)h->T * (double)h->S);
        max_adv = std::max<int64_t>(max_adv, d.q1 - d.q0);
    }
    if (items.empty()) return engine_err(e, where);
    // Simulations are launched in groups of one kernel and shared-memory size
    // each.  Groups run concurrently on their own streams, the resident
    // clusters shared among them by work; largest first in each.
    auto cls_of = [&](int s) { return group_of(e->slot_mesh[s]->S, e->slot_mesh[s]->R); };
    if (e->cluster_auto) e->cluster = choose_cluster(e, items);
    const int csize = e->cluster;
    size_t g_data[kGroups] = {0};
    for (int32_t s : items) {
        const rdsplit_mesh* h = e->slot_mesh[s];
        const size_t need = sm_need(h->T, h->S, h->R, csize);
        e->h_desc[s].wshift = words_shift(h->T, csize);
        e->h_desc[s].sm = need > 0 ? 1 : 0;
        g_data[cls_of(s)] = std::max(g_data[cls_of(s)], need > 0 ? need : kListBytes);
    }
    std::vector<size_t> idx(items.size());
    std::iota(idx.begin(), idx.end(), 0);
    std::stable_sort(idx.begin(), idx.end(), [&](size_t a, size_t b) {
        const int ga = cls_of(items[a]), gb = cls_of(items[b]);
        return ga != gb ? ga < gb : work[a] > work[b];
    });
    std::vector<int32_t> order(items.size());
    int g_begin[kGroups + 1] = {0};
    double g_work[kGroups] = {0.0};
    int g_count[kGroups] = {0};
    for (size_t k = 0; k < idx.size(); ++k) {
        order[k] = items[idx[k]];
        const int g = cls_of(order[k]);
        g_count[g] += 1;
        g_work[g] += work[idx[k]];
    }
    for (int g = 0; g < kGroups; ++g) g_begin[g + 1] = g_begin[g] + g_count[g];
    int n_groups = 0;
    for (int g = 0; g < kGroups; ++g) n_groups += g_count[g] > 0 ? 1 : 0;
    cudaStream_t st = e->stream;
    cudaError_t ce = cudaMemcpyAsync(e->d_desc, e->h_desc.data(), sizeof(SlotDesc) * e->max_slots,
                                     cudaMemcpyHostToDevice, st);
    if (ce == cudaSuccess)
        ce = cudaMemcpyAsync(e->d_order, order.data(), sizeof(int32_t) * order.size(), cudaMemcpyHostToDevice, st);
    if (ce == cudaSuccess) ce = cudaMemsetAsync(e->d_head, 0, sizeof(int32_t) * kGroups, st);
    if (ce != cudaSuccess) {
        cudaGetLastError();
        return rdapi::fail(RDSPLIT_ECUDA, "%s: upload failed: %s", where, cudaGetErrorString(ce));
    }
    if (e->timing && !e->ev[0]) {
        cudaEventCreate(&e->ev[0]);
        cudaEventCreate(&e->ev[1]);
    }
    if (e->timing) cudaEventRecord(e->ev[0], st);
    int used = 0, fit = 0;
    if (n_groups == 1) {
        int g = 0;
        while (g_count[g] == 0) ++g;
        // default: as many clusters as can be resident at once (one CTA per
        // SM where the GPCs allow it)
        EngineLaunch L{e->d_desc, e->d_mp, e->d_order, g_count[g], e->d_head, e->err, e->processed,
                       e->timing ? e->d_times : nullptr, st, e->sms, e->concurrency, 1};
        L.data = g_data[g];
        ce = launch_group(g, csize, L);
        used = L.used;
        fit = L.max_active;
    } else {
        // the clusters that fit, shared by work (at least one per group)
        EngineLaunch Q{e->d_desc, e->d_mp, e->d_order, 1, e->d_head, e->err, e->processed, nullptr, st, e->sms, 0, 1};
        Q.query_only = true;
        ce = launch_group(7, csize, Q);
        fit = Q.max_active;
        const int budget = e->concurrency > 0 ? std::min(e->concurrency, fit) : fit;
        double total = 0.0;
        for (int g = 0; g < kGroups; ++g) total += g_work[g];
        int share[kGroups] = {0};
        int given = 0;
        for (int g = 0; g < kGroups; ++g) {
            if (!g_count[g]) continue;
            share[g] = std::max(1, (int)((double)budget * g_work[g] / std::max(total, 1.0)));
            share[g] = std::min(share[g], g_count[g]);
            given += share[g];
        }
        while (given > std::max(budget, n_groups)) {   // trim the largest shares
            int gm = -1;
            for (int g = 0; g < kGroups; ++g)
                if (share[g] > 1 && (gm < 0 || share[g] > share[gm])) gm = g;
            if (gm < 0) break;
            share[gm] -= 1;
            given -= 1;
        }
        if (!e->ev_fork) {
            cudaEventCreateWithFlags(&e->ev_fork, cudaEventDisableTiming);
            for (int g = 0; g < kGroups; ++g) {
                cudaStreamCreateWithFlags(&e->aux[g], cudaStreamNonBlocking);
                cudaEventCreateWithFlags(&e->ev_join[g], cudaEventDisableTiming);
            }
        }
        if (ce == cudaSuccess) ce = cudaEventRecord(e->ev_fork, st);
        for (int g = 0; g < kGroups && ce == cudaSuccess; ++g) {
            if (!g_count[g]) continue;
            ce = cudaStreamWaitEvent(e->aux[g], e->ev_fork, 0);
            EngineLaunch L{e->d_desc, e->d_mp, e->d_order + g_begin[g], g_count[g], e->d_head + g, e->err,
                           e->processed, e->timing ? e->d_times : nullptr, e->aux[g], e->sms, share[g], 1};
            L.data = g_data[g];
                if (ce == cudaSuccess) ce = launch_group(g, csize, L);
            used += L.used;
            if (ce == cudaSuccess) ce = cudaEventRecord(e->ev_join[g], e->aux[g]);
            if (ce == cudaSuccess) ce = cudaStreamWaitEvent(st, e->ev_join[g], 0);
        }
    }
    EngineLaunch L{};
    L.used = used;
    L.max_active = fit;
    e->last_in_flight = L.used;
    e->last_max_active = L.max_active;
    e->last_groups = n_groups;
    if (e->timing) cudaEventRecord(e->ev[1], st);
    note_launch();
    e->launches += 1;
    if (ce == cudaSuccess) ce = cudaGetLastError();
    if (ce != cudaSuccess) {
        cudaGetLastError();
        return rdapi::fail(RDSPLIT_ECUDA, "%s: launch failed: %s", where, cudaGetErrorString(ce));
    }
    int rc = engine_err(e, where);
    if (e->timing) {
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, e->ev[0], e->ev[1]) == cudaSuccess) {
            e->timing_ms += ms;
            e->timing_n += 1;
        }
        cudaGetLastError();
    }
    e->steps += max_adv;
    // the slice leaves each simulation's counts in N[(q1 - q0) & 1]
    for (int32_t s : items) {
        SlotDesc& d = e->h_desc[s];
        rdsplit_mesh* h = e->slot_mesh[s];
        if (((d.q1 - d.q0) & 1) && !d.N2) {
            std::swap(d.N[0], d.N[1]);
            std::swap(h->cnt, h->rem);
        }
        e->slot_q[s] = d.q1;
        if (d.q1 == d.P) finish_slot(e, s);
    }
    return rc;
}

int rdsplit_engine_poll(rdsplit_engine_t e, int32_t* slots, int32_t max, int32_t* n_out) {
    if (!e || !n_out) return rdapi::fail(RDSPLIT_EINVAL, "rdsplit_engine_poll: NULL argument");
    int32_t n = 0;
    while (n < max && !e->finished.empty()) {
        slots[n++] = e->finished.front();
        e->finished.erase(e->finished.begin());
    }
    *n_out = n;
    return RDSPLIT_OK;
}

int rdsplit_engine_active(rdsplit_engine_t e, int32_t* n_slots, int64_t* n_tets) {
    if (!e) return rdapi::fail(RDSPLIT_EINVAL, "rdsplit_engine_active: NULL engine");
    int32_t n = 0;
    for (int s = 0; s < e->max_slots; ++s) n += e->slot_mesh[s] ? 1 : 0;
    if (n_slots) *n_slots = n;
    if (n_tets) *n_tets = e->active_tets;
    return RDSPLIT_OK;
}

int rdsplit_engine_set_concurrency(rdsplit_engine_t e, int32_t in_flight, int32_t cluster) {
    if (!e || in_flight < 0 || !(cluster == 1 || cluster == 2 || cluster == 4 || cluster == 8))
        return rdapi::fail(RDSPLIT_EINVAL, "rdsplit_engine_set_concurrency: bad argument");
    e->concurrency = in_flight;
    e->cluster = cluster;
    return RDSPLIT_OK;
}

int rdsplit_engine_set_slice_work(rdsplit_engine_t e, int64_t max_tet_periods) {
    if (!e || max_tet_periods < 0) return rdapi::fail(RDSPLIT_EINVAL, "rdsplit_engine_set_slice_work: bad argument");
    e->slice_work = max_tet_periods;
    return RDSPLIT_OK;
}

int rdsplit_engine_schedule(rdsplit_engine_t e, int32_t* in_flight, int32_t* cluster, int32_t* max_active) {
    if (!e) return rdapi::fail(RDSPLIT_EINVAL, "rdsplit_engine_schedule: NULL engine");
    if (in_flight) *in_flight = e->last_in_flight;
    if (cluster) *cluster = e->cluster;
    if (max_active) *max_active = e->last_max_active;
    return RDSPLIT_OK;
}

int rdsplit_engine_set_timing(rdsplit_engine_t e, int32_t on) {
    if (!e || on < 0) return rdapi::fail(RDSPLIT_EINVAL, "rdsplit_engine_set_timing: bad argument");
    e->timing = on;
    e->timing_ms = 0.0;
    e->timing_n = 0;
    return RDSPLIT_OK;
}

int rdsplit_engine_stats(rdsplit_engine_t e, int64_t* steps, int64_t* processed, double* timing_ms,
                         int64_t* timing_n) {
    if (!e) return rdapi::fail(RDSPLIT_EINVAL, "rdsplit_engine_stats: NULL engine");
    unsigned long long p = 0;
    cudaError_t ce = cudaMemcpyAsync(&p, e->processed, sizeof p, cudaMemcpyDeviceToHost, e->stream);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(e->stream);
    if (ce != cudaSuccess) {
        cudaGetLastError();
        return rdapi::fail(RDSPLIT_ECUDA, "rdsplit_engine_stats: %s", cudaGetErrorString(ce));
    }
    if (steps) *steps = e->steps;
    if (processed) *processed = (int64_t)p;
    if (timing_ms) *timing_ms = e->timing_ms;
    if (timing_n) *timing_n = e->timing_n;
    return RDSPLIT_OK;
}

int rdsplit_engine_slot_times(rdsplit_engine_t e, int64_t* out, int32_t max_slots) {
    if (!e || !out || max_slots < 0)
        return rdapi::fail(RDSPLIT_EINVAL, "rdsplit_engine_slot_times: bad argument");
    const int32_t n = std::min(max_slots, e->max_slots);
    std::vector<unsigned long long> buf(4 * (size_t)n);
    cudaError_t ce = cudaMemcpyAsync(buf.data(), e->d_times, sizeof(unsigned long long) * 4 * (size_t)n,
                                     cudaMemcpyDeviceToHost, e->stream);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(e->stream);
    for (int32_t i = 0; ce == cudaSuccess && i < n; ++i)
        for (int k = 0; k < 3; ++k) out[3 * i + k] = (int64_t)buf[4 * i + k];
    if (ce != cudaSuccess) {
        cudaGetLastError();
        return rdapi::fail(RDSPLIT_ECUDA, "rdsplit_engine_slot_times: %s", cudaGetErrorString(ce));
    }
    return RDSPLIT_OK;
}

int rdsplit_engine_destroy(rdsplit_engine_t e) {
    if (!e) return RDSPLIT_OK;
    cudaStreamSynchronize(e->stream);
    delete e;
    return RDSPLIT_OK;
}

int rdsplit_ensemble_run(int32_t n, const rdsplit_mesh_t* meshes, const double* t_end, const uint64_t* seeds) {
    const char* where = "rdsplit_ensemble_run";
    if (n < 1 || !meshes || !t_end || !seeds) return rdapi::fail(RDSPLIT_EINVAL, "%s: bad arguments", where);
    int64_t tets = 0;
    for (int i = 0; i < n; ++i) {
        if (!meshes[i]) return rdapi::fail(RDSPLIT_EINVAL, "%s: NULL mesh %d", where, i);
        tets += meshes[i]->T;
    }
    rdsplit_engine_t e = nullptr;
    int rc = rdsplit_engine_create(n, tets, &e);
    if (rc) return rc;
    e->stream = meshes[0]->stream;
    e->cluster_auto = true;
    for (int i = 0; i < n && rc == RDSPLIT_OK; ++i) rc = rdsplit_engine_add(e, meshes[i], t_end[i], seeds[i], nullptr);
    if (rc == RDSPLIT_OK) rc = rdsplit_engine_step(e, INT64_MAX / 4);
    rdsplit_engine_destroy(e);
    return rc;
}

}  // extern "C"
