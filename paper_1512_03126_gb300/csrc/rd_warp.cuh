// One period (Algorithm 1 of arXiv:1512.03126, Steps 2 and 3) for the 32 tets
// of a warp, one per lane, with the tets' counts in shared memory.
//
// What bounds a period of a small mesh is the serial chain of its slowest
// tet, and of a large one the instructions and bytes spent on tets where
// nothing happens.  Three things follow from that here:
//
//  * Counts live in shared-memory columns ([species][lane]), so that loops
//    over species and reactions index them at run time without a register
//    array per species count (no local memory, one code path for 1 to 16
//    species, fewer registers).
//  * The diffusion draws of all lanes and species form one list of Philox
//    blocks (four molecules each) that the warp works off 32 at a time
//    (draw_all).
//  * The reaction phase runs in single precision with error bounds that
//    certify every decision (react_fast); only a decision inside its bound
//    repeats the tet in double precision (react_exact).
//
// Against kernels with the counts in registers, one whole-warp pass per tet of
// ten molecules or more, the reaction phase in double precision and one launch a
// period, this step and the kernels around it take, on GB300 (a run of periods,
// counts in and out): 3,072-tet point source, 217 periods, 5.0 -> 0.8 ms;
// 48,000-tet A/B/C cube, 200 periods, 4.1 -> 1.8 ms; six species, 68,034 tets,
// 100 periods, 9.3 -> 2.0 ms; 2.4 M-tet bar, 24 periods, 9.5 -> 3.4 ms.
//
// Every draw uses the words of the same keyed stream as the sequential
// definition, so the counts are the same whole numbers.
#pragma once
#include "rd_device.cuh"
#include "rd_internal.h"
#include "rd_period.cuh"

namespace rdk {

constexpr unsigned kAllLanes = 0xffffffffu;
// A species with more draws than this is drawn by the whole warp together
// (at least a full round of 32 Philox blocks); below it its blocks go to the
// shared list.
constexpr int32_t kCoopMin = 128;
// A tet with this many molecules of a species is deferred to the pass with the
// double-precision samplers: below it, with at most kMoleculeCut / 2 made or
// consumed in the period, N* stays below kMoleculeCut.
constexpr int32_t kDeferMin = (int32_t)kMoleculeCut / 2;
constexpr int kListWords = 64;   // draw list of a warp (a round takes 32 entries)

// Shared memory of one warp: N, D (draws of species a reaction touched) and
// acc[0], acc[1] (leavers per face, two 16-bit counts a word) as columns
// [species][32], and the draw list.
__host__ __device__ inline int warp_words(int S, bool react) { return 32 * S * (react ? 4 : 3) + kListWords; }

struct WarpMem {
    int32_t* N;
    int32_t* D;
    uint32_t* acc0;
    uint32_t* acc1;
    uint32_t* list;
    const uint2* rx;      // reaction table (ModelParams::rx) in shared memory
    __device__ __forceinline__ WarpMem(int32_t* base, int S, bool react, const uint2* rx_) : rx(rx_) {
        N = base;
        acc0 = reinterpret_cast<uint32_t*>(N + 32 * S);
        acc1 = acc0 + 32 * S;
        list = acc1 + 32 * S;
        D = react ? reinterpret_cast<int32_t*>(list + kListWords) : N;
    }
};

// What a period pass needs beside the mesh and the model.
struct PeriodView {
    uint32_t period;
    double tau_k;
    float tau_kf;
    uint64_t seed;
    const uint4* thr;    // thresholds of (species s, tet t) at (s T + t) * thr_stride
    int thr_stride;
};

// Which species of a lane's tet have molecules, which more than one, which
// more than kCoopMin or kDeferMin: kept beside the column, so that loops run over set bits
// only.
struct Presence {
    uint32_t any = 0, two = 0;
    uint32_t many = 0;   // lower half: more than kCoopMin; upper half: kDeferMin or more
    // a species not seen before
    __device__ __forceinline__ void add(int s, int32_t n) {
        if (n > 0) any |= 1u << s;
        if (n > 1) two |= 1u << s;
        if (n > kCoopMin) many |= (n >= kDeferMin ? 0x10001u : 1u) << s;
    }
    __device__ __forceinline__ void set(int s, int32_t n) {
        const uint32_t bit = 1u << s;
        any &= ~bit;
        two &= ~bit;
        many &= ~(bit * 0x10001u);
        add(s, n);
    }
};

__device__ __forceinline__ Presence presence_of(const int32_t* Ncol, int S) {
    Presence pr;
    for (int s = 0; s < S; ++s) pr.add(s, Ncol[32 * s]);
    return pr;
}

// Reactions of `on` whose reactants are present.
__device__ __forceinline__ uint32_t possible_by_presence(const ModelParams& mp, const Presence& pr, int S, uint32_t on) {
    uint32_t m = on;
#pragma unroll 4
    for (int s = 0; s < S; ++s) {
        if (!((pr.any >> s) & 1u)) m &= ~mp.needs[s];
        if (!((pr.two >> s) & 1u)) m &= ~mp.needs2[s];
    }
    return m;
}

// Propensity of a reaction of the table in single precision (relative error
// below 8 * 2^-24: three roundings in the rate, three in the combinations, one
// in their product).
__device__ __forceinline__ float propensity_f(const uint2 rx, const int32_t* Ncol, float2 avf) {
    float c = __uint_as_float(rx.x);
    const uint32_t kind = (rx.y >> 8) & 3u;
    if (kind == 0u) return c * avf.x;
    const int32_t na = Ncol[32 * (rx.y & 15u)];
    if (kind == 1u) return c * (float)na;
    c = c * avf.y;
    if (kind == 3u) return c * (0.5f * (float)na * (float)(na - 1));
    return c * ((float)na * (float)Ncol[32 * ((rx.y >> 4) & 15u)]);
}

enum : int { kReactNone = 0, kReactDone = 1, kReactDoubt = 2 };

// The reaction phase of one tet (Gillespie's direct method over one period,
// Step 2 and 2.1) in single precision.  Time is x = t / tau_k.  The mean
// occupancy telescopes: with N_end the final count and dn_i the change at
// event time x_i, N-bar = N_end - sum_i dn_i x_i, so the stochastically
// rounded N* = ceil(N-bar - u) is N_end - floor(sum_i dn_i x_i + u), whose
// error does not grow with the counts.
//
// Bounds, in units of e = 2^-24 (the reference values are the double-precision
// ones, whose own error is below 1e-10 of these), with m the largest number of
// possible reactions met: propensities 8, their sum m - 1 more; -log u1 8: by
// log1pf (1 ulp) of u1 - 1 above one half (condition at most 1.45), else of its
// mantissa beside exponent times ln 2; times tau 2, __fdividef 4 (2 ulp).  So a
// waiting time is off by at most (21 + m) e of itself and, with one rounding
// per event, an event time by (21 + m + k) e after k events.  Comparisons with
// tau_k or tau_k / 2 keep (26 + m + 2 k) e away from their limit, the choice of
// the reaction (22 + 2 m) e of the total propensity (twice the sum's error,
// and two roundings of the target), and the rounding of N-bar (30 + m + 3 k) e
// per molecule made or consumed + 4 e (event times, products, the k sums, and
// u) + 2^-20 (the double-precision sums, for counts below 2^20); inside a
// margin the function undoes its changes and answers kReactDoubt.  The margins
// matter for speed: at 128, 128 and 256 e one of the 68,034 tets of a
// six-species box met one in most periods, and its double-precision repeat set
// the period (29 us).
// Waiting times beyond the period are first ruled out by -log u >= 1 - u
// without a logarithm.
// Replaces a double-precision chain of one logarithm (24 dependent operations
// and a division) and three further divisions an event: at 64 cycles an FP64
// operation it set the period of every small mesh with reactions.
// On kReactDone: Ncol holds the counts after the phase, *touched the species
// that changed, and Dcol, for those, N* (mean rule) or the mid-period count
// (half-step rule).  scratch: the lane's column of one word per species.
__device__ __forceinline__ int react_fast(const ModelParams& mp, const uint2* rx, int S, int key, const PeriodView& v,
                                          uint32_t on, uint32_t poss, float2 avf, int32_t* Ncol, int32_t* Dcol,
                                          uint32_t* scratch, Presence& pr, uint32_t* touched_out) {
    constexpr float e = 5.9604644775390625e-08f;   // 2^-24
    constexpr int kMaxEvents = 64;
    // A tet that expects more events than this at the start of the period would
    // go past kMaxEvents, mostly (162 tets of two species, about 75 events a
    // period, 20 periods: 12.5 ms with the attempt, 11.5 without).
    float longest = 72.0f;
    const bool mid = mp.rule == kRuleMid;
    const uint32_t k0 = (uint32_t)v.seed, k1 = (uint32_t)(v.seed >> 32);
    float x = 0.0f, dsum = 0.0f;
    uint32_t touched = 0;
    int k = 0, m = 0;
    // block k of the tet's reaction stream: u1 and u2 of event k; the next one
    // is drawn beside the waiting time, off the chain from event to event
    uint4 rw = rdd::philox_block(0u, (uint32_t)key, v.period, rdd::kPurposeReaction << 16, k0, k1);
    bool past = false, doubt = !(v.tau_kf < 1e6f);   // (keeps underflowed rates below 1e-13 a period)
    while (!doubt) {
        if (k > 0) poss = possible_by_presence(mp, pr, S, on);
        if (!poss) break;                          // total propensity 0
        const uint64_t x1 = ((uint64_t)(rw.x >> 5) << 26) | (rw.y >> 6);
        float a0 = 0.0f;
        for (uint32_t bits = poss; bits; bits &= bits - 1u) a0 += propensity_f(rx[__ffs(bits) - 1], Ncol, avf);
        const float at = a0 * v.tau_kf;
        m = max(m, __popc(poss));
        const float eps = (float)(26 + m + 2 * k) * e;
        const uint64_t y = 9007199254740991ull - x1;                    // (1 - u1) 2^53
        const float ylo = (float)(uint32_t)(y >> 29) * e;               // at most 1 - u1
        if (!(at < longest)) { doubt = true; break; }
        if (ylo > 0.0f && ylo >= at * ((1.0f + eps) - x) * 1.0001f) break;   // no event before tau_k
        if (!(at > 1e-6f)) { doubt = true; break; }
        const uint4 rw_next =
            rdd::philox_block((uint32_t)(k + 1), (uint32_t)key, v.period, rdd::kPurposeReaction << 16, k0, k1);
        float arg = -(float)y * 1.1102230246251565e-16f, ex = 0.0f;     // u1 - 1
        if (y > 4503599627370496ull) {
            // u1 = 2^ex (1 + arg) below one half, arg in [-0.3, 0.42)
            const uint32_t ub = __float_as_uint((float)(x1 + 1ull) * 1.1102230246251565e-16f);
            const int ei = (int)((ub + 0x4afb0du) >> 23) - 127;
            ex = (float)ei;
            arg = __uint_as_float(ub - ((uint32_t)ei << 23)) - 1.0f;
        }
        const float E = -(log1pf(arg) + ex * 0.693147182f);
        const float xn = x + __fdividef(E, at);
        if (xn >= 1.0f + eps) break;
        if (xn > 1.0f - eps) { doubt = true; break; }
        if (mid && !past) {
            if (xn >= 0.5f + eps) {
                for (int s = 0; s < S; ++s) Dcol[32 * s] = Ncol[32 * s];
                past = true;
            } else if (xn > 0.5f - eps) {
                doubt = true;
                break;
            }
        }
        // the first reaction whose cumulated propensity exceeds u2 a0
        const float target = (float)(((uint64_t)(rw.z >> 5) << 26) | (rw.w >> 6)) * 1.1102230246251565e-16f * a0;
        const float margin = (float)(22 + 2 * m) * e * a0;
        int mu = -1;
        float cum = 0.0f;
        for (uint32_t bits = poss; bits; bits &= bits - 1u) {
            const int r = __ffs(bits) - 1;
            cum += propensity_f(rx[r], Ncol, avf);
            if (target < cum - margin) { mu = r; break; }
            if (target <= cum + margin) break;
        }
        if (mu < 0) { doubt = true; break; }
        float dmax = 0.0f;
        for (uint32_t bits = rx[mu].y >> 16; bits; bits &= bits - 1u) {
            const int s = __ffs(bits) - 1;
            const int dn = mp.delta[mu][s];
            const int32_t n = Ncol[32 * s];
            if (n >= (1 << 20)) doubt = true;
            if (!((touched >> s) & 1u)) {
                scratch[32 * s] = (uint32_t)n;     // to undo
                if (!mid) Dcol[32 * s] = __float_as_int(0.0f);
                touched |= 1u << s;
            }
            if (!mid) Dcol[32 * s] = __float_as_int(__int_as_float(Dcol[32 * s]) + (float)dn * xn);
            Ncol[32 * s] = n + dn;
            pr.set(s, n + dn);
            dmax = fmaxf(dmax, fabsf((float)dn));
        }
        dsum += dmax;
        longest = 1e30f;
        x = xn;
        rw = rw_next;
        if (++k > kMaxEvents || dsum > (float)(kMoleculeCut - kDeferMin - 1)) doubt = true;
    }
    if (!doubt && touched) {
        const float eps = dsum * ((float)(30 + m + 3 * k) * e) + (4.0f * e + 9.5367431640625e-07f);
        for (uint32_t bits = touched; bits; bits &= bits - 1u) {
            const int s = __ffs(bits) - 1;
            if (mid) {
                if (!past) Dcol[32 * s] = Ncol[32 * s];
            } else if (mp.rule == kRuleMean) {
                rdd::Stream rs(v.seed, (uint32_t)key, v.period, rdd::kPurposeRounding, (uint32_t)s);
                const float w = __int_as_float(Dcol[32 * s]) + (float)rs.bits53() * 1.1102230246251565e-16f;
                const float fl = floorf(w);
                if (w - fl < eps || (fl + 1.0f) - w < eps) { doubt = true; break; }
                Dcol[32 * s] = Ncol[32 * s] - (int32_t)fl;
            }
        }
    }
    if (doubt) {
        for (uint32_t bits = touched; bits; bits &= bits - 1u) {
            const int s = __ffs(bits) - 1;
            Ncol[32 * s] = (int32_t)scratch[32 * s];
            pr.set(s, Ncol[32 * s]);
        }
        return kReactDoubt;
    }
    *touched_out = touched;
    return touched ? kReactDone : kReactNone;
}

// The same phase by the double-precision definition (Algorithm 1, Step 2 and
// 2.1: the first event at or past tau_k is discarded; before a species' count
// changes, its occupancy integral advances by N * (t_event - t_last); under
// the half-step rule N* is the count at tau_k / 2, that after every event
// before it), for a tet whose single-precision pass met a decision inside its
// error bound, or counts or event numbers beyond it.  Only reactions whose
// reactants are present are evaluated (the others add exact zeros), each rate
// constant once.  Returns the touched species, error bits in the upper half.
static __device__ __noinline__ uint32_t react_exact(const ModelParams& mp, int key, uint32_t period, double tau_k,
                                                    uint64_t seed, double vol_t, uint32_t on, int32_t* Ncol,
                                                    int32_t* Dcol, uint32_t* err) {
    const double avv = kAvogadro * (vol_t * 1000.0);
    const bool want_mid = mp.rule == kRuleMid;
    const double half = 0.5 * tau_k;
    const int S = mp.S;
    int64_t N[kMaxS], nmid[kMaxS];
    double occ[kMaxS], tl[kMaxS], c[kMaxR], a[kMaxR];
    for (int s = 0; s < S; ++s) {
        N[s] = Ncol[32 * s];
        occ[s] = 0.0;
        tl[s] = 0.0;
    }
    uint32_t touched = 0, bad = 0, have = 0;
    bool past_half = false;
    rdd::Stream st(seed, (uint32_t)key, period, rdd::kPurposeReaction, 0);
    double tc = 0.0;
    for (int events = 0;;) {
        uint32_t poss = on & mp.kpos;
        for (int s = 0; s < S; ++s) {
            if (N[s] <= 0) poss &= ~mp.needs[s];
            else if (N[s] == 1) poss &= ~mp.needs2[s];
        }
        if (!poss) break;                          // a0 = 0
        // propensity a_r = c_r h_r, h_r the number of reactant combinations
        double a0 = 0.0;
        for (uint32_t bits = poss; bits; bits &= bits - 1u) {
            const int r = __ffs(bits) - 1, a1 = mp.rs1[r], a2 = mp.rs2[r];
            if (!((have >> r) & 1u)) {
                const double kr = mp.k[r];
                const int o = mp.order[r];
                c[r] = o == 0 ? kr * avv : (o == 1 ? kr : kr / avv);
                have |= 1u << r;
            }
            int64_t h = 1;
            if (a1 >= 0) {
                if (a2 < 0) h = N[a1];
                else if (a1 == a2) h = N[a1] * (N[a1] - 1) / 2;
                else h = N[a1] * N[a2];
            }
            a[r] = c[r] * (double)h;
            a0 = a0 + a[r];
        }
        if (!(a0 > 0.0)) break;
        const double tn = tc + (-rdd::own_log(st.u01_open0())) / a0;
        if (tn >= tau_k) break;
        if (want_mid && !past_half && tn >= half) {
            for (int s = 0; s < S; ++s) nmid[s] = N[s];
            past_half = true;
        }
        const double target = st.u01() * a0;
        int mu = -1, positive = -1;
        double cum = 0.0;
        for (uint32_t bits = poss; bits; bits &= bits - 1u) {
            const int r = __ffs(bits) - 1;
            cum = cum + a[r];
            if (a[r] > 0.0) positive = r;
            if (target < cum) { mu = r; break; }
        }
        if (mu < 0) mu = positive;
        for (uint32_t bits = mp.rx[mu].y >> 16; bits; bits &= bits - 1u) {
            const int s = __ffs(bits) - 1;
            occ[s] = occ[s] + (double)N[s] * (tn - tl[s]);
            tl[s] = tn;
            touched |= 1u << s;
            N[s] += mp.delta[mu][s];
        }
        tc = tn;
        if (++events >= kEventCap) { atomicOr(err, kErrEventCap); break; }
    }
    if (want_mid && !past_half)
        for (int s = 0; s < S; ++s) nmid[s] = N[s];
    for (uint32_t bits = touched; bits; bits &= bits - 1u) {
        const int s = __ffs(bits) - 1;
        int64_t n = N[s], star = 0;
        if (want_mid) {
            star = nmid[s];
        } else {
            occ[s] = occ[s] + (double)N[s] * (tau_k - tl[s]);
            rdd::Stream rs(seed, (uint32_t)key, period, rdd::kPurposeRounding, (uint32_t)s);
            const double nbar = occ[s] / tau_k;
            const double fl = floor(nbar);
            star = (int64_t)fl + (rs.u01() < nbar - fl ? 1 : 0);
        }
        if (n < 0) { bad |= kErrNegative; n = 0; }
        if (n > 2147483647) { bad |= kErrOverflow; n = 2147483647; }
        if (star > 2147483647) star = 2147483647;
        Ncol[32 * s] = (int32_t)n;
        Dcol[32 * s] = (int32_t)star;
    }
    return touched | (bad << 16);
}

// Step 3 for N* >= kMoleculeCut: min(Binomial(N*, zeta), N) split over the
// faces by conditional binomials (double precision).
static __device__ __noinline__ int4 diffuse_binomial(const double* __restrict__ G, const double* __restrict__ gface,
                                                     int t, int key, int s, double Dsp, uint32_t period, double tau_k,
                                                     uint64_t seed, int64_t Nt, int64_t Nstar) {
    const double z = zeta_of(tau_k, Dsp, G[t]);
    int4 o = make_int4(0, 0, 0, 0);
    if (!(z > 0.0)) return o;
    rdd::Stream ds(seed, (uint32_t)key, period, rdd::kPurposeDiffusion, (uint32_t)s);
    int64_t n = rdd::binomial(Nstar, z, ds);
    if (n > Nt) n = Nt;
    if (n == 0) return o;
    double g[4], suf[4], acc = 0.0;
    for (int f = 0; f < 4; ++f) g[f] = gface[4 * (int64_t)t + f];
    for (int f = 3; f >= 0; --f) { acc = g[f] + acc; suf[f] = acc; }
    int last = -1;
    for (int f = 0; f < 4; ++f)
        if (g[f] > 0.0) last = f;
    int64_t rest = n, nf[4] = {0, 0, 0, 0};
    for (int f = 0; f < 4; ++f) {
        if (!(g[f] > 0.0)) continue;
        if (f == last) { nf[f] = rest; break; }
        const int64_t x = rdd::binomial(rest, g[f] / suf[f], ds);
        nf[f] = x;
        rest -= x;
    }
    return make_int4((int)nf[0], (int)nf[1], (int)nf[2], (int)nf[3]);
}

// The molecule-by-molecule draw that stops once all Nt molecules have left:
// only where N* exceeds the count and more than Nt of the N* draws leave.
__device__ __forceinline__ int4 draw_capped(uint64_t seed, uint32_t period, int key, int s, int32_t Nstar,
                                                int32_t Nt, uint4 C) {
    int4 o = make_int4(0, 0, 0, 0);
    rdd::Stream ds(seed, (uint32_t)key, period, rdd::kPurposeDiffusion, (uint32_t)s);
    int32_t moved = 0;
    for (int32_t i = 0; i < Nstar && moved < Nt; ++i) {
        const uint32_t u = ds.u32();
        if (rdd::below(u, C.x)) { o.x += 1; ++moved; }
        else if (rdd::below(u, C.y)) { o.y += 1; ++moved; }
        else if (rdd::below(u, C.z)) { o.z += 1; ++moved; }
        else if (rdd::below(u, C.w)) { o.w += 1; ++moved; }
    }
    return o;
}

// Leavers per face among the first m words of a Philox block, two 16-bit
// counts a word.  The thresholds are cumulative (C.x <= ... <= C.w), so
// a word is below C_f for every face from its own on: faces are counted by
// differences.  0xffffffff means "always".
__device__ __forceinline__ void count_block(const uint4& w, int m, const uint4& C, uint32_t& a0, uint32_t& a1) {
    const uint32_t u0 = w.x;
    const uint32_t u1 = m > 1 ? w.y : 0xffffffffu;
    const uint32_t u2 = m > 2 ? w.z : 0xffffffffu;
    const uint32_t u3 = m > 3 ? w.w : 0xffffffffu;
    if (min(min(u0, u1), min(u2, u3)) >= C.w && C.w != 0xffffffffu) return;
    auto under = [&](uint32_t c) -> uint32_t {
        const uint32_t n = (u0 < c) + (u1 < c) + (u2 < c) + (u3 < c);
        return c == 0xffffffffu ? (uint32_t)m : n;
    };
    const uint32_t nx = under(C.x), ny = under(C.y), nz = under(C.z), nw = under(C.w);
    a0 += nx | ((ny - nx) << 16);
    a1 += (nz - ny) | ((nw - nz) << 16);
}

// The diffusion draws of a warp's tets (Step 3; Eq. 2-3): every (lane,
// species) with molecules contributes ceil(n / 4) Philox blocks to one list;
// in each turn every lane adds its next block (of its next species when one is
// done), so neighbouring entries belong to different lanes, and 32 entries
// make a round with one block a lane.  The cost follows the number of blocks,
// not the largest count of a lane or the species present in any lane.
// Before the list, (kCalls) species with kMoleculeCut draws or more are drawn by
// big(sp, N*), and those with more than kCoopMin by the whole warp.  Returns the
// species whose acc words hold leavers-to-be.  All lanes must call it.  The per-lane loop
// with a whole-warp pass per species and tet from 10 molecules on took one
// serial pass a tet: 600 cycles each, up to 32 a warp.
// With one species (kOne) every lane draws its own first block, without the
// list, and only counts above four go on to it.  pre: the lane's thresholds
// of species 0, when kPre says that they are loaded.
template <bool kOne, bool kPre, bool kCalls, class Big>
__device__ __forceinline__ uint32_t draw_all(int S, int64_t T, const WarpMem& w, const PeriodView& v, int t, int key,
                                             uint32_t present, uint32_t many, uint32_t touched, uint4 pre, Big big) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const uint32_t k0 = (uint32_t)v.seed, k1 = (uint32_t)(v.seed >> 32);
    auto draws_of = [&](int sp) -> int {
        return ((touched >> sp) & 1u) ? w.D[32 * sp + lane] : w.N[32 * sp + lane];
    };
    // the species of each lane with draws of a usual number, and the others
    uint32_t heavy = present & many & 0xffffu;
    for (uint32_t bits = touched & present; bits; bits &= bits - 1u) {
        const int sp = __ffs(bits) - 1;
        const int n = w.D[32 * sp + lane];
        heavy = n > kCoopMin ? heavy | 1u << sp : heavy & ~(1u << sp);
        if (n <= 0) present &= ~(1u << sp);
    }
    uint32_t drawn = present & ~heavy;
    uint32_t todo = drawn;
    if (kCalls) {
        // the binomials of all lanes side by side, one species of each lane a
        // turn (one lane at a time, a mesh of 5,000 molecules a tet took up to
        // 14 times as long)
        uint32_t binom = 0;
        for (uint32_t bits = heavy; bits; bits &= bits - 1u) {
            const int sp = __ffs(bits) - 1;
            if (draws_of(sp) >= (int)kMoleculeCut) binom |= 1u << sp;
        }
        heavy &= ~binom;
        while (__ballot_sync(kAllLanes, binom != 0u)) {
            if (binom) {
                const int sp = __ffs(binom) - 1;
                binom &= binom - 1u;
                big(sp, draws_of(sp));
            }
            __syncwarp();
        }
    }
    for (;;) {
        const unsigned hm = __ballot_sync(kAllLanes, heavy != 0u);
        if (hm == 0u) break;
        const int src = __ffs(hm) - 1;
        const int sp_own = !kOne && heavy ? __ffs(heavy) - 1 : 0;
        const int sp = kOne ? 0 : __shfl_sync(kAllLanes, sp_own, src);
        const int nn = __shfl_sync(kAllLanes, heavy ? draws_of(sp_own) : 0, src);
        if (lane == src) heavy &= heavy - 1u;
        const int tt = __shfl_sync(kAllLanes, t, src), kk = __shfl_sync(kAllLanes, key, src);
        const uint4 C = __ldg(v.thr + ((int64_t)sp * T + tt) * v.thr_stride);
        uint32_t a0 = 0, a1 = 0;
        for (int blk = lane; 4 * blk < nn; blk += 32)
            count_block(rdd::philox_block((uint32_t)blk, (uint32_t)kk, v.period,
                                          (rdd::kPurposeDiffusion << 16) | (uint32_t)sp, k0, k1),
                        min(4, nn - 4 * blk), C, a0, a1);
        a0 = __reduce_add_sync(kAllLanes, a0);
        a1 = __reduce_add_sync(kAllLanes, a1);
        if (lane == src) {
            w.acc0[32 * sp + lane] = a0;
            w.acc1[32 * sp + lane] = a1;
            drawn |= 1u << sp;
        }
    }
    int sp = 0, n = 0, b = 0, nb = 0;
    if (kOne && todo) {
        n = draws_of(0);
        uint32_t a0 = 0, a1 = 0;
        const uint4 C = kPre ? pre : __ldg(v.thr + (int64_t)t * v.thr_stride);
        count_block(rdd::philox_block(0u, (uint32_t)key, v.period, rdd::kPurposeDiffusion << 16, k0, k1), min(4, n), C,
                    a0, a1);
        w.acc0[lane] = a0;
        w.acc1[lane] = a1;
        nb = (n + 3) >> 2;
        b = 1;
    }
    int cnt = 0;
    for (;;) {
        if (!kOne && b >= nb && todo) {
            sp = __ffs(todo) - 1;
            todo &= todo - 1u;
            n = draws_of(sp);
            nb = (n + 3) >> 2;
            b = 0;
            w.acc0[32 * sp + lane] = 0u;
            w.acc1[32 * sp + lane] = 0u;
        }
        const unsigned act = __ballot_sync(kAllLanes, b < nb);
        if (b < nb)
            w.list[cnt + __popc(act & lt)] =
                (uint32_t)lane | ((uint32_t)(min(4, n - 4 * b) - 1) << 5) | ((uint32_t)sp << 7) | ((uint32_t)b << 11);
        ++b;
        cnt += __popc(act);
        if (cnt >= 32 || (act == 0u && cnt > 0)) {
            // one round: the last min(32, cnt) entries, one a lane
            __syncwarp();
            const int take = min(cnt, 32);
            cnt -= take;
            const bool mine = lane < take;
            const uint32_t en = mine ? w.list[cnt + lane] : (uint32_t)lane;
            const int owner = (int)(en & 31u);
            const int tu = __shfl_sync(kAllLanes, t, owner), ku = __shfl_sync(kAllLanes, key, owner);
            if (mine) {
                const int su = kOne ? 0 : (int)((en >> 7) & 15u);
                const uint4 C = __ldg(v.thr + ((int64_t)su * T + tu) * v.thr_stride);
                uint32_t a0 = 0, a1 = 0;
                count_block(rdd::philox_block(en >> 11, (uint32_t)ku, v.period,
                                              (rdd::kPurposeDiffusion << 16) | (uint32_t)su, k0, k1),
                            (int)((en >> 5) & 3u) + 1, C, a0, a1);
                if (a0) atomicAdd(w.acc0 + 32 * su + owner, a0);
                if (a1) atomicAdd(w.acc1 + 32 * su + owner, a1);
            }
            __syncwarp();
        }
        if (act == 0u) break;
    }
    return drawn;
}

// Steps 2 and 3 for the warp's tets: column N of each live lane holds its
// counts and `pr` says which are not zero (all clear for a lane that is not
// live); mask: the tet's reaction mask.  After it N and pr hold what stays;
// emit(sp, o) was called by a lane for each species of which molecules leave
// (o: per face).  Bits of the species whose count changed are added to *dirty.
// Returns error bits.  All lanes must call it.
//
// kCalls = false leaves out what is rare and needs a function call (the
// double-precision repeat of a reaction phase, the binomial sampler): such a
// tet is left as it was and *deferred set; its lane goes through the form
// with kCalls afterwards (tried: its single-precision pass met a doubt
// before and is not repeated).  A call in the hot loop costs every turn of it: what
// lives across the call is spilled (80 to 100 local-memory instructions per 32
// tets with three calls inside).  With kDefer every tet whose first waiting
// time may fall inside the period is deferred, too.
// kLean: one species without reactions draws a warp's few molecules in registers.
template <bool kOne, bool kReact, bool kDefer, bool kCalls, bool kPre = false, bool kLean = false, class Emit>
__device__ __forceinline__ uint32_t warp_step(const DevMesh& m, const ModelParams& mp, int S, const WarpMem& w,
                                              const PeriodView& v, int t, bool live, uint32_t mask, Presence& pr,
                                              uint32_t* dirty, bool* deferred, uint32_t* err, Emit& emit,
                                              uint4 pre = make_uint4(0u, 0u, 0u, 0u), bool tried = false) {
    const int lane = threadIdx.x & 31;
    const int key = live ? key_of(m, t) : 0;
    uint32_t bad = 0, touched = 0;
    uint32_t present = pr.any & mp.moves;
    if (!kCalls && (pr.many >> 16)) *deferred = true;
    if (kReact) {
        const uint32_t on = mask & mp.kpos;
        const uint32_t poss = live && (kCalls || !*deferred) ? possible_by_presence(mp, pr, S, on) : 0u;
        // The lanes come from loops over their own inbox words: unless they are
        // brought together here, each goes through the reaction phase by itself
        // (10,368 tets of eleven species, up to 475 events a period, 60 periods: 82
        // ms instead of 42).
        if (__ballot_sync(kAllLanes, poss != 0u) && poss) {
            const float2 avf = __ldg(m.avv + t);
            if (kDefer) {
                // only the first waiting time, by its bound
                float a0 = 0.0f;
                for (uint32_t bits = poss; bits; bits &= bits - 1u)
                    a0 += propensity_f(w.rx[__ffs(bits) - 1], w.N + lane, avf);
                rdd::Stream st(v.seed, (uint32_t)key, v.period, rdd::kPurposeReaction, 0);
                const uint64_t y = 9007199254740991ull - st.bits53();
                const float need = a0 * v.tau_kf * 1.0001f * 1.0001f;
                *deferred = !(need < 3.0e38f) || !((float)(uint32_t)(y >> 29) * 5.9604644775390625e-08f >= need) ||
                            (y >> 29) == 0ull;
            } else {
                uint32_t tch = 0;
                int r = kReactDoubt;
                if (!kCalls || !tried)
                    r = react_fast(mp, w.rx, S, key, v, on, poss, avf, w.N + lane, w.D + lane, w.acc0 + lane, pr, &tch);
                if (r == kReactDoubt) {
                    if constexpr (kCalls) {
                        tch = react_exact(mp, key, v.period, v.tau_k, v.seed, m.vol[t], mask, w.N + lane, w.D + lane,
                                          err);
                        bad |= tch >> 16;
                        tch &= 0xffffu;
                        for (uint32_t bits = tch; bits; bits &= bits - 1u)
                            pr.set(__ffs(bits) - 1, w.N[32 * (__ffs(bits) - 1) + lane]);
                    } else {
                        *deferred = true;
                    }
                }
                *dirty |= tch;
                if (mp.rule != kRuleEnd) touched = tch;   // first order: the draw uses N(tau_k)
                present = pr.any & mp.moves;
            }
        }
    }
    if constexpr (kLean && kOne && !kReact && !kCalls) {
        // At most eight molecules in each tet: no list, no leavers in shared
        // memory (a point source in 279,936 tets, 2,000 periods: 16.2 -> 14.1 ms;
        // within one cluster it gains nothing and costs 1 %).
        const int32_t n = present ? w.N[lane] : 0;
        if (!__any_sync(kAllLanes, n > 8)) {
            if (n == 0) return 0u;
            const uint4 C = __ldg(v.thr + (int64_t)t * v.thr_stride);
            uint32_t a0 = 0, a1 = 0;
            for (int b = 0; 4 * b < n; ++b)
                count_block(rdd::philox_block((uint32_t)b, (uint32_t)key, v.period, rdd::kPurposeDiffusion << 16,
                                              (uint32_t)v.seed, (uint32_t)(v.seed >> 32)),
                            min(4, n - 4 * b), C, a0, a1);
            if (a0 | a1) {
                const int4 o = make_int4((int)(a0 & 0xffffu), (int)(a0 >> 16), (int)(a1 & 0xffffu), (int)(a1 >> 16));
                const int32_t left = n - (o.x + o.y + o.z + o.w);
                w.N[lane] = left;
                pr.set(0, left);
                *dirty |= 1u;
                emit(0, o);
            }
            return 0u;
        }
    }
    if (!kCalls && *deferred) present = 0u;
    const uint32_t drawn = draw_all<kOne, kPre, kCalls>(S, m.T, w, v, t, key, present, pr.many, touched, pre,
                                                        [&](int sp, int32_t star) {
        if constexpr (kCalls) {
            const int32_t Nt = w.N[32 * sp + lane];
            const int4 o = diffuse_binomial(m.G, m.g, t, key, sp, mp.D[sp], v.period, v.tau_k, v.seed, Nt, star);
            const int32_t all = o.x + o.y + o.z + o.w;
            if (all > 0) {
                w.N[32 * sp + lane] = Nt - all;
                pr.set(sp, Nt - all);
                *dirty |= 1u << sp;
                emit(sp, o);
            }
        }
    });
    for (uint32_t bits = drawn; bits; bits &= bits - 1u) {
        const int sp = __ffs(bits) - 1;
        const uint32_t a = w.acc0[32 * sp + lane], b = w.acc1[32 * sp + lane];
        if ((a | b) == 0u) continue;
        int4 o = make_int4((int)(a & 0xffffu), (int)(a >> 16), (int)(b & 0xffffu), (int)(b >> 16));
        const int32_t Nt = w.N[32 * sp + lane];
        if (o.x + o.y + o.z + o.w > Nt)
            o = draw_capped(v.seed, v.period, key, sp, w.D[32 * sp + lane], Nt,
                            __ldg(v.thr + ((int64_t)sp * m.T + t) * v.thr_stride));
        const int32_t left = Nt - (o.x + o.y + o.z + o.w);
        w.N[32 * sp + lane] = left;
        pr.set(sp, left);
        *dirty |= 1u << sp;
        emit(sp, o);
    }
    return bad;
}

}  // namespace rdk
