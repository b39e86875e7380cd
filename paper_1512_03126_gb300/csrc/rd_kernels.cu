// Kernels of the operator-splitting hot path (Algorithm 1 of
// arXiv:1512.03126) for sm_103a.
//
//   k_mesh_setup   face coefficients g = A/(V dist), G = sum g, reverse-face
//                  table, mesh validation, max G           (setup, Sec. II.A)
//   k_tau          tau = tau_scale / max_s(D_s * max_t G_t) (Algorithm 1, precompute)
//   k_thresholds   cumulative 32-bit face thresholds of zeta * w_f
//   k_count_ge     tets with G >= x (rank selection for the outlier option)
//   k_zeta_hist    histogram of zeta over the tets (diagnostic, Fig. 1d)
//   k_period       per tet: the previous period's transfers, SSA reactions
//                  with occupancy (Step 2), mean-corrected binomial count and
//                  multinomial split (Step 3); in one pass, or in two with
//                  the tets whose reactions have to run in the second
//   k_run          many periods in one cooperative launch, for a mesh whose
//                  tets are all resident at once
//   k_run_cluster  the same within one thread-block cluster, for small meshes
//   k_gather       the closing synchronous transfer of a run
//
// Layout: counts are species-major int32 [S][T] (coalesced), updated in
// place; transfers go through inboxes int32 [T][4][Sp]: a tet writes what
// leaves through face f into the neighbour's slot (a scattered store that
// nothing waits for) and reads its own four slots, contiguous, in the next
// period, instead of gathering from its neighbours.  Only what is not zero
// is written, and the reader clears it.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <mutex>
#include <utility>
#include <vector>

#include "rd_device.cuh"
#include "rd_internal.h"
#include "rd_period.cuh"
#include "rd_warp.cuh"

namespace rdk {

namespace {
std::atomic<int64_t> g_launches{0};
constexpr int kBlock = 256;

inline int grid_for(int64_t n) { return (int)((n + kBlock - 1) / kBlock); }

// The most that a block of kBlock threads asks for (k_period, k_run).
constexpr size_t block_shared_most(bool react) { return (size_t)(kBlock / 32) * warp_words(kMaxS, react) * sizeof(int32_t); }
// The most that a CTA of k_run_cluster may take.
constexpr size_t kClusterShared = 200u * 1024u;
}  // namespace

namespace {
// Sets an attribute of a kernel once on each device.
cudaError_t set_once(const void* kern, cudaFuncAttribute attr, int value) {
    static std::mutex mu;
    static std::vector<std::pair<std::pair<const void*, int>, int>> done;
    int dev = 0;
    cudaError_t ce = cudaGetDevice(&dev);
    if (ce != cudaSuccess) return ce;
    const auto what = std::make_pair(std::make_pair(kern, (int)attr), dev);
    std::lock_guard<std::mutex> lock(mu);
    if (std::find(done.begin(), done.end(), what) != done.end()) return cudaSuccess;
    ce = cudaFuncSetAttribute(kern, attr, value);
    if (ce == cudaSuccess) done.push_back(what);
    return ce;
}
}  // namespace

cudaError_t allow_shared(const void* kern, size_t bytes, size_t most) {
    if (bytes <= kDefaultShared) return cudaSuccess;
    return set_once(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}

int sm_count() {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
        cudaGetLastError();
        n = 1;
    }
    return n;
}

int64_t launches() { return g_launches.load(); }
void note_launch() { ++g_launches; }

// ---------------------------------------------------------------- setup ----
__global__ void k_mesh_setup(int32_t T, const int32_t* __restrict__ adj, const double* __restrict__ vol,
                             const double* __restrict__ area, const double* __restrict__ dist,
                             int4* __restrict__ src, double* __restrict__ g, double* __restrict__ G,
                             unsigned long long* gmax_bits, uint32_t* err) {
    // the block's largest G first: one atomic a tet on one address took 1.4 of
    // this kernel's 1.55 ms on 2.4 M tets
    __shared__ unsigned long long block_max;
    if (threadIdx.x == 0) block_max = 0ull;
    __syncthreads();
    const int t_ = blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = t_ < T;
    const int t = live ? t_ : T - 1;   // a lane past the end repeats the last tet, stores nothing
    uint32_t e = 0;
    double V = vol[t];
    if (!(V > 0.0) || !(V < HUGE_VAL)) e |= kErrVolume;
    int s4[4];
    double gf[4];
    double Gt = 0.0;
    for (int f = 0; f < 4; ++f) {
        int u = adj[4 * t + f];
        s4[f] = -1;
        gf[f] = 0.0;
        if (u >= 0) {
            if (u >= T || u == t) {
                e |= kErrAdjRange;
            } else {
                int slot = -1, hits = 0;
                for (int r = 0; r < 4; ++r)
                    if (adj[4 * u + r] == t) { slot = r; ++hits; }
                if (hits != 1) e |= kErrAdjAsym;
                else s4[f] = 4 * u + slot;
                double A = area[4 * t + f], d = dist[4 * t + f];
                if (!(A >= 0.0) || !(A < HUGE_VAL) || !(d > 0.0) || !(d < HUGE_VAL)) e |= kErrFace;
                else gf[f] = A / (V * d);
            }
        } else if (u != -1) {
            e |= kErrAdjRange;
        }
        Gt = Gt + gf[f];
    }
    if (live) {
        src[t] = make_int4(s4[0], s4[1], s4[2], s4[3]);
        for (int f = 0; f < 4; ++f) g[4 * t + f] = gf[f];
        G[t] = Gt;
        if (e) atomicOr(err, e);
    }
    // G >= 0: bit order is value order
    unsigned long long b = e == 0 && Gt < HUGE_VAL ? (unsigned long long)__double_as_longlong(Gt) : 0ull;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, b, d);
        b = o > b ? o : b;
    }
    if ((threadIdx.x & 31) == 0 && b) atomicMax(&block_max, b);
    __syncthreads();
    if (threadIdx.x == 0 && block_max) atomicMax(gmax_bits, block_max);
}

void launch_mesh_setup(int32_t T, const int32_t* adj, const double* vol, const double* area,
                       const double* dist, int4* src, double* g, double* G,
                       unsigned long long* gmax_bits, uint32_t* err, cudaStream_t st) {
    k_mesh_setup<<<grid_for(T), kBlock, 0, st>>>(T, adj, vol, area, dist, src, g, G, gmax_bits, err);
    ++g_launches;
}

// Rounding is monotone, so max_{s,t} fl(D_s G_t) = max_s fl(D_s max_t G_t).
__global__ void k_tau(const double* D, int32_t S, const unsigned long long* gmax_bits, double tau_scale,
                      double* tau_out) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    double Gmax = __longlong_as_double((long long)*gmax_bits);
    double dmax = 0.0;
    for (int s = 0; s < S; ++s) {
        double d = D[s] * Gmax;
        if (d > dmax) dmax = d;
    }
    *tau_out = dmax > 0.0 ? tau_scale / dmax : __longlong_as_double(0x7ff0000000000000ll);
}

void launch_tau(const double* D, int32_t S, const unsigned long long* gmax_bits, double tau_scale,
                double* tau_out, cudaStream_t st) {
    k_tau<<<1, 32, 0, st>>>(D, S, gmax_bits, tau_scale, tau_out);
    ++g_launches;
}

// Number of tets with G_t >= x (x given by its bit pattern; G >= 0, so bit
// order is value order): one step of the rank selection behind the outlier
// option of Sec. II.A.
__global__ void k_count_ge(int32_t T, const double* __restrict__ G, unsigned long long xbits, unsigned int* count) {
    unsigned int c = 0;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < T; t += gridDim.x * blockDim.x)
        c += (unsigned long long)__double_as_longlong(G[t]) >= xbits ? 1u : 0u;
    c = __reduce_add_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(count, c);
}

void launch_count_ge(int32_t T, const double* G, unsigned long long xbits, unsigned int* count, cudaStream_t st) {
    k_count_ge<<<std::min(grid_for(T), 1024), kBlock, 0, st>>>(T, G, xbits, count);
    ++g_launches;
}

// Histogram of zeta_t = min(1, tau * (D * G_t)) over the tets (Fig. 1d: the
// fastest species' zeta), bins of width 1/nbins on [0, 1] with zeta = 1 in the
// last; also the sum and the largest value (as bits; zeta >= 0).
__global__ void k_zeta_hist(int32_t T, const double* __restrict__ G, double tau, double D, int32_t nbins,
                            unsigned long long* counts, double* sum, unsigned long long* maxbits) {
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < T; t += gridDim.x * blockDim.x) {
        double z = tau * (D * G[t]);
        if (z > 1.0) z = 1.0;
        int b = (int)(z * (double)nbins);
        if (b >= nbins) b = nbins - 1;
        atomicAdd(counts + b, 1ull);
        atomicAdd(sum, z);
        atomicMax(maxbits, (unsigned long long)__double_as_longlong(z));
    }
}

void launch_zeta_hist(int32_t T, const double* G, double tau, double D, int32_t nbins, unsigned long long* counts,
                      double* sum, unsigned long long* maxbits, cudaStream_t st) {
    k_zeta_hist<<<std::min(grid_for(T), 1024), kBlock, 0, st>>>(T, G, tau, D, nbins, counts, sum, maxbits);
    ++g_launches;
}

// C_f = floor(2^32 zeta (g_0 + ... + g_f) / G): a molecule leaves through the
// first face f whose threshold exceeds its 32-bit draw, and stays if none does.
// By the definition's operations:
static __device__ __noinline__ uint4 thresholds_by_definition(double tau_k, double D, double Gt, const double* cum) {
    const double z = zeta_of(tau_k, D, Gt);
    uint32_t C[4] = {0, 0, 0, 0};
    if (z > 0.0)
        for (int f = 0; f < 4; ++f) C[f] = rdd::threshold_of(z * (cum[f] / Gt));
    return make_uint4(C[0], C[1], C[2], C[3]);
}

// A positive double as hi + lo in single precision: its first 24 bits and the
// 29 after them (lo rounded: off by at most 2^-24 of itself, 2^-48 of the
// value).  By integer operations, since FP64 conversions run at FP64 speed.
// hi is 0 or within (2^-100, 2^100), else *ok is cleared.
__device__ __forceinline__ float2 split_double(double x, bool* ok) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int ex = (int)(b >> 52) - 1023;
    if (b == 0ull) return make_float2(0.0f, 0.0f);
    *ok = *ok && ex > -100 && ex < 100;
    const uint32_t hi = ((uint32_t)(ex + 127) << 23) | ((uint32_t)(b >> 29) & 0x7fffffu);
    const float unit = __uint_as_float((uint32_t)(ex - 52 + 127 > 0 ? ex - 52 + 127 : 1) << 23);
    *ok = *ok && ex - 52 + 127 > 0;
    return make_float2(__uint_as_float(hi), (float)((uint32_t)b & 0x1fffffffu) * unit);
}

// One tet a thread, all species.  Below zeta = 1 the G's cancel: 2^32 zeta
// cum_f / G = (2^32 tau D) cum_f, in exact arithmetic; the definition's five
// roundings move it by at most 6 * 2^-53 of itself.  The product of the two
// factors' float pairs is off by at most 2^-45 of itself (2^-48 from each
// split, 2^-48 for the dropped lo lo, 3 * 2^-48 in the two sums), so by 2^-13
// at most: its floor is the definition's unless it lies within 2^-12 of a
// whole number.  Such a face (one in 2,048), and every tet whose zeta is not
// clearly below 1, takes the definition's operations.  2.4 M tets of 8 species
// (403 MB, 59 us at the copy rate): 2060 us with one thread a (species, tet)
// and FP64 divisions (64 cycles an FP64 operation, 562 a division), 467 with
// one FP64 product and conversion a face.
__global__ void k_thresholds(int32_t T, const __grid_constant__ ModelParams mp, const double* __restrict__ g,
                             const double* __restrict__ G, double tau_k, uint4* __restrict__ thr) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    const double2 g01 = reinterpret_cast<const double2*>(g)[2 * (int64_t)t];
    const double2 g23 = reinterpret_cast<const double2*>(g)[2 * (int64_t)t + 1];
    double cum[4];
    cum[0] = 0.0 + g01.x;
    cum[1] = cum[0] + g01.y;
    cum[2] = cum[1] + g23.x;
    cum[3] = cum[2] + g23.y;
    bool ok = true;
    float2 c[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) c[f] = split_double(cum[f], &ok);
    for (int s = 0; s < mp.S; ++s) {
        bool sure = ok;
        const float2 sc = split_double(tau_k * mp.D[s] * 4294967296.0, &sure);   // 2^32 tau D
        uint32_t C[4];
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            const float p = c[f].x * sc.x;
            const float r = __fmaf_rn(c[f].x, sc.y, __fmaf_rn(c[f].y, sc.x, __fmaf_rn(c[f].x, sc.x, -p)));
            const float whole = floorf(p);
            const float rest = (p - whole) + r;
            const float fl = floorf(rest);
            const float frac = rest - fl;
            sure = sure && p < 4294967296.0f * 0.999f && (p == 0.0f || (frac > 2.44140625e-4f && frac < 1.0f - 2.44140625e-4f));
            C[f] = (uint32_t)whole + (uint32_t)(int)fl;
        }
        uint4 v = make_uint4(C[0], C[1], C[2], C[3]);
        if (!sure) v = thresholds_by_definition(tau_k, mp.D[s], G[t], cum);
        thr[(int64_t)s * T + t] = v;
    }
}

void launch_thresholds(int32_t T, const ModelParams& mp, const double* g, const double* G, double tau_k,
                       uint4* thr, cudaStream_t st) {
    k_thresholds<<<grid_for(T), kBlock, 0, st>>>(T, mp, g, G, tau_k, thr);
    ++g_launches;
}

__global__ void k_pack_mask(int32_t T, int32_t R, const uint8_t* __restrict__ m8, uint32_t* __restrict__ m32,
                            const int32_t* __restrict__ perm) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    const int c = perm ? perm[t] : t;
    uint32_t bits = 0;
    for (int r = 0; r < R; ++r)
        if (m8[(size_t)r * T + c]) bits |= 1u << r;
    m32[t] = bits;
}

void launch_pack_mask(int32_t T, int32_t R, const uint8_t* mask8, uint32_t* mask32, const int32_t* perm,
                      cudaStream_t st) {
    k_pack_mask<<<grid_for(T), kBlock, 0, st>>>(T, R, mask8, mask32, perm);
    ++g_launches;
}

// Counts between the caller's canonical [T][S] order and the stored [S][T]
// (stored tet t is canonical tet perm[t], or t without a reordering).  A block
// takes 256 tets: species by species on the stored side, and the caller's
// side through shared memory so that both are contiguous (no alignment is
// asked of the caller's array).
__global__ void k_counts_in(int32_t T, int32_t S, const int32_t* __restrict__ ts, int32_t* __restrict__ sm,
                            uint32_t* err, const int32_t* __restrict__ perm) {
    extern __shared__ int32_t tile[];   // [256][S + 1 - S % 2]: an odd stride, free of bank conflicts
    const int ld = S | 1;
    const int64_t t0 = (int64_t)blockIdx.x * kBlock;
    const int n = (int)min((int64_t)kBlock, T - t0);
    if (!perm) {
        for (int i = threadIdx.x; i < n * S; i += kBlock) {
            const int r = i / S;
            tile[r * ld + (i - r * S)] = ts[t0 * S + i];
        }
        __syncthreads();
    }
    const int r = threadIdx.x;
    if (r >= n) return;
    const int64_t c = perm ? perm[t0 + r] : 0;
    uint32_t bad = 0;
    for (int s = 0; s < S; ++s) {
        int32_t v = perm ? ts[c * S + s] : tile[r * ld + s];
        if (v < 0) { bad |= kErrNegative; v = 0; }
        sm[(int64_t)s * T + t0 + r] = v;
    }
    if (bad) atomicOr(err, bad);
}

__global__ void k_counts_out(int32_t T, int32_t S, const int32_t* __restrict__ sm, int32_t* __restrict__ ts,
                             const int32_t* __restrict__ perm, const uint32_t* __restrict__ err) {
    extern __shared__ int32_t tile[];
    if (err && ((err[0] & kErrTimeout) || err[1])) return;   // gave up, or left early
    const int ld = S | 1;
    const int64_t t0 = (int64_t)blockIdx.x * kBlock;
    const int n = (int)min((int64_t)kBlock, T - t0);
    const int r = threadIdx.x;
    if (r < n) {
        const int64_t c = perm ? perm[t0 + r] : 0;
        for (int s = 0; s < S; ++s) {
            const int32_t v = sm[(int64_t)s * T + t0 + r];
            if (perm) ts[c * S + s] = v;
            else tile[r * ld + s] = v;
        }
    }
    if (perm) return;
    __syncthreads();
    for (int i = threadIdx.x; i < n * S; i += kBlock) {
        const int q = i / S;
        ts[t0 * S + i] = tile[q * ld + (i - q * S)];
    }
}

void launch_counts_in(int32_t T, int32_t S, const int32_t* ts, int32_t* sm, uint32_t* err, const int32_t* perm,
                      cudaStream_t st) {
    k_counts_in<<<grid_for(T), kBlock, kBlock * (S | 1) * sizeof(int32_t), st>>>(T, S, ts, sm, err, perm);
    ++g_launches;
}

void launch_counts_out(int32_t T, int32_t S, const int32_t* sm, int32_t* ts, const int32_t* perm, const uint32_t* err,
                       cudaStream_t st) {
    k_counts_out<<<grid_for(T), kBlock, kBlock * (S | 1) * sizeof(int32_t), st>>>(T, S, sm, ts, perm, err);
    ++g_launches;
}

// ---------------------------------------------------------------- period ---
void finish_model_params(ModelParams& mp) {
    mp.kpos = 0;
    mp.moves = 0;
    for (int s = 0; s < mp.S; ++s)
        if (mp.D[s] > 0.0) mp.moves |= 1u << s;
    for (int s = 0; s < kMaxS; ++s) mp.needs[s] = mp.needs2[s] = 0u;
    for (int r = 0; r < mp.R; ++r) {
        mp.rs1[r] = mp.rs2[r] = -1;
        for (int s = 0; s < mp.S; ++s) {
            if (mp.lhs[r][s] == 2) { mp.rs1[r] = mp.rs2[r] = (int8_t)s; }
            else if (mp.lhs[r][s] == 1) {
                if (mp.rs1[r] < 0) mp.rs1[r] = (int8_t)s;
                else mp.rs2[r] = (int8_t)s;
            }
        }
        mp.kf[r] = (float)mp.k[r];
        if (mp.k[r] > 0.0) mp.kpos |= 1u << r;
        for (int s = 0; s < mp.S; ++s) {
            if (mp.lhs[r][s] >= 1) mp.needs[s] |= 1u << r;
            if (mp.lhs[r][s] >= 2) mp.needs2[s] |= 1u << r;
        }
        uint32_t changed = 0;
        for (int s = 0; s < mp.S; ++s) changed |= mp.delta[r][s] != 0 ? 1u << s : 0u;
        const int a = mp.rs1[r], b = mp.rs2[r];
        const uint32_t kind = a < 0 ? 0u : (b < 0 ? 1u : (a == b ? 3u : 2u));
        std::memcpy(&mp.rx[r].x, &mp.kf[r], sizeof(float));
        mp.rx[r].y = (uint32_t)std::max(a, 0) | (uint32_t)std::max(b, 0) << 4 | kind << 8 | changed << 16;
    }
}

__global__ void k_avv(int32_t T, const double* __restrict__ vol, float2* __restrict__ avv) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    double a = kAvogadro * (vol[t] * 1000.0);
    avv[t] = make_float2((float)a, (float)(1.0 / a));
}

void launch_avv(int32_t T, const double* vol, float2* avv, cudaStream_t st) {
    k_avv<<<grid_for(T), kBlock, 0, st>>>(T, vol, avv);
    ++g_launches;
}

// A tet's molecules that arrived in the previous period, added to its column
// (clamped at 2^31-1), and its inbox words cleared for their next use.  Up to
// two species a nonzero word is the message; from three on a byte (16 bits
// from nine species on) a face says which species' words are valid, so a tet
// reads 4 or 8 bytes unless something came: 256 of the 356 bytes a
// tet-period of eight species moved were inbox words, nearly all zero.
// Returns error bits.  first: the words of one species, if the caller has loaded
// them (kLoaded).
template <bool kLoaded = false>
__device__ __forceinline__ uint32_t take_inbox(const PeriodArgs& a, int t, int S, int lane, int32_t* N,
                                               Presence& pr, uint32_t* dirty, int4 first = make_int4(0, 0, 0, 0)) {
    const int Sp = inbox_stride(S);
    uint32_t bad = 0;
    auto add = [&](int sp, int64_t v) {
        int64_t n = N[32 * sp + lane] + v;
        if (n > 2147483647) { bad |= kErrOverflow; n = 2147483647; }
        if (n < 0) { bad |= kErrNegative; n = 0; }
        N[32 * sp + lane] = (int32_t)n;
        pr.set(sp, (int32_t)n);
        *dirty |= 1u << sp;
    };
    if (S <= 2) {
        int4* p = reinterpret_cast<int4*>(a.in_prev + (int64_t)t * 4 * Sp);
        const int4 x = kLoaded ? first : __ldcg(p);
        int4 y = make_int4(0, 0, 0, 0);
        if (S == 2) y = __ldcg(p + 1);
        if (x.x | x.y | x.z | x.w) {
            *p = make_int4(0, 0, 0, 0);
            if (S == 1) add(0, (int64_t)x.x + x.y + x.z + x.w);
        }
        if (S == 2) {
            if (y.x | y.y | y.z | y.w) p[1] = make_int4(0, 0, 0, 0);
            if (x.x | x.z | y.x | y.z) add(0, (int64_t)x.x + x.z + y.x + y.z);
            if (x.y | x.w | y.y | y.w) add(1, (int64_t)x.y + x.w + y.y + y.w);
        }
        return bad;
    }
    uint64_t bits;
    if (S <= 8) {
        uint32_t* p = reinterpret_cast<uint32_t*>(a.mask_prev) + t;
        bits = __ldcg(p);
        if (bits) *p = 0u;
    } else {
        unsigned long long* p = reinterpret_cast<unsigned long long*>(a.mask_prev) + t;
        bits = __ldcg(p);
        if (bits) *p = 0ull;
    }
    const int shift = S <= 8 ? 3 : 4;   // log2 of the bits a face
    while (bits) {
        const int i = __ffsll((long long)bits) - 1;
        bits &= bits - 1ull;
        const int f = i >> shift, sp = i & ((1 << shift) - 1);
        add(sp, __ldcg(a.in_prev + ((int64_t)t * 4 + f) * Sp + sp));
    }
    return bad;
}

// What a tet's emit writes: leavers into its neighbours' inbox words, and
// the valid bits of each face's slot at the end (one writer a slot).
struct Sender {
    const PeriodArgs& a;
    const int4* src;
    int t, S;
    int4 sr;
    bool have;
    uint64_t bits;

    __device__ __forceinline__ Sender(const PeriodArgs& a_, const int4* src_, int t_, int S_)
        : a(a_), src(src_), t(t_), S(S_), sr(make_int4(-1, -1, -1, -1)), have(false), bits(0) {}

    __device__ __forceinline__ void load() {
        if (!have) sr = __ldg(src + t);
        have = true;
    }
    // Partitioned runs export slots of tets the rank never reads (and so
    // never clears): there every slot is written in full.
    __device__ __forceinline__ void clear_all() {
        load();
        const int slot[4] = {sr.x, sr.y, sr.z, sr.w};
        if (S <= 2)
            for (int f = 0; f < 4; ++f)
                if (slot[f] >= 0)
                    for (int s = 0; s < S; ++s) a.in_cur[(int64_t)slot[f] * S + s] = 0;
    }
    __device__ __forceinline__ void operator()(int sp, const int4& o) {
        load();
        const int slot[4] = {sr.x, sr.y, sr.z, sr.w}, n[4] = {o.x, o.y, o.z, o.w};
        const int Sp = inbox_stride(S);
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            if (n[f] <= 0 || slot[f] < 0) continue;
            a.in_cur[(int64_t)slot[f] * Sp + sp] = n[f];
            bits |= 1ull << (16 * f + sp);
        }
    }
    __device__ __forceinline__ void finish(bool all) {
        if (S <= 2 || (!all && bits == 0)) return;
        const int slot[4] = {sr.x, sr.y, sr.z, sr.w};
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            const uint32_t b = (uint32_t)(bits >> (16 * f)) & 0xffffu;
            if (slot[f] < 0 || (!all && b == 0u)) continue;
            if (S <= 8) a.mask_cur[slot[f]] = (uint8_t)b;
            else reinterpret_cast<uint16_t*>(a.mask_cur)[slot[f]] = (uint16_t)b;
        }
    }
};

// The deferred tets of a warp (warp_step without calls), one a lane, with the
// double-precision samplers: rare, and kept out of line so that the kernels'
// registers and loops are free of them.  Returns the species whose count
// changed, error bits in the upper half.
template <bool kReact>
static __device__ __noinline__ uint32_t step_deferred(const DevMesh& m, const ModelParams& mp, int32_t* column0,
                                                      const uint2* rx, uint32_t period, double tau_k, uint64_t seed,
                                                      const uint4* thr, int32_t* in_cur, uint8_t* mask_cur, int t,
                                                      bool live, bool tried, bool dense, uint32_t* err) {
    const int S = mp.S, lane = threadIdx.x & 31;
    const WarpMem w(column0, S, kReact, rx);
    const PeriodView v{period, tau_k, (float)tau_k, seed, thr, 1};
    PeriodArgs a{};
    a.in_cur = in_cur;
    a.mask_cur = mask_cur;
    Presence pr;
    if (live) pr = presence_of(w.N + lane, S);
    const uint32_t mask = kReact && mp.has_mask && live ? __ldg(m.mask + t) : 0xffffffffu;
    Sender send(a, m.src, t, S);
    if (live && dense) send.load();
    uint32_t dirty = 0;
    bool none = false;
    const uint32_t bad = warp_step<false, kReact, false, true>(m, mp, S, w, v, t, live, mask, pr, &dirty, &none, err, send,
                                                               make_uint4(0u, 0u, 0u, 0u), tried);
    if (live) send.finish(dense);
    return (live ? dirty : 0u) | (bad << 16);
}

// Passes of a period: all in one kernel, or a first pass that defers the tets
// whose reaction phase has to run to a queue and a second one over the queue.
enum { kPassAll = 0, kPassFirst = 1, kPassQueue = 2 };

// One period for every tet, one a lane: the previous period's transfers, the
// reaction phase, the diffusion draws, leavers pushed to the neighbours'
// inboxes (rd_warp.cuh).  Counts stay in place in cnt (only their own
// tet reads or writes them) and are written back where they changed.
// S_ > 0 fixes the species count at compile time.  Four blocks an SM (64
// registers): 2.4 M-tet bar, 24 periods, 3.36 ms, with 3 blocks 4.00 and 5 blocks
// 3.75; one species, 384,000-tet cube, 100 periods, 1.80, with 3 blocks 1.84, 2
// blocks 1.86.  One species loads its inbox words beside the count, and the
// reverse faces beside the thresholds where it holds molecules, instead of one
// after the other (162,000 tets of one molecule, 100 periods: 0.84 -> 0.66 ms; for
// several species the words held in registers cost the bar 18 %).
template <int S_, bool kReact, int kPass>
__global__ void __launch_bounds__(kBlock, 4)
k_period(const __grid_constant__ DevMesh m, const __grid_constant__ ModelParams mp, DevState s,
         const __grid_constant__ PeriodArgs a, int32_t* __restrict__ queue, int32_t* qcount, int32_t parity) {
    extern __shared__ int32_t sm[];
    const int S = S_ > 0 ? S_ : mp.S;
    const int lane = threadIdx.x & 31;
    __shared__ uint2 rx[kReact ? kMaxR : 1];
    const WarpMem w(sm + (threadIdx.x >> 5) * warp_words(S, kReact), S, kReact, rx);
    if (kReact) {
        if (threadIdx.x < kMaxR) rx[threadIdx.x] = mp.rx[threadIdx.x];
        __syncthreads();
    }
    const int64_t T = m.T;
    const PeriodView v{a.period, a.tau_k, a.tau_kf, a.seed, a.thr, 1};
    const int hi = kPass == kPassQueue ? qcount[parity] : (a.t_hi > 0 ? a.t_hi : m.T);
    const int lo = kPass == kPassQueue ? 0 : a.t_lo;
    if (kPass == kPassFirst && blockIdx.x == 0 && threadIdx.x == 0) qcount[parity ^ 1] = 0;
    for (int64_t base = lo + (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < hi;
         base += (int64_t)gridDim.x * blockDim.x) {
        bool live = base + lane < hi;
        const int t = !live ? 0 : (kPass == kPassQueue ? queue[base + lane] : (int)(base + lane));
        uint32_t bad = 0, dirty = 0;
        Presence pr;
        const uint32_t mask = kReact && mp.has_mask && live ? __ldg(m.mask + t) : 0xffffffffu;
        if (live) {
            int4 words = make_int4(0, 0, 0, 0);
            if (S_ == 1 && kPass != kPassQueue && !a.first) words = __ldcg(reinterpret_cast<const int4*>(a.in_prev) + t);
            for (int s0 = 0; s0 < S; s0 += 8) {
                int32_t n[8];
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (s0 + k < S) n[k] = s.cnt[(int64_t)(s0 + k) * T + t];
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (s0 + k < S) {
                        w.N[32 * (s0 + k) + lane] = n[k];
                        pr.add(s0 + k, n[k]);
                    }
            }
            if (kPass != kPassQueue && !a.first) bad |= take_inbox<S_ == 1>(a, t, S, lane, w.N, pr, &dirty, words);
        }
        Sender send(a, m.src, t, S);
        if (S_ == 1 && !kReact && pr.any) send.load();   // beside the thresholds
        if (a.dense && live) send.clear_all();
        bool deferred = false;
        if (kPass == kPassQueue) {
            deferred = live;
        } else {
            bad |= warp_step<S_ == 1, kReact, kPass == kPassFirst, false, false, true>(m, mp, S, w, v, t, live, mask, pr,
                                                                                       &dirty, &deferred, s.err, send);
            if (live && !deferred) send.finish(a.dense != 0);
        }
        if (kPass != kPassFirst && __ballot_sync(0xffffffffu, deferred)) {
            const uint32_t x = step_deferred<kReact>(m, mp, w.N, w.rx, a.period, a.tau_k, a.seed, a.thr, a.in_cur,
                                                     a.mask_cur, t, deferred, kPass == kPassAll && (pr.many >> 16) == 0u,
                                                     a.dense != 0, s.err);
            dirty |= x & 0xffffu;
            bad |= x >> 16;
        }
        if (kPass == kPassFirst) {
            const unsigned dm = __ballot_sync(0xffffffffu, deferred);
            if (dm) {
                const int leader = __ffs(dm) - 1;
                int at = 0;
                if (lane == leader) at = atomicAdd(qcount + parity, __popc(dm));
                at = __shfl_sync(0xffffffffu, at, leader);
                if (deferred) queue[at + __popc(dm & ((1u << lane) - 1u))] = t;
            }
        }
        if (live)
            for (uint32_t bits = dirty; bits; bits &= bits - 1u) {
                const int sp = __ffs(bits) - 1;
                s.cnt[(int64_t)sp * T + t] = w.N[32 * sp + lane];
            }
        if (bad) atomicOr(s.err, bad);
        __syncwarp();
    }
}

// Grid barrier of a cooperative launch: the counter only grows, by one per
// block and barrier; the wait ends when it reaches `target` (modulo 2^32).
// The launch holds every block resident, so the wait is as long as the slowest
// block's period, which can be minutes (see longest_period_ns).  Past the limit
// the block sets kErrTimeout and gives up, and the others follow it.
__device__ __forceinline__ bool grid_barrier(uint32_t* counter, uint32_t target, uint32_t* err,
                                             unsigned long long limit_ns, volatile int* gave_up) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();   // the block's inbox words before its arrival
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(counter) : "memory");
        unsigned long long start = 0ull;
        for (uint32_t i = 1;; ++i) {
            uint32_t c;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(counter) : "memory");
            if ((int32_t)(c - target) >= 0) break;
            if ((i & 1023u) == 0u) {
                unsigned long long now;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
                if (start == 0ull) start = now;
                if (now - start > limit_ns || (__ldcg(err) & kErrTimeout)) {
                    atomicOr(err, kErrTimeout);
                    *gave_up = 1;
                    break;
                }
            }
        }
    }
    __syncthreads();
    return *gave_up == 0;
}

// A stretch of periods in one launch, for a mesh whose tets are all resident
// at once (one lane each): counts stay in shared memory, the code, the
// thresholds and the neighbour records in the SM's caches, and a grid barrier
// takes the place of the launch between two periods.  Started alone, a
// period of a small mesh is mostly cold instruction and constant fetches
// (48,000-tet A/B/C cube, 48 periods: 0.63 ms one launch a period, 0.42 here).
// Ends with the closing transfer, all inbox words and masks cleared.
template <int S_, bool kReact, int kBlocks>
__global__ void __launch_bounds__(kBlock, kBlocks)
k_run(const __grid_constant__ DevMesh m, const __grid_constant__ ModelParams mp, DevState s,
      const __grid_constant__ RunArgs r) {
    extern __shared__ int32_t sm[];
    if (r.left && __ldcg(r.left)) return;   // queued behind a launch that left early
    __shared__ int gave_up;
    const int S = S_ > 0 ? S_ : mp.S;
    const int lane = threadIdx.x & 31;
    __shared__ uint2 rx[kReact ? kMaxR : 1];
    const WarpMem w(sm + (threadIdx.x >> 5) * warp_words(S, kReact), S, kReact, rx);
    if (kReact) {
        if (threadIdx.x < kMaxR) rx[threadIdx.x] = mp.rx[threadIdx.x];
        __syncthreads();
    }
    const int64_t T = m.T;
    const int64_t tt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = tt < T;
    const int t = live ? (int)tt : 0;
    if (threadIdx.x == 0) gave_up = 0;
    Presence pr;
    const uint32_t mask = kReact && mp.has_mask && live ? __ldg(m.mask + t) : 0xffffffffu;
    if (live)
        for (int sp = 0; sp < S; ++sp) {
            const int32_t n = s.cnt[sp * T + t];
            w.N[32 * sp + lane] = n;
            pr.add(sp, n);
            if (r.save) r.save[sp * T + t] = n;
        }
    uint32_t bad = 0, dirty = 0, target = r.barrier_base;
    for (int q = 0; q <= r.periods; ++q) {
        PeriodArgs a{};
        const int p = q & 1;
        a.in_prev = r.inbox[p ^ 1];
        a.in_cur = r.inbox[p];
        a.mask_prev = r.mask[p ^ 1];
        a.mask_cur = r.mask[p];
        if (q > 0) {
            target += gridDim.x;
            if (!grid_barrier(r.barrier, target, s.err, r.wait_limit_ns, &gave_up)) return;
            if (live) bad |= take_inbox(a, t, S, lane, w.N, pr, &dirty);
        }
        if (q == r.periods) break;
        const bool last = r.last_short && q == r.periods - 1;
        const PeriodView v{r.period0 + (uint32_t)q, last ? r.tau_last : r.tau, last ? r.tau_lastf : r.tauf, r.seed,
                           last ? r.thr_last : r.thr, 1};
        Sender send(a, m.src, t, S);
        bool deferred = false;
        bad |= warp_step<S_ == 1, kReact, false, false, false, true>(m, mp, S, w, v, t, live, mask, pr, &dirty, &deferred,
                                                                     s.err, send);
        if (live && !deferred) send.finish(false);
        if (__ballot_sync(0xffffffffu, deferred)) {
            const uint32_t x = step_deferred<kReact>(m, mp, w.N, w.rx, v.period, v.tau_k, v.seed, v.thr, a.in_cur,
                                                     a.mask_cur, t, deferred, (pr.many >> 16) == 0u, false, s.err);
            dirty |= x & 0xffffu;
            bad |= x >> 16;
            if (deferred) pr = presence_of(w.N + lane, S);
        }
    }
    if (live)
        for (uint32_t bits = dirty; bits; bits &= bits - 1u) {
            const int sp = __ffs(bits) - 1;
            s.cnt[sp * T + t] = w.N[32 * sp + lane];
        }
    if (bad) atomicOr(s.err, bad);
}

// The same for a mesh that one thread-block cluster holds: inboxes and masks
// live in the cluster's shared memory, leavers are stores into the neighbour
// tet's CTA, and the hardware cluster barrier takes the place of the grid
// barrier, its memory fence and the polling of a counter in L2 (3 to 4 us of a
// period together).
__device__ __forceinline__ uint32_t map_to_cta(uint32_t addr, uint32_t cta) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(cta));
    return r;
}

__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// Leavers into the words of neighbours' slots; face f's slot is number
// slot & 0xfff of CTA slot >> 12 (none: 0xffffffff).
struct ClusterSender {
    uint32_t slot[4];
    uint32_t words, masks;      // shared addresses of this parity's words and masks
    int S;
    uint64_t bits;

    __device__ __forceinline__ void operator()(int sp, const int4& o) {
        const int n[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            if (n[f] <= 0 || slot[f] == 0xffffffffu) continue;
            asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(
                             map_to_cta(words + ((slot[f] & 0xfffu) * S + sp) * 4u, slot[f] >> 12)), "r"(n[f]) : "memory");
            bits |= 1ull << (16 * f + sp);
        }
    }
    __device__ __forceinline__ void finish() {
        if (S <= 2 || bits == 0) return;
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            const uint32_t b = (uint32_t)(bits >> (16 * f)) & 0xffffu;
            if (b == 0u || slot[f] == 0xffffffffu) continue;
            asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(
                             map_to_cta(masks + (slot[f] & 0xfffu) * 2u, slot[f] >> 12)), "h"((uint16_t)b) : "memory");
        }
    }
};

// At most 16 multiprocessors hold the mesh.  Where most tets need the
// double-precision samplers their FP64 units set the period, and the whole
// device would share that work: a warp that left kLeaveLanes or more of its tets
// to them asks all CTAs to leave after the period, and the caller goes on with
// the mesh spread over the device (k_run) for a while.  7,986 tets of 5,000
// molecules, 12 periods: 6.9 ms within the cluster, 2.7 so.  Up to four
// warps a CTA the FP64 units of 16 multiprocessors serve as well, and with many
// reactions, most of whose work is not theirs, up to eight: RunArgs::left is null
// there (2 reactions, 6 warps a CTA, 100 events: 17.2 ms within the cluster, 14.3
// spread; 30 reactions of eleven species, 7 warps: 36.9 and 40.5; 21 of eight, 12
// warps: 114 and 96).
constexpr int kLeaveLanes = 16;
inline int leave_above_warps(const ModelParams& mp) { return mp.any_reaction && mp.R + mp.S > 8 ? 8 : 4; }

template <bool kReact>
static __device__ __noinline__ uint32_t step_deferred_in_cluster(const DevMesh& m, const ModelParams& mp,
                                                                 int32_t* column0, const uint2* rx, uint32_t period,
                                                                 double tau_k, uint64_t seed, const uint4* thr,
                                                                 uint4 slot, uint32_t words, uint32_t masks, int t,
                                                                 bool live, bool tried, uint32_t* err,
                                                                 uint32_t stop_at, uint32_t after) {
    const int S = mp.S, lane = threadIdx.x & 31;
    const WarpMem w(column0, S, kReact, rx);
    const PeriodView v{period, tau_k, (float)tau_k, seed, thr, 1};
    Presence pr;
    if (live) pr = presence_of(w.N + lane, S);
    const uint32_t mask = kReact && mp.has_mask && live ? __ldg(m.mask + t) : 0xffffffffu;
    ClusterSender send{{slot.x, slot.y, slot.z, slot.w}, words, masks, S, 0};
    uint32_t dirty = 0;
    bool none = false;
    const uint32_t bad = warp_step<false, kReact, false, true>(m, mp, S, w, v, t, live, mask, pr, &dirty, &none, err, send,
                                                               make_uint4(0u, 0u, 0u, 0u), tried);
    if (live) send.finish();
    if (stop_at != 0u && __popc(__ballot_sync(kAllLanes, live)) >= kLeaveLanes && lane < (int)gridDim.x)
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(map_to_cta(stop_at, (uint32_t)lane)), "r"(after) : "memory");
    return (live ? dirty : 0u) | (bad << 16);
}

// Dynamic shared memory of a CTA of `warps` warps, in words: the warps'
// (rd_warp.cuh), then per tet two parities of four slots of S words and of
// four 16-bit masks, and a word that says when to leave.
__host__ __device__ inline int cluster_words(int S, bool react, int warps) {
    return warps * warp_words(S, react) + 32 * warps * (8 * S + 4) + 4;
}

template <int S_, bool kReact>
__global__ void __launch_bounds__(512, 1)
k_run_cluster(const __grid_constant__ DevMesh m, const __grid_constant__ ModelParams mp, DevState s,
              const __grid_constant__ RunArgs r) {
    extern __shared__ __align__(16) int32_t sm[];
    if (r.left && __ldcg(r.left)) return;   // queued behind a launch that left early
    const int S = S_ > 0 ? S_ : mp.S;
    const int lane = threadIdx.x & 31;
    const int warps = blockDim.x >> 5, B = blockDim.x;
    __shared__ uint2 rx[kReact ? kMaxR : 1];
    const WarpMem w(sm + (threadIdx.x >> 5) * warp_words(S, kReact), S, kReact, rx);
    if (kReact)
        for (int i = threadIdx.x; i < kMaxR; i += B) rx[i] = mp.rx[i];
    int32_t* words = sm + warps * warp_words(S, kReact);                      // [2][B][4][S]
    unsigned long long* masks = reinterpret_cast<unsigned long long*>(words + 8 * S * B);   // [2][B]
    for (int i = threadIdx.x; i < 8 * S * B; i += B) words[i] = 0;
    for (int i = threadIdx.x; i < 2 * B + 1; i += B) masks[i] = 0ull;   // and the word to leave
    // Warp w of the cluster's W takes tets w, w + W, w + 2 W, ...: a compact
    // cloud's crowded tets go to different warps (a warp's 32 consecutive tets
    // around a point source made all others wait: 3,072-tet cube 4.7 us a
    // period).
    const int64_t T = m.T;
    const int W = gridDim.x * warps;
    const int64_t tt = (int64_t)lane * W + blockIdx.x * warps + (threadIdx.x >> 5);
    const bool live = tt < T;
    const int t = live ? (int)tt : 0;
    Presence pr;
    const uint32_t mask = kReact && mp.has_mask && live ? __ldg(m.mask + t) : 0xffffffffu;
    ClusterSender send;
    send.S = S;
    {
        const int4 sr = live ? __ldg(m.src + t) : make_int4(-1, -1, -1, -1);
        const int f4[4] = {sr.x, sr.y, sr.z, sr.w};
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            send.slot[f] = 0xffffffffu;
            if (f4[f] < 0) continue;
            const int u = f4[f] >> 2, wu = u % W;   // its warp, and thread of the CTA
            send.slot[f] = (uint32_t)(wu / warps) << 12 | (uint32_t)(((wu % warps) * 32 + u / W) * 4 + (f4[f] & 3));
        }
    }
    if (live)
        for (int sp = 0; sp < S; ++sp) {
            const int32_t n = s.cnt[sp * T + t];
            w.N[32 * sp + lane] = n;
            pr.add(sp, n);
        }
    uint32_t bad = 0, dirty = 0;
    cluster_sync_all();   // every CTA's words and masks are zero
    const uint32_t words_at = (uint32_t)__cvta_generic_to_shared(words);
    const uint32_t masks_at = (uint32_t)__cvta_generic_to_shared(masks);
    const uint32_t stop_at = masks_at + (uint32_t)(B * 16);   // the period after which a warp asked to leave, plus 1
    int end = r.periods;
    for (int q = 0; q <= r.periods; ++q) {
        const int p = q & 1;
        if (q > 0) {
            cluster_sync_all();
            // all CTAs agree: a request made in period q - 1 reads q, nobody starts
            // period q before all have finished that, and one made in it reads q + 1
            uint32_t asked;
            asm volatile("ld.shared.u32 %0, [%1];" : "=r"(asked) : "r"(stop_at) : "memory");
            if (asked == (uint32_t)q) end = q;
            if (live) {
                auto add = [&](int sp, int64_t v) {
                    int64_t n = w.N[32 * sp + lane] + v;
                    if (n > 2147483647) { bad |= kErrOverflow; n = 2147483647; }
                    w.N[32 * sp + lane] = (int32_t)n;
                    pr.set(sp, (int32_t)n);
                    dirty |= 1u << sp;
                };
                int32_t* own = words + ((p ^ 1) * B + (int)threadIdx.x) * 4 * S;
                if (S <= 2) {
                    int4* a = reinterpret_cast<int4*>(own);
                    for (int k = 0; k < S; ++k) {
                        const int4 x = a[k];
                        if ((x.x | x.y | x.z | x.w) == 0) continue;
                        a[k] = make_int4(0, 0, 0, 0);
                        if (S == 1) {
                            add(0, (int64_t)x.x + x.y + x.z + x.w);
                        } else {
                            if (x.x | x.z) add(0, (int64_t)x.x + x.z);
                            if (x.y | x.w) add(1, (int64_t)x.y + x.w);
                        }
                    }
                } else {
                    unsigned long long bits = masks[(p ^ 1) * B + threadIdx.x];
                    if (bits) masks[(p ^ 1) * B + threadIdx.x] = 0ull;
                    while (bits) {
                        const int i = __ffsll((long long)bits) - 1;
                        bits &= bits - 1ull;
                        add(i & 15, own[(i >> 4) * S + (i & 15)]);
                    }
                }
            }
        }
        if (q == end) break;
        const bool last = r.last_short && q == r.periods - 1;
        const PeriodView v{r.period0 + (uint32_t)q, last ? r.tau_last : r.tau, last ? r.tau_lastf : r.tauf, r.seed,
                           last ? r.thr_last : r.thr, 1};
        send.bits = 0;
        send.words = words_at + (uint32_t)(p * B * 16 * S);
        send.masks = masks_at + (uint32_t)(p * B * 8);
        bool deferred = false;
        bad |= warp_step<S_ == 1, kReact, false, false>(m, mp, S, w, v, t, live, mask, pr, &dirty, &deferred, s.err,
                                                        send);
        if (live && !deferred) send.finish();
        if (__ballot_sync(0xffffffffu, deferred)) {
            const uint32_t x = step_deferred_in_cluster<kReact>(
                m, mp, w.N, w.rx, v.period, v.tau_k, v.seed, v.thr,
                make_uint4(send.slot[0], send.slot[1], send.slot[2], send.slot[3]), send.words, send.masks, t, deferred,
                (pr.many >> 16) == 0u, s.err, r.left ? stop_at : 0u, (uint32_t)q + 1u);
            dirty |= x & 0xffffu;
            bad |= x >> 16;
            if (deferred) pr = presence_of(w.N + lane, S);
        }
    }
    if (end < r.periods && blockIdx.x == 0 && threadIdx.x == 0) *r.left = (uint32_t)end + 1u;
    if (live)
        for (uint32_t bits = dirty; bits; bits &= bits - 1u) {
            const int sp = __ffs(bits) - 1;
            s.cnt[sp * T + t] = w.N[32 * sp + lane];
        }
    if (bad) atomicOr(s.err, bad);
}

// CTAs of k_run_cluster for T tets, at most `most`, and the warps of each (at
// most 16: slot numbers below 4,096, registers; shared memory within 200 KB),
// or 0.
int cluster_shape(int64_t T, int S, bool react, int most, int* warps) {
    const int64_t chunks = (T + 31) / 32;
    int n = 1;
    while (n < most && n < chunks) n <<= 1;
    const int64_t per = (chunks + n - 1) / n;
    *warps = (int)per;
    if (per > 16 || (size_t)cluster_words(S, react, (int)per) * sizeof(int32_t) > kClusterShared) return 0;
    return n;
}

template <int S_, bool kReact>
cudaError_t launch_cluster_s(const DevMesh& m, const ModelParams& mp, const DevState& s, const RunArgs& r, int ctas,
                             int warps, cudaStream_t st) {
    auto kern = k_run_cluster<S_, kReact>;
    const size_t smem = (size_t)cluster_words(mp.S, kReact, warps) * sizeof(int32_t);
    cudaError_t ce = allow_shared((const void*)kern, smem, kClusterShared);
    if (ce == cudaSuccess && ctas > 8) ce = set_once((const void*)kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (ce != cudaSuccess) return ce;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas, 1, 1);
    cfg.blockDim = dim3(32 * warps, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = ctas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    RunArgs r_ = r;
    if (warps <= leave_above_warps(mp)) r_.left = nullptr;
    ce = cudaLaunchKernelEx(&cfg, kern, m, mp, s, r_);
    if (ce == cudaSuccess) ++g_launches;
    return ce;
}

// Warps a block and blocks of k_run for T tets, or 0 if they do not fit: the
// 32-tet warps are spread over all SMs first (a warp that has an SM's issue
// slots and caches to itself is fastest), in at most 3 blocks of 8 warps an SM.
// Up to 2 blocks an SM (77,824 tets on 152 SMs) the kernel has 128 registers,
// above it 80 (eleven species on 12,870 tets, 60 periods: 1.27 ms with 128,
// 1.36 with 80; 3,072-tet cube, 217 periods, 1.30 and 1.47).
int run_shape(int64_t T, int sms, int* warps) {
    const int64_t chunks = (T + 31) / 32;
    const int64_t per_sm = (chunks + sms - 1) / sms;
    if (per_sm > 24) return 0;
    const int64_t blocks_per_sm = (per_sm + 7) / 8;
    *warps = (int)((per_sm + blocks_per_sm - 1) / blocks_per_sm);
    return (int)((chunks + *warps - 1) / *warps);
}

// What a period of k_run may take at most, doubled: the event cap, at 12,000
// cycles an event and 1,000 for each reaction and species of the model (10,000
// measured with two of each, 16,000 with 30 reactions and eleven species), a
// clock of half the usual 2 GHz, and the warps of a multiprocessor sharing its
// FP64 unit, which four of them keep busy.
unsigned long long longest_period_ns(const ModelParams& mp, int warps_per_sm) {
    const unsigned long long cycles = 12000ull + 1000ull * (unsigned)(mp.R + mp.S);
    return (unsigned long long)kEventCap * cycles * (unsigned)std::max(4, warps_per_sm) / 4ull;
}

template <int S_, bool kReact, int kBlocks>
cudaError_t launch_run_b(const DevMesh& m, const ModelParams& mp, const DevState& s, const RunArgs& r, int grid,
                         int warps, int sms, cudaStream_t st) {
    auto kern = k_run<S_, kReact, kBlocks>;
    const size_t smem = (size_t)warps * warp_words(mp.S, kReact) * sizeof(int32_t);
    cudaError_t ce = allow_shared((const void*)kern, smem, block_shared_most(kReact));
    int fit = 0;
    if (ce == cudaSuccess) ce = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kern, 32 * warps, smem);
    if (ce == cudaSuccess && (int64_t)fit * sms < grid) ce = cudaErrorCooperativeLaunchTooLarge;
    if (ce != cudaSuccess) return ce;
    DevMesh m_ = m;
    ModelParams mp_ = mp;
    DevState s_ = s;
    RunArgs r_ = r;
    if (r.periods > 1) r_.left = nullptr;   // nothing that may leave is queued before it
    if (r_.wait_limit_ns == 0) r_.wait_limit_ns = longest_period_ns(mp, warps * ((grid + sms - 1) / sms));
    void* args[] = {&m_, &mp_, &s_, &r_};
    ce = cudaLaunchCooperativeKernel((const void*)kern, dim3(grid), dim3(32 * warps), args, smem, st);
    if (ce == cudaSuccess) ++g_launches;
    return ce;
}

template <int S_, bool kReact>
cudaError_t launch_run_s(const DevMesh& m, const ModelParams& mp, const DevState& s, const RunArgs& r, int grid,
                         int warps, int sms, cudaStream_t st) {
    if (grid <= 2 * sms) return launch_run_b<S_, kReact, 2>(m, mp, s, r, grid, warps, sms, st);
    return launch_run_b<S_, kReact, 3>(m, mp, s, r, grid, warps, sms, st);
}

bool launch_run(const DevMesh& m, const ModelParams& mp, const DevState& s, const RunArgs& r, int sms, int* grid,
                cudaStream_t st) {
    int warps = 0;
    cudaError_t ce = cudaErrorInvalidConfiguration;
    // 16 CTAs are beyond the portable cluster size: where the device has no
    // room for one, 8 (a launch that cannot be placed fails with no effect)
    for (int most = r.spread ? 0 : 16; most >= 8; most >>= 1) {
        const int ctas = cluster_shape(m.T, mp.S, mp.any_reaction != 0, most, &warps);
        if (ctas == 0) break;
        if (mp.S == 1)
            ce = mp.any_reaction ? launch_cluster_s<1, true>(m, mp, s, r, ctas, warps, st)
                                 : launch_cluster_s<1, false>(m, mp, s, r, ctas, warps, st);
        else
            ce = mp.any_reaction ? launch_cluster_s<0, true>(m, mp, s, r, ctas, warps, st)
                                 : launch_cluster_s<0, false>(m, mp, s, r, ctas, warps, st);
        *grid = 0;   // no grid barrier
        if (ce == cudaSuccess) return true;
        cudaGetLastError();
    }
    *grid = run_shape(m.T, sms, &warps);
    if (*grid == 0) return false;
    if (mp.S == 1)
        ce = mp.any_reaction ? launch_run_s<1, true>(m, mp, s, r, *grid, warps, sms, st)
                             : launch_run_s<1, false>(m, mp, s, r, *grid, warps, sms, st);
    else
        ce = mp.any_reaction ? launch_run_s<0, true>(m, mp, s, r, *grid, warps, sms, st)
                             : launch_run_s<0, false>(m, mp, s, r, *grid, warps, sms, st);
    if (ce != cudaSuccess) cudaGetLastError();   // no room for a cooperative launch: one launch a period
    return ce == cudaSuccess;
}

template <int S_, bool kReact, int kPass>
void launch_pass(const DevMesh& m, const ModelParams& mp, const DevState& s, const PeriodArgs& a, int32_t* queue,
                 int32_t* qcount, int32_t parity, int grid, int block, cudaStream_t st) {
    const size_t smem = (size_t)(block / 32) * warp_words(mp.S, kReact) * sizeof(int32_t);
    // large blocks of many species; a failure is reported as the launch's (last error)
    if (allow_shared((const void*)k_period<S_, kReact, kPass>, smem, block_shared_most(kReact)) != cudaSuccess) return;
    k_period<S_, kReact, kPass><<<grid, block, smem, st>>>(m, mp, s, a, queue, qcount, parity);
    ++g_launches;
}

template <int S_>
void launch_period_s(const DevMesh& m, const ModelParams& mp, const DevState& s, const PeriodArgs& a, int block,
                     int32_t* queue, int32_t* qcount, int32_t parity, bool split, cudaStream_t st) {
    const int64_t n = (a.t_hi > 0 ? a.t_hi : m.T) - a.t_lo;
    const int grid = (int)((n + block - 1) / block);
    if (!mp.any_reaction) {
        // no reaction phase to defer: without reactions one pass is both
        launch_pass<S_, false, kPassAll>(m, mp, s, a, nullptr, nullptr, 0, grid, block, st);
    } else if (!split) {
        launch_pass<S_, true, kPassAll>(m, mp, s, a, nullptr, nullptr, 0, grid, block, st);
    } else {
        launch_pass<S_, true, kPassFirst>(m, mp, s, a, queue, qcount, parity, grid, block, st);
        launch_pass<S_, true, kPassQueue>(m, mp, s, a, queue, qcount, parity,
                                          std::min(grid_for(n), 2 * sm_count()), kBlock, st);
    }
}

static void launch_any(const DevMesh& m, const ModelParams& mp, const DevState& s, const PeriodArgs& a, int block,
                       int32_t* queue, int32_t* qcount, int32_t parity, bool split, cudaStream_t st) {
    if (mp.S == 1) launch_period_s<1>(m, mp, s, a, block, queue, qcount, parity, split, st);
    else launch_period_s<0>(m, mp, s, a, block, queue, qcount, parity, split, st);
}

void launch_period(const DevMesh& m, const ModelParams& mp, const DevState& s, const PeriodArgs& a, int block,
                   cudaStream_t st) {
    launch_any(m, mp, s, a, block, nullptr, nullptr, 0, false, st);
}

void launch_period_split(const DevMesh& m, const ModelParams& mp, const DevState& s, const PeriodArgs& a,
                         int32_t* queue, int32_t* qcount, int32_t parity, int block, cudaStream_t st) {
    launch_any(m, mp, s, a, block, queue, qcount, parity, true, st);
}

// The closing synchronous transfer of a run, in place; leaves every inbox
// word and mask of its tets cleared.
__global__ void k_gather(int32_t T, int32_t S, DevState s, PeriodArgs a) {
    extern __shared__ int32_t sm[];
    const int t = a.t_lo + blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (a.t_hi > 0 ? a.t_hi : T)) return;
    const int lane = threadIdx.x & 31;
    int32_t* N = sm + (threadIdx.x >> 5) * 32 * S;
    for (int sp = 0; sp < S; ++sp) N[32 * sp + lane] = s.cnt[(int64_t)sp * T + t];
    uint32_t dirty = 0;
    Presence pr;
    const uint32_t bad = take_inbox(a, t, S, lane, N, pr, &dirty);
    for (uint32_t bits = dirty; bits; bits &= bits - 1u) {
        const int sp = __ffs(bits) - 1;
        s.cnt[(int64_t)sp * T + t] = N[32 * sp + lane];
    }
    if (bad) atomicOr(s.err, bad);
}

void launch_gather(const DevMesh& m, int32_t S, const DevState& s, const PeriodArgs& a, cudaStream_t st) {
    const int64_t n = (a.t_hi > 0 ? a.t_hi : m.T) - a.t_lo;
    k_gather<<<grid_for(n), kBlock, (size_t)kBlock * S * sizeof(int32_t), st>>>(m.T, S, s, a);
    ++g_launches;
}

// Inbox slots packed as int32 [n][S] (words without a valid bit are zero).
__global__ void k_inbox_export(int32_t S, const int32_t* __restrict__ inbox, const uint8_t* __restrict__ mask,
                               const int32_t* __restrict__ slots, int32_t n, int32_t* __restrict__ buf) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)n * S) return;
    const int64_t k = i / S;
    const int sp = (int)(i - k * S);
    const int64_t slot = slots[k];
    bool valid = true;
    if (S > 8) valid = (reinterpret_cast<const uint16_t*>(mask)[slot] >> sp) & 1;
    else if (S > 2) valid = (mask[slot] >> sp) & 1;
    buf[i] = valid ? inbox[slot * inbox_stride(S) + sp] : 0;
}

__global__ void k_inbox_import(int32_t S, int32_t* __restrict__ inbox, uint8_t* __restrict__ mask,
                               const int32_t* __restrict__ slots, int32_t n, const int32_t* __restrict__ buf) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int64_t slot = slots[k];
    uint32_t bits = 0;
    for (int sp = 0; sp < S; ++sp) {
        const int32_t v = buf[k * S + sp];
        inbox[slot * inbox_stride(S) + sp] = v;
        if (v != 0) bits |= 1u << sp;
    }
    if (S > 8) reinterpret_cast<uint16_t*>(mask)[slot] = (uint16_t)bits;
    else if (S > 2) mask[slot] = (uint8_t)bits;
}

void launch_inbox_export(int32_t S, const int32_t* inbox, const uint8_t* mask, const int32_t* slots, int32_t n,
                         int32_t* buf, cudaStream_t st) {
    if (n <= 0) return;
    k_inbox_export<<<grid_for((int64_t)n * S), kBlock, 0, st>>>(S, inbox, mask, slots, n, buf);
    ++g_launches;
}

void launch_inbox_import(int32_t S, int32_t* inbox, uint8_t* mask, const int32_t* slots, int32_t n,
                         const int32_t* buf, cudaStream_t st) {
    if (n <= 0) return;
    k_inbox_import<<<grid_for(n), kBlock, 0, st>>>(S, inbox, mask, slots, n, buf);
    ++g_launches;
}

}  // namespace rdk
