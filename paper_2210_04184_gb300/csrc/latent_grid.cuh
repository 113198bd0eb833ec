// Arithmetic and compact form of the latent state (K = 1, 2).
//
// For one offset tau, source pixel m and band c the NP = (2K+1)^2 entries s_k = Sig'_{tau k}(m) of an
// iteration are all driven by the same difference delta = X(m) - X(m - tau) (see k_latent.cuh):
//   s_k' = clamp(s_k - delta, -mu_k, mu_k),   sum_k G_k = NP delta + 2 sum_k s_k' - sum_k s_k.
//
// Grid.  X (in the update of s), mu_k and therefore s_k are kept on a grid g Z, g a power of two
// with mu_max <= 2^B g (B = 24 in FP32, 53 in FP64; mu_max = lambda2/rho times the largest weight):
// X and mu_k are rounded to the grid, to nearest.  Every s_k is then a multiple of g of at
// most 2^B g, an exact value of the iterate type, the update is exact, and so is the sum over k in
// any order.  In the topmost binade below mu_max the grid is the iterate type's own spacing; smaller
// values keep the same absolute step.
//
// Where it is used.  The iterate type keeps small values to more bits than the grid does, so a solve is
// on the grid only while its range 2^B g (mu_max to the next power of two) is at most the size of X,
// taken from the rms of the Y_l samples (latent_begin_kernel); else, and with weights that are not finite or negative, it runs
// the arithmetic of the iterate type.  Error of X from the latent update alone, all else in FP64
// (relative, 40 iterations, means over three 32 x 32 scenes, 25 entries), by range / rms:
//   0.26  grid 1.44e-7, FP32 entries 1.48e-7        4.1  grid 1.86e-7, FP32 entries 1.39e-7
//   0.52  grid 1.50e-7, FP32 entries 1.52e-7       16.5  grid 4.54e-7, FP32 entries 1.30e-7
//   0.86  grid 1.38e-7, FP32 entries 1.38e-7        132  grid 2.62e-6, FP32 entries 1.05e-7
//   2.1   grid 1.47e-7, FP32 entries 1.40e-7
// (mu_k rounded down, all in one direction, gave 1.7e-7, 2.7e-7 and 3.2e-7 in the first three rows.)
//
// Compact form.  With w = -sum_t delta_t (in units of g) s is, as a function of its threshold mu, the
// state of a stop operator driven by w.  In ascending order of mu it consists of levels: a run of
// ranks saturated in the direction of the last move, s = sigma mu; runs that left their threshold
// when w was e and have moved with w since, s = sigma mu + (w - e); and the ranks that never
// reached it, s = w - e.  s is 1-Lipschitz in mu, so a move saturates a prefix of the ranks.  The sum
// over the ranks is linear in w, S(w) = alpha + beta w (beta = the ranks that are not saturated),
// until an event: w turns while some ranks are saturated, or reaches the value `trig` at which the
// next rank saturates.  A record holds alpha, beta and the bounds of the linear stretch, so an
// iteration without an event reads one record and writes nothing.  Measured on the HS+MS workload
// (25 entries): 1.4 levels on average after 50 iterations; events in 5% of the records per
// iteration from the 20th on.
#pragma once
#include <type_traits>

#include "common.cuh"

// The level arithmetic is also compiled for the host, to be checked there against the entry-by-entry
// update.
#ifndef FUSE_LEVEL_FN
#define FUSE_LEVEL_FN __device__ __forceinline__
#endif

namespace fuse {

// Integer type of the codes (multiples of g).  Sums: 2 sum s' - sum s <= 75 2^24 < 2^31 in FP32.
template <typename T> struct grid_code;
template <> struct grid_code<float> {
    using type = int32_t;
    using utype = uint32_t;
    static constexpr int B = 24;
};
template <> struct grid_code<double> {
    using type = int64_t;
    using utype = uint64_t;
    static constexpr int B = 53;
};
template <typename T> using code_t = typename grid_code<T>::type;
// The running sums, levels and records are kept modulo 2^32 (2^64), as unsigned integers; a difference
// of values less than half the modulus apart is signed(a - b).
template <typename T> using ucode_t = typename grid_code<T>::utype;
FUSE_LEVEL_FN int32_t signed_of(uint32_t v) { return (int32_t)v; }
FUSE_LEVEL_FN int64_t signed_of(uint64_t v) { return (int64_t)v; }

__host__ __device__ constexpr bool latent_grid_k(int K) { return K == 1 || K == 2; }

template <typename T> struct LatentGrid {
    T g, ig;                    // grid step and its reciprocal (powers of two)
    T wmax;                     // the largest weight it was made for; infinite if one is not a finite
                                // number >= 0
};

// What the latent state of a context holds, kept on the device: the calls that change it and the
// kernels that depend on it are ordered by the stream, and a captured call that is replayed later finds
// the state as it is then.
//   kStateEntries  entries of the iterate type, updated in its arithmetic
//   kStateGrid     entries on the grid, those of a run on the current weights
//   kStateLevels   levels, formed with the current weights or, with `was`, with the ones before them
//   kStateGiven    entries not looked at yet: set by the caller, or left by other weights
// latent_begin_kernel: most blocks of a problem, samples of a block at a time
constexpr int kBeginBlocks = 256, kBeginSamples = 8192;
enum : int { kStateEntries = 0, kStateGrid = 1, kStateLevels = 2, kStateGiven = 3 };
struct LatentCtl {
    int mode;
    int was;                    // omega_was and grid[1] describe the levels
    int table;                  // the threshold table is that of the current weights
    int off;                    // some entry is not that of a run on the current weights
    int fit;                    // the grid carries the thresholds and X of the last solve's inputs
    unsigned done;              // blocks of the running kernel that have finished
    double part[kBeginBlocks], seen[kBeginBlocks];
};
// Whether an entry kernel is to run: ctl NULL, always; else where the state is entries, on the grid or not
// as the kernel's arithmetic.
__device__ __forceinline__ bool entries_due(const LatentCtl* ctl, bool grid) {
    if (!ctl) return true;
    const int mode = ctl->mode;
    return grid ? mode == kStateGrid : mode == kStateEntries || mode == kStateGiven;
}

// The grid of thresholds coef w, 0 <= w <= wmax: 2^e >= coef wmax, g = 2^(e - B).
inline __host__ __device__ LatentGrid<float> latent_grid(float coef, float wmax) {
    int e = 0;
    const float m = fminf(coef * wmax, 1e38f);
    if (m > 0.0f) frexpf(m, &e);
    e = e < -96 ? -96 : e;
    return {ldexpf(1.0f, e - grid_code<float>::B), ldexpf(1.0f, grid_code<float>::B - e), wmax};
}
inline __host__ __device__ LatentGrid<double> latent_grid(double coef, double wmax) {
    int e = 0;
    const double m = fmin(coef * wmax, 1e307);
    if (m > 0.0) frexp(m, &e);
    e = e < -900 ? -900 : e;
    return {ldexp(1.0, e - grid_code<double>::B), ldexp(1.0, grid_code<double>::B - e), wmax};
}

// Code of a threshold: rounded to nearest.
__device__ __forceinline__ int32_t mu_code(float mu, float ig) {
    const float cap = 16777216.0f;                              // 2^B
    const float c = fabsf(mu) * ig;
    return __float2int_rn(c <= cap ? c : cap);
}
__device__ __forceinline__ int64_t mu_code(double mu, double ig) {
    const double cap = 9007199254740992.0;                      // 2^B
    const double c = fabs(mu) * ig;
    return __double2ll_rn(c <= cap ? c : cap);
}
// The threshold of one weight column: in the iterate type, or as a code on the grid.
template <typename T, bool GRID>
struct latent_bound {
    SymBound<T> b;
    __device__ __forceinline__ static latent_bound of(T mu, T) { return {SymBound<T>::of(mu)}; }
    __device__ __forceinline__ T clamp(T u) const { return b.clamp(u); }
};
template <typename T>
struct latent_bound<T, true> {
    code_t<T> m;
    SymBound<T> b;
    __device__ __forceinline__ static latent_bound of(T mu, T ig) { return {mu_code(mu, ig), SymBound<T>::of(mu)}; }
    __device__ __forceinline__ code_t<T> clamp(code_t<T> u) const { return u > m ? m : (u < -m ? -m : u); }
    // The entry of code s, as it is stored.  An entry at a threshold that was rounded up is stored as the
    // threshold itself, so |s| <= mu holds for every stored state; its code is that of mu.
    __device__ __forceinline__ T entry(code_t<T> s, T g) const { return b.clamp((T)s * g); }
};
// Code of an X value: rounded to nearest, modulo 2^32 (FP64: 2^64).  Differences of codes are taken
// modulo as well; they are used only where |delta| < kBigMove g.
__device__ __forceinline__ int32_t x_code(float x, float ig) {
    const float t = rintf(x * ig);
    if (fabsf(t) < 2147483648.0f) return __float2int_rn(t);
    const float m = fabsf(t);                                   // a multiple of 2^32 from 2^55 on
    const uint32_t u = m < 9.0e18f ? (uint32_t)__float2ull_rz(m) : 0u;
    return (int32_t)(t < 0.0f ? 0u - u : u);
}
__device__ __forceinline__ int64_t x_code(double x, double ig) {
    const double t = rint(x * ig);
    if (fabs(t) < 9.0e18) return __double2ll_rn(t);
    const double m = fmod(fabs(t), 18446744073709551616.0);     // NaN for infinities: converts to 0
    const uint64_t u = __double2ull_rz(m);
    return (int64_t)(t < 0.0 ? 0ull - u : u);
}
// A move of at least this many steps saturates every entry whatever its state (thresholds are at
// most 2^B steps).  Not-a-number counts as such a move.
__device__ __forceinline__ bool big_move(float delta, float g) { return !(fabsf(delta) < 67108864.0f * g); }
__device__ __forceinline__ bool big_move(double delta, double g) { return !(fabs(delta) < 36028797018963968.0 * g); }
// Code of delta = a - b for the entry-by-entry update.
template <typename T>
__device__ __forceinline__ code_t<T> delta_code(T a, T b, const LatentGrid<T>& gr) {
    using C = code_t<T>;
    using U = typename grid_code<T>::utype;
    const T d = a - b;
    if (big_move(d, gr.g)) return d < T(0) ? -(C(4) << grid_code<T>::B) : (C(4) << grid_code<T>::B);
    return (C)((U)x_code(a, gr.ig) - (U)x_code(b, gr.ig));
}
__device__ __forceinline__ int32_t to_code(float v) { return __float2int_rn(v); }
__device__ __forceinline__ int64_t to_code(double v) { return __double2ll_rn(v); }

// H = sum_k G_k = NP delta + g (2 sum s' - sum s) from the codes' sums; the same rounding in every
// kernel.
template <int NP>
__device__ __forceinline__ float latent_h(float delta, int32_t t, float g) {
    return __fmaf_rn((float)NP, delta, __fmul_rn(g, __int2float_rn(t)));
}
template <int NP>
__device__ __forceinline__ double latent_h(double delta, int64_t t, double g) {
    return __fma_rn((double)NP, delta, __dmul_rn(g, __ll2double_rn(t)));
}

// Levels of one (tau, c, m): bit r of E is set when rank r (ascending mu) ends a level, bit r of G
// when that level has sigma = +1; q ranks are saturated (the lowest level, when q > 0), in direction
// `up`; free: the highest level has sigma = 0.  The values e are stored by height: the highest
// level's in plane 0, the next lower one's in plane 1, ...; the saturated level has none.
struct Levels {
    uint32_t E, G;
    int q;
    bool up, free;
};
// Record: S(w) = alpha + beta w.  With q > 0 the stretch ends when w turns or reaches the next
// rank's threshold value t (trig = -t going up, t + 1 going down, see level_due); with q = 0 when w
// leaves [trig, trig + half].  meta: beta (bits 0-4), free (5), q > 0 (30), q > 0 and up (31), and with
// 9 ranks E (bits 6-14) and G (bits 15-23); with 25 ranks E and G have their own words.
constexpr uint32_t kRecordSat = 1u << 30, kRecordUp = 1u << 31;
template <typename C>
struct alignas(4 * sizeof(C)) LevelRecord {
    C alpha, trig, half;
    uint32_t meta;
};

template <int NP>
FUSE_LEVEL_FN uint32_t levels_meta(const Levels& l) {
    uint32_t m = (uint32_t)(NP - l.q) | (l.free ? 32u : 0u) | (l.q > 0 ? kRecordSat | (l.up ? kRecordUp : 0u) : 0u);
    if constexpr (NP == 9) m |= l.E << 6 | l.G << 15;
    return m;
}
template <int NP>
FUSE_LEVEL_FN Levels levels_of(uint32_t meta, uint2 masks) {
    Levels l;
    l.q = NP - (int)(meta & 31u);
    l.up = meta & kRecordUp;
    l.free = meta & 32u;
    if constexpr (NP == 9) {
        l.E = (meta >> 6) & 0x1ffu;
        l.G = (meta >> 15) & 0x1ffu;
    } else {
        l.E = masks.x;
        l.G = masks.y;
    }
    return l;
}

FUSE_LEVEL_FN int bits_set(uint32_t v) {
#ifdef __CUDA_ARCH__
    return __popc(v);
#else
    return __builtin_popcount(v);
#endif
}
FUSE_LEVEL_FN int lowest_bit(uint32_t v) {      // 1-based, v != 0
#ifdef __CUDA_ARCH__
    return __ffs((int)v);
#else
    return __builtin_ffs((int)v);
#endif
}

// The range of w without an event when no rank is saturated: |w - centre| < mu (w = centre for mu = 0).
template <typename C>
FUSE_LEVEL_FN void level_free_range(LevelRecord<C>& rec, C centre, C mu) {
    rec.trig = mu > 0 ? centre - mu + 1 : centre;
    rec.half = mu > 0 ? 2 * mu - 2 : C(0);
}

// An event: the levels and the record after the move from w0 to w1 (all: a big move, which saturates
// every rank) in the direction `up`.  P(r): sum of the r smallest threshold codes (r = 0 .. NP);
// ld(p) / st(p, e): the value e of plane p.  Only the levels that the move reaches are visited:
// alpha changes by their ranks' terms.
template <int NP, typename C, typename FP, typename FL, typename FS>
FUSE_LEVEL_FN void level_event(Levels& l, LevelRecord<C>& rec, C w0, C w1, bool up, bool all, FP P, FL ld, FS st) {
    const int np = bits_set(l.E) - (l.q > 0);         // stored levels
    uint32_t Er = l.E;
    int q = 0, pl = l.q > 0 ? np : np - 1;            // ranks saturated so far; height of the level
    bool top = l.q > 0, plus = false, fr = false;
    C Pq = 0, Pn = 0, e = 0;                          // P(q), P(q + 1), the level's value
    C alpha = rec.alpha;
    while (!all) {
        const int lo = q, hi = lowest_bit(Er);
        const C Plo = Pq;
        plus = (l.G >> (hi - 1)) & 1u;
        fr = l.free && (Er & (Er - 1)) == 0;
        e = top ? w0 : ld(pl);
        const auto a = signed_of(up ? w1 - e : e - w1);
        if (!fr && plus == up) {                      // on its way back: as a whole, at w = e
            Pq = a >= 0 ? P(hi) : Plo;
            q = a >= 0 ? hi : lo;
        } else {
            const auto thr = fr ? a : (a >> 1);       // ranks with mu <= thr reach their threshold
            Pn = P(q + 1);
            int b = hi;
            for (int near = 0; q < b && thr >= 0;) {  // two ranks in turn, then by halves
                const int mid = near++ < 2 ? q : (q + b) >> 1;
                const C Pm = mid == q ? Pq : P(mid), Pm1 = mid == q ? Pn : P(mid + 1);
                if (signed_of(Pm1 - Pm) <= thr) {
                    q = mid + 1;
                    Pq = Pm1;
                    if (q < b) Pn = P(q + 1);
                } else {
                    b = mid;
                }
            }
        }
        // the terms of the ranks [lo, q): sigma mu - e, for the level saturated until now sigma mu
        const C run = fr ? C(0) : (plus ? Pq - Plo : Plo - Pq);
        alpha -= run - (top ? C(0) : (C)(q - lo) * e);
        if (q < hi) {
            if (top) {                                // its other ranks leave the threshold now
                st(np, w0);
                alpha -= (C)(hi - q) * w0;
            }
            break;
        }
        Er &= Er - 1;
        all = Er == 0;
        top = false;
        --pl;
    }
    C trig = 0, half = 0;
    if (!all) {
        const C mu = P(q + 1) - Pq;
        alpha += up ? Pq : C(0) - Pq;
        if (q > 0) {
            const C a = fr ? mu : (plus == up ? C(0) : 2 * mu);
            trig = up ? C(0) - (e + a) : e - a + 1;
        } else {
            level_free_range<C>(rec, fr ? e : (plus ? e - mu : e + mu), mu);
            trig = rec.trig;
            half = rec.half;
        }
    } else {
        q = NP;
        const C s = P(NP);
        alpha = up ? s : C(0) - s;
        l.free = false;
    }
    const uint32_t below = (1u << q) - 1u;
    l.E &= ~below;
    l.G &= ~below;
    if (q > 0) {
        l.E |= 1u << (q - 1);
        if (up) l.G |= 1u << (q - 1);
    }
    l.q = q;
    l.up = up;
    rec.alpha = alpha;
    rec.trig = trig;
    rec.half = half;
    rec.meta = levels_meta<NP>(l);
}

// The frequent event: w goes on in the direction of the saturated ranks and the next level's first
// ranks (at most kGrowRanks, not the whole level) reach their threshold.  A rank that does so at
// w = trig goes from sigma mu + (w - e) to the constant it has there, so alpha gains trig; the
// next trig is further by the difference of the thresholds (twice it for a level of the opposite
// sigma).  Returns false, with nothing changed, for any other event.
constexpr int kGrowRanks = 4;
template <int NP, typename C, typename FP>
FUSE_LEVEL_FN bool level_grow(Levels& l, LevelRecord<C>& rec, C w0, C w1, bool big, FP P) {
    if (l.q == 0 || l.q == NP || big || signed_of(l.up ? w1 - w0 : w0 - w1) < 0) return false;
    const uint32_t Er = l.E >> l.q;
    const int hi = l.q + lowest_bit(Er);
    const bool fr = l.free && (Er & (Er - 1)) == 0;
    if (!fr && (((l.G >> (hi - 1)) & 1u) != 0) == l.up) return false;
    int q = l.q;
    C alpha = rec.alpha, trig = l.up ? C(0) - rec.trig : rec.trig - 1;
    if (signed_of(l.up ? w1 - trig : trig - w1) < 0) return false;
    C P1 = P(q + 1), mu = P1 - P(q);
    for (int i = 0; i < kGrowRanks; ++i) {
        if (q + 1 == hi) return false;
        const C P2 = P(q + 2), mu2 = P2 - P1, d = fr ? mu2 - mu : 2 * (mu2 - mu);
        alpha += trig;
        trig = l.up ? trig + d : trig - d;
        ++q;
        P1 = P2;
        mu = mu2;
        if (signed_of(l.up ? w1 - trig : trig - w1) < 0) {
            l.E = (l.E & ~((1u << q) - 1u)) | 1u << (q - 1);
            l.G = (l.G & ~((1u << q) - 1u)) | (l.up ? 1u << (q - 1) : 0u);
            l.q = q;
            rec.alpha = alpha;
            rec.trig = l.up ? C(0) - trig : trig + 1;
            rec.meta = levels_meta<NP>(l);
            return true;
        }
    }
    return false;
}

// The levels and the record of given entries s (ascending thresholds mu, |s| <= mu, 1-Lipschitz in mu)
// at w; st(p, e) as above.  The saturated prefix first, as long as it goes, so that w lies strictly
// inside the stretch; then from the largest threshold down: a level is extended while one of its
// forms s = d, s = mu + d, s = -mu + d still fits (d = w - e).
template <int NP, typename C, typename FS>
FUSE_LEVEL_FN void levels_from_entries(const C (&s)[NP], const C (&mu)[NP], C w, Levels& l, LevelRecord<C>& rec, FS st) {
    int qu = 0, qd = 0;
    C P = 0;
    for (int r = 0; r < NP; ++r) {
        if (qu == r && s[r] == mu[r]) ++qu;
        if (qd == r && s[r] == C(0) - mu[r]) ++qd;
    }
    l = Levels{0u, 0u, qu >= qd ? qu : qd, qu >= qd, false};
    C alpha = 0, run = 0, low = 0, d0 = 0, dp = 0, dm = 0, le = 0;
    bool f0 = false, fp = false, fm = false, plus = false;
    int height = 0, end = NP - 1;
    auto close = [&](int first) {                     // ranks [first, end]
        const bool fr = f0;
        plus = !fr && fp;
        le = w - (fr ? d0 : (fp ? dp : dm));
        st(height++, le);
        l.E |= 1u << end;
        if (plus) l.G |= 1u << end;
        if (fr) l.free = true;
        alpha += (fr ? C(0) : (plus ? run : C(0) - run)) - (C)(end + 1 - first) * le;
    };
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int r = NP - 1; r >= 0; --r) {
        if (r < l.q) {
            P += mu[r];
            continue;
        }
        const bool k0 = f0 && s[r] == d0, kp = fp && s[r] - mu[r] == dp, km = fm && s[r] + mu[r] == dm;
        if (k0 || kp || km) {
            f0 = k0;
            fp = kp;
            fm = km;
            run += mu[r];
        } else {
            if (r < NP - 1) close(r + 1);
            end = r;
            run = mu[r];
            f0 = r == NP - 1;                         // sigma = 0: the highest level only
            fp = fm = true;
            d0 = s[r];
            dp = s[r] - mu[r];
            dm = s[r] + mu[r];
        }
        low = mu[r];
    }
    rec.trig = rec.half = 0;
    if (l.q < NP) {
        close(l.q);
        const bool fr = f0;
        const C a = fr ? low : (plus == l.up ? C(0) : 2 * low);
        if (l.q > 0) rec.trig = l.up ? C(0) - (le + a) : le - a + 1;
        else level_free_range<C>(rec, fr ? le : (plus ? le - low : le + low), low);
    }
    if (l.q > 0) {
        l.E |= 1u << (l.q - 1);
        if (l.up) l.G |= 1u << (l.q - 1);
        alpha += l.up ? P : C(0) - P;
    }
    rec.alpha = alpha;
    rec.meta = levels_meta<NP>(l);
}

// Whether the linear stretch of a record ends with the move from w0 to w1 = w0 - delta: up = delta < 0,
// down = delta > 0, big = big_move.  With every rank saturated (beta = 0) only a turn ends it; else, with
// m = -1 for ranks saturated upwards, the stretch is (w1 ^ m) - trig <= (w0 ^ m) - trig as unsigned
// integers: w1 in [w0, t) or (t, w0].
template <typename C>
FUSE_LEVEL_FN bool level_due(const LevelRecord<C>& r, C w0, C w1, bool up, bool down, bool big) {
    const C m = (C)(typename std::make_signed<C>::type)((int32_t)r.meta >> 31);
    const C a = (w1 ^ m) - r.trig, b = (r.meta & kRecordSat) ? (w0 ^ m) - r.trig : r.half;
    return (r.meta & 31u) ? (a > b || big) : ((r.meta & kRecordUp) ? down : up);
}

// A point: X and the running sum of its codes after the current X update and before it, and z = 2
// after - before.  Points [L_s][H][W + 2S]: each row with S points of its other end on either side,
// so the pass reads m - tau without a wrap.
template <typename T>
struct alignas(4 * sizeof(T)) LevelPoint {
    T x;
    ucode_t<T> after, before, z;
};
template <typename T>
__device__ __forceinline__ LevelPoint<T> load_point(const LevelPoint<T>* p) {
    LevelPoint<T> r;
    if constexpr (sizeof(T) == 4) {
        const int4 v = __ldg(reinterpret_cast<const int4*>(p));
        r.x = __int_as_float(v.x);
        r.after = (uint32_t)v.y;
        r.before = (uint32_t)v.z;
        r.z = (uint32_t)v.w;
    } else {
        const longlong2 a = __ldg(reinterpret_cast<const longlong2*>(p)), b = __ldg(reinterpret_cast<const longlong2*>(p) + 1);
        r.x = __longlong_as_double(a.x);
        r.after = (uint64_t)a.y;
        r.before = (uint64_t)b.x;
        r.z = (uint64_t)b.y;
    }
    return r;
}
template <typename T>
__device__ __forceinline__ void store_point(LevelPoint<T>* p, T x, ucode_t<T> after, ucode_t<T> before) {
    const ucode_t<T> z = 2 * after - before;
    if constexpr (sizeof(T) == 4) {
        *reinterpret_cast<int4*>(p) = make_int4(__float_as_int(x), (int)after, (int)before, (int)z);
    } else {
        longlong2 a, b;
        a.x = __double_as_longlong(x);
        a.y = (long long)after;
        b.x = (long long)before;
        b.y = (long long)z;
        reinterpret_cast<longlong2*>(p)[0] = a;
        reinterpret_cast<longlong2*>(p)[1] = b;
    }
}
// The point of column x of a row (row: its first point, the halo's) from the new X; first: the sums
// start at zero.
template <typename T>
__device__ __forceinline__ void update_point(LevelPoint<T>* row, int x, int W, int S, T v, T ig, int first) {
    LevelPoint<T>* p = row + S + x;
    const ucode_t<T> was = first ? ucode_t<T>(0) : p->after;
    const ucode_t<T> now = was + (ucode_t<T>)x_code(v, ig);
    store_point<T>(p, v, now, was);
    if (x < S) store_point<T>(p + W, v, now, was);
    if (x >= W - S) store_point<T>(p - W, v, now, was);
}

}  // namespace fuse
