// Arithmetic and compact form of the latent state (K = 1, 2).
//
// For one offset tau, source pixel m and band c the NP = (2K+1)^2 entries s_k = Sig'_{tau k}(m) of an
// iteration are all driven by the same difference delta = X(m) - X(m - tau) (see k_latent.cuh):
//   s_k' = clamp(s_k - delta, -mu_k, mu_k),   sum_k G_k = NP delta + 2 sum_k s_k' - sum_k s_k.
//
// Grid.  X (in the update of s), mu_k and therefore s_k are kept on a grid g Z, g a power of two
// with mu_max <= 2^B g (B = 24 in FP32, 53 in FP64; mu_max = lambda2/rho times the largest weight):
// X is rounded to the grid and mu_k rounded down to it.  Every s_k is then a multiple of g of at
// most 2^B g, an exact value of the iterate type, the update is exact, and so is the sum over k in
// any order.  The grid is as fine as the iterate type's own spacing below mu_max.
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
    T wmax;                     // the largest weight it was made for
};

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

// Code of a threshold: rounded down; a weight that is not a number or infinite acts as the largest.
__device__ __forceinline__ int32_t mu_code(float mu, float ig) {
    const float cap = 16777216.0f;                              // 2^B
    const float c = fabsf(mu) * ig;
    return __float2int_rz(c <= cap ? c : cap);
}
__device__ __forceinline__ int64_t mu_code(double mu, double ig) {
    const double cap = 9007199254740992.0;                      // 2^B
    const double c = fabs(mu) * ig;
    return __double2ll_rz(c <= cap ? c : cap);
}
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
template <typename T> __device__ __forceinline__ bool big_move(T delta, T ig);
template <> __device__ __forceinline__ bool big_move<float>(float delta, float ig) {
    return !(fabsf(delta) * ig < 67108864.0f);                  // 2^26
}
template <> __device__ __forceinline__ bool big_move<double>(double delta, double ig) {
    return !(fabs(delta) * ig < 36028797018963968.0);           // 2^55
}
// Code of delta = a - b for the entry-by-entry update.
template <typename T>
__device__ __forceinline__ code_t<T> delta_code(T a, T b, T ig) {
    using C = code_t<T>;
    using U = typename grid_code<T>::utype;
    const T d = a - b;
    if (big_move<T>(d, ig)) return d < T(0) ? -(C(4) << grid_code<T>::B) : (C(4) << grid_code<T>::B);
    return (C)((U)x_code(a, ig) - (U)x_code(b, ig));
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
// rank's threshold, at w >= trig going up and w < trig going down; with q = 0 when |w - trig| reaches
// half.  meta: beta (bits 0-4), free (5), q > 0 (30), not up (31), and with 9 ranks E (bits 6-14) and
// G (bits 15-23); with 25 ranks E and G have their own words.
constexpr uint32_t kRecordSat = 1u << 30, kRecordDown = 1u << 31;
template <typename C>
struct alignas(4 * sizeof(C)) LevelRecord {
    C alpha, trig, half;
    uint32_t meta;
};

template <int NP>
FUSE_LEVEL_FN uint32_t levels_meta(const Levels& l) {
    uint32_t m = (uint32_t)(NP - l.q) | (l.free ? 32u : 0u) | (l.q > 0 ? kRecordSat : 0u) | (l.up ? 0u : kRecordDown);
    if constexpr (NP == 9) m |= l.E << 6 | l.G << 15;
    return m;
}
template <int NP>
FUSE_LEVEL_FN Levels levels_of(uint32_t meta, uint2 masks) {
    Levels l;
    l.q = NP - (int)(meta & 31u);
    l.up = !(meta & kRecordDown);
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
            trig = up ? e + a : e - a + 1;
        } else {
            trig = fr ? e : (plus ? e - mu : e + mu);
            half = mu;
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
    C alpha = rec.alpha, trig = l.up ? rec.trig : rec.trig - 1;
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
            rec.trig = l.up ? trig : trig + 1;
            rec.meta = levels_meta<NP>(l);
            return true;
        }
    }
    return false;
}

// Whether the linear stretch of a record ends with the move to w1 = w0 - delta: up = delta < 0,
// down = delta > 0, big = big_move.  With every rank saturated (beta = 0) only a turn ends it.
template <typename C>
FUSE_LEVEL_FN bool level_due(const LevelRecord<C>& r, C w1, bool up, bool down, bool big) {
    const bool dn = (r.meta & kRecordDown) != 0, sat = (r.meta & kRecordSat) != 0;
    const auto c = signed_of(w1 - r.trig);
    const auto v = sat ? (dn ? ~c : c) : (c < 0 ? -c : c) - signed_of(r.half);
    return (sat && (dn ? up : down)) || ((r.meta & 31u) != 0 && (v >= 0 || big));
}

}  // namespace fuse
