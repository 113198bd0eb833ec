// Latent pass on the compact state (latent_grid.cuh): the update of eqs. Qj_main and dualvar3_main
// and the adjoint sums A, V of k_latent.cuh (same planes, same order of summation over tau2), with the
// NP entries of a (tau, c, m) kept as levels.  Layouts: records [|W|][L_s][H][W] (|W| the kept
// offsets) and, for 25 entries, the level masks in the same order; level values [|W|][NP][L_s][H][W]
// (plane p of a (tau, c, m) in use for its level of height p); prefix sums of the sorted threshold
// codes of every patch window [|W|][H][W][NP], formed once per weights; points (X with its running sums,
// written by points_kernel from the new X), so w = after(m - tau) - after(m).
//
// One block owns rows [y0, y0 + Ty) of one tau1 row and nb bands.  Per band and tau2 (a step) a thread
// reads its pixel's record and the shifted point; with its own point these give delta, w and the
// previous w, and where the linear stretch holds H_tau(m) follows from them.  The (pixel, step) pairs
// with an event are collected in a list of the block; its threads then take the pairs in turn and try
// the frequent event (level_grow), collecting the others in a second list that is processed last: the
// rare paths run with full warps, evenly spread.  Every H_tau of the block is kept in shared memory, and
// A(m) = sum H_tau(m), V(m) = sum H_tau(m + (0, tau2)) are formed at the end in the order of tau2,
// whatever the order of the lists.
//
// A state that is not kept as levels (LatentCtl) runs the entry kernels instead: an iteration launches
// both, side by side in a captured loop, and the one whose turn it is not returns at once.
#pragma once
#include <type_traits>

#include "latent_grid.cuh"

namespace fuse {

template <typename T, typename WT>
struct LevelArgs {
    const T* X;
    const WT* omega;
    LevelRecord<ucode_t<T>>* rec;
    uint2* masks;
    ucode_t<T>* e;
    const code_t<T>* tab;
    const LevelPoint<T>* pt;
    T* planes;
    int H, W, Ls, S, Ty, nb;
    T coef;
    const LatentGrid<T>* grid;  // device
    int half;
    LatentCtl* ctl;             // device
};

// Whether this is the last block of a launch to finish; true for all of its threads or none.  What the
// other blocks wrote before is visible to it, and no block reads the state's mode after that.
__device__ __forceinline__ bool last_block(LatentCtl* ctl, unsigned blocks) {
    __shared__ int last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(&ctl->done, 1u) == blocks - 1;
        if (last) ctl->done = 0;
        __threadfence();
    }
    __syncthreads();
    return last;
}

template <typename C>
__device__ __forceinline__ LevelRecord<C> load_record(const LevelRecord<C>* p) {
    LevelRecord<C> r;
    if constexpr (sizeof(C) == 4) {
        const int4 v = *reinterpret_cast<const int4*>(p);
        r.alpha = (C)v.x;
        r.trig = (C)v.y;
        r.half = (C)v.z;
        r.meta = (uint32_t)v.w;
    } else {
        const longlong2 a = reinterpret_cast<const longlong2*>(p)[0], b = reinterpret_cast<const longlong2*>(p)[1];
        r.alpha = (C)a.x;
        r.trig = (C)a.y;
        r.half = (C)b.x;
        r.meta = (uint32_t)b.y;
    }
    return r;
}
template <typename C>
__device__ __forceinline__ void store_record(LevelRecord<C>* p, const LevelRecord<C>& r) {
    if constexpr (sizeof(C) == 4) {
        *reinterpret_cast<int4*>(p) = make_int4((int)r.alpha, (int)r.trig, (int)r.half, (int)r.meta);
    } else {
        longlong2 a, b;
        a.x = (long long)r.alpha;
        a.y = (long long)r.trig;
        b.x = (long long)r.half;
        b.y = (long long)r.meta;
        reinterpret_cast<longlong2*>(p)[0] = a;
        reinterpret_cast<longlong2*>(p)[1] = b;
    }
}

// The points of one row of the new X (a warp); first: the sums start at zero.
template <typename T>
__device__ __forceinline__ void points_row(const T* __restrict__ X, LevelPoint<T>* __restrict__ pt, int W, int S,
                                           const LatentGrid<T>* grid, int first, size_t row, int lane) {
    const T ig = grid->ig;
    for (int x = lane; x < W; x += 32)
        update_point<T>(pt + row * (W + 2 * S), x, W, S, X[row * W + x], ig, first);
}
// Eight rows per block.
template <typename T>
__global__ void __launch_bounds__(256)
points_kernel(const T* __restrict__ X, LevelPoint<T>* __restrict__ pt, int rows, int W, int S,
              const LatentGrid<T>* grid, int first, const LatentCtl* ctl) {
    if (ctl->mode != kStateLevels) return;
    const int row = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (row < rows) points_row<T>(X, pt, W, S, grid, first, row, threadIdx.x & 31);
}

template <typename C>
__device__ __forceinline__ void order2(C& a, C& b) {
    const C lo = a < b ? a : b, hi = a < b ? b : a;
    a = lo;
    b = hi;
}

// Batcher's merge exchange (Knuth, TAOCP 5.2.2 M) on N registers; every index is a compile-time
// constant after unrolling.
template <int N, typename C>
__device__ __forceinline__ void sort_network(C (&v)[N]) {
    constexpr int T = N <= 16 ? 4 : 5;
    static_assert(N > 8 && N <= 32, "9 to 32 values");
#pragma unroll
    for (int lp = T - 1; lp >= 0; --lp) {
#pragma unroll
        for (int step = 0; step <= T - 1 - lp; ++step) {
            const int p = 1 << lp;
            const int d = step == 0 ? p : ((1 << (T - 1)) >> (step - 1)) - p;
            const int r = step == 0 ? 0 : p;
#pragma unroll
            for (int i = 0; i < N; ++i)
                if (i + d < N && (i & p) == r) order2(v[i], v[i + d]);
        }
    }
}

// Pixels of a run that a block of the conversions takes at a time, a thread each: two columns of shared
// memory per thread fit 48 KB.
template <typename T, int K>
__host__ __device__ constexpr int window_run() { return sizeof(T) == 8 && K == 2 ? 64 : 128; }

// Threshold codes of the patch window of (y, x): code of coef omega_tau(m + k), k in row-major order; the
// thresholds themselves to a column of shared memory ([NP][window_run]), where given.
template <typename T, typename WT, int K>
__device__ __forceinline__ void window_codes(const WT* __restrict__ om, int y, int x, int H, int W, T coef, T ig,
                                             code_t<T> (&v)[(2 * K + 1) * (2 * K + 1)], T* mus = nullptr) {
    constexpr int PS = 2 * K + 1;
    int col[PS];
#pragma unroll
    for (int j = 0; j < PS; ++j) col[j] = wrap1(x + j - K, W);
#pragma unroll
    for (int i = 0; i < PS; ++i) {
        const WT* row = om + (size_t)wrap1(y + i - K, H) * W;
#pragma unroll
        for (int j = 0; j < PS; ++j) {
            const T mu = coef * (T)wload(row + col[j]);
            v[i * PS + j] = mu_code(mu, ig);
            if (mus) mus[(i * PS + j) * window_run<T, K>()] = mu;
        }
    }
}

// Prefix sums of the sorted threshold codes of every window, where levels need them and they are not those
// of the current weights already; `work` runs of 128 pixels of one kept offset, shared out over the blocks.
template <typename T, typename WT, int K>
__global__ void __launch_bounds__(128)
level_table_kernel(const WT* __restrict__ omega, code_t<T>* __restrict__ tab, int H, int W, int S, int half, T coef,
                   const LatentGrid<T>* grid, int work, LatentCtl* ctl) {
    using C = code_t<T>;
    constexpr int NP = (2 * K + 1) * (2 * K + 1);
    __shared__ C sm[128 * NP];                        // NP is odd: conflict-free
    if (ctl->table || ctl->mode != kStateLevels) return;
    const size_t n = (size_t)H * W;
    const int runs = (int)((n + 127) / 128);
    const TauMap tm{S, half};
    const LatentGrid<T> gr = *grid;
    for (int job = blockIdx.x; job < work; job += gridDim.x) {
        const int si = job / runs;
        const size_t p0 = (size_t)(job - si * runs) * 128, p = p0 + threadIdx.x;
        int t1, t2;
        tau_of_state_index(si, S, half, &t1, &t2);
        if (p < n) {
            C v[NP];
            window_codes<T, WT, K>(omega + (size_t)tm.w_index(t1, t2) * n, (int)(p / W), (int)(p % W), H, W, coef, gr.ig,
                                   v);
            sort_network<NP>(v);
            C sum = 0;
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                sum += v[q];
                sm[threadIdx.x * NP + q] = sum;
            }
        }
        __syncthreads();
        const int cnt = (int)(n - p0 < 128 ? n - p0 : 128) * NP;
        C* out = tab + ((size_t)si * n + p0) * NP;
        for (int i = threadIdx.x; i < cnt; i += 128) out[i] = sm[i];
        __syncthreads();
    }
    if (last_block(ctl, gridDim.x) && threadIdx.x == 0) ctl->table = 1;
}

// Steps (bands x offsets) of a block: one bit each in a thread's event mask, five in a list entry.
constexpr int kLevelSteps = 32;
constexpr int kLevelTile = 2048;                      // pixels of a block: eleven bits in a list entry

// The zero state.  As levels: no rank has reached its threshold, e = 0, and the first event is |w|
// reaching the smallest threshold.  Else zero entries, with `clear`.  Grid (ceil(n / 128), kept offsets).
template <typename T, int K>
__global__ void __launch_bounds__(128)
levels_init_kernel(LevelRecord<ucode_t<T>>* __restrict__ rec, uint2* __restrict__ masks, ucode_t<T>* __restrict__ e,
                   const code_t<T>* __restrict__ tab, size_t n, int Ls, int clear,
                   const LatentCtl* ctl) {
    constexpr int NP = (2 * K + 1) * (2 * K + 1);
    using U = ucode_t<T>;
    const size_t p = (size_t)blockIdx.x * 128 + threadIdx.x;
    if (p >= n) return;
    const size_t si = blockIdx.y, kst = (size_t)Ls * n;
    if (ctl->mode != kStateLevels) {
        U* eb = e + si * NP * kst + p;
        for (int i = 0; clear && i < NP * Ls; ++i) eb[(size_t)i * n] = 0;
        return;
    }
    LevelRecord<U> q{0, 0, 0, levels_meta<NP>(Levels{1u << (NP - 1), 0u, 0, true, true})};
    level_free_range<U>(q, 0, (U)tab[(si * n + p) * NP]);
    for (int c = 0; c < Ls; ++c) {
        const size_t o = si * kst + (size_t)c * n + p;
        store_record(rec + o, q);
        if constexpr (NP != 9) masks[o] = make_uint2(1u << (NP - 1), 0u);
        e[si * NP * kst + (size_t)c * n + p] = 0;
    }
}

// Shared memory: H [steps][tile], the first event list [steps tile] and the second [steps tile / 16].
template <typename T>
__host__ __device__ constexpr size_t levels_smem(int steps, int tile) {
    return (size_t)steps * tile * sizeof(T) + ((size_t)steps * tile + (size_t)steps * tile / 16) * sizeof(uint16_t);
}

template <typename T, typename WT, int K>
__device__ __forceinline__ void latent_levels_body(const LevelArgs<T, WT>& a, int bx, int gz, int row,
                                                   unsigned char* smem_raw) {
    using U = ucode_t<T>;
    constexpr int NP = (2 * K + 1) * (2 * K + 1);
    if (a.ctl->mode != kStateLevels) return;
    const int H = a.H, W = a.W, Ls = a.Ls, S = a.S;
    const int nt = blockDim.x, tid = threadIdx.x, lane = tid & 31;
    const TauMap tm{S, a.half};
    const int t1 = tm.t1_of_block(row);
    const int nt2 = tm.nt2(t1);
    const int c0 = gz * a.nb;
    const int nb = min(a.nb, Ls - c0);
    const int tile = a.Ty * W, cap = nb * nt2 * tile;
    T* Hs = reinterpret_cast<T*>(smem_raw);                           // [nb][nt2][tile]
    uint16_t* list1 = reinterpret_cast<uint16_t*>(Hs + cap);
    uint16_t* list2 = list1 + cap;
    __shared__ int cnt[2];
    const int y0 = bx * a.Ty;
    const int npix = min(a.Ty, H - y0) * W;
    const uint32_t n = (uint32_t)H * W;
    const int side = 2 * S + 1;
    const LatentGrid<T> gr = *a.grid;
    const int Wp = W + 2 * S;
    const LevelPoint<T>* pt = a.pt + (size_t)c0 * H * Wp;
    const size_t kst = (size_t)Ls * n;                                // records of one offset
    const size_t s0i = (size_t)tm.s_index(t1, tm.t2_of(t1, 0));       // kept offsets of a row are consecutive
    LevelRecord<U>* rec = a.rec + s0i * kst + (size_t)c0 * n;
    if (tid < 2) cnt[tid] = 0;
    __syncthreads();
    // every step: the linear stretches; events to list1
    const int t2first = tm.t2_of(t1, 0);
    const int gap = !a.half && t1 == 0 ? S : nt2;                     // the offsets skip tau2 = 0 there
    for (int base = 0; base < npix; base += nt) {
        const int p = base + tid;
        uint32_t ev = 0;                                              // steps with an event
        if (p < npix) {
            const int r = a.Ty == 1 ? 0 : p / W, x = p - r * W, y = y0 + r;
            const uint32_t pix = (uint32_t)y * W + x;
            const LevelPoint<T>* pu = pt + ((size_t)y * Wp + S + x);
            const LevelPoint<T>* pr = pt + ((size_t)wrap1(y - t1, H) * Wp + S + x - t2first);
            T* Hp = Hs + p;
            uint32_t bit = 1u;
            for (int b = 0; b < nb; ++b, pu += (size_t)H * Wp, pr += (size_t)H * Wp) {
                const LevelPoint<T> u = load_point(pu);
                for (int part = 0; part < nt2; part += gap) {         // one part but for that skip
                    const LevelPoint<T>* pv = pr - part - (part ? 1 : 0);
                    const LevelRecord<U>* rb = rec + (size_t)part * kst + (size_t)b * n + pix;
                    // D steps whose records are loaded together
                    auto batch = [&](auto dd) {
                        constexpr int D = decltype(dd)::value;
                        LevelRecord<U> q[D];
                        LevelPoint<T> v[D];
#pragma unroll
                        for (int i = 0; i < D; ++i) {
                            q[i] = load_record(rb);
                            rb += kst;
                        }
#pragma unroll
                        for (int i = 0; i < D; ++i) v[i] = load_point(pv - i);
                        pv -= D;
#pragma unroll
                        for (int i = 0; i < D; ++i) {
                            const T delta = u.x - v[i].x;
                            const U w1 = v[i].after - u.after, w0 = v[i].before - u.before;
                            if (level_due<U>(q[i], w0, w1, delta < T(0), delta > T(0), big_move(delta, gr.g))) ev |= bit;
                            const U t = q[i].alpha + (q[i].meta & 31u) * (v[i].z - u.z);
                            *Hp = latent_h<NP>(delta, signed_of(t), gr.g);
                            Hp += tile;
                            bit <<= 1;
                        }
                    };
                    int left = part + gap < nt2 ? gap : nt2 - part;
                    for (; left >= 4; left -= 4) batch(std::integral_constant<int, 4>{});
                    if (left == 3) batch(std::integral_constant<int, 3>{});
                    else if (left == 2) batch(std::integral_constant<int, 2>{});
                    else if (left == 1) batch(std::integral_constant<int, 1>{});
                }
            }
        }
        if (!__any_sync(0xffffffffu, ev != 0)) continue;
        int pos = __popc(ev);                                         // inclusive scan over the warp
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int up = __shfl_up_sync(0xffffffffu, pos, o);
            if (lane >= o) pos += up;
        }
        int first = 0;
        if (lane == 31) first = atomicAdd(&cnt[0], pos);
        pos += __shfl_sync(0xffffffffu, first, 31) - __popc(ev);
        for (uint32_t m = ev; m; m &= m - 1) list1[pos++] = (uint16_t)(p | (lowest_bit(m) - 1) << 11);
    }
    __syncthreads();
    int todo = cnt[0];
    if (todo > 0) {
        const uint16_t* src = list1;
        const int per_nt2 = 65536 / nt2 + 1, per_w = 65536 / W + 1;
        // one (pixel, step) pair: the event, then its H_tau
        auto pair = [&](int item, bool grow) {
            // quotients by multiplication: steps < 32, and more than one row only of less than 128 pixels
            const int p = item & (kLevelTile - 1), step = item >> 11, b = (step * per_nt2) >> 16, jt = step - b * nt2;
            const int r = a.Ty == 1 ? 0 : (p * per_w) >> 16, x = p - r * W, y = y0 + r;
            const uint32_t pix = (uint32_t)y * W + x;
            const size_t o = (size_t)b * n + pix;
            uint2* mp = NP == 9 ? nullptr : a.masks + (s0i + jt) * kst + (size_t)c0 * n + o;
            LevelRecord<U>* rp = rec + jt * kst + o;
            LevelRecord<U> q = load_record(rp);
            const uint2 mk = NP == 9 ? make_uint2(0u, 0u) : *mp;
            const LevelPoint<T>* pb = pt + (size_t)b * H * Wp + S + x;
            const LevelPoint<T> u = load_point(pb + (size_t)y * Wp);
            const LevelPoint<T> v = load_point(pb + ((ptrdiff_t)wrap1(y - t1, H) * Wp - tm.t2_of(t1, jt)));
            const T delta = u.x - v.x;
            const U w1 = v.after - u.after, w0 = v.before - u.before;
            const U s0 = q.alpha + (q.meta & 31u) * w0;
            Levels l = levels_of<NP>(q.meta, mk);
            const bool big = big_move(delta, gr.g);
            const code_t<T>* Pc = a.tab + ((s0i + jt) * n + pix) * NP - 1;
            auto P = [&](int k) { return k == 0 ? U(0) : (U)__ldg(Pc + k); };
            if (grow) {
                if (!level_grow<NP, U>(l, q, w0, w1, big, P)) return false;
            } else {
                U* ep = a.e + (s0i + jt) * NP * kst + (size_t)c0 * n + o;
                level_event<NP, U>(
                    l, q, w0, w1, delta < T(0), big, P, [&](int pl) { return ep[(size_t)pl * kst]; },
                    [&](int pl, U e) { ep[(size_t)pl * kst] = e; });
            }
            store_record(rp, q);
            if constexpr (NP != 9) *mp = make_uint2(l.E, l.G);
            const U s1 = q.alpha + (q.meta & 31u) * w1;
            Hs[step * tile + p] = latent_h<NP>(delta, signed_of(2 * s1 - s0), gr.g);
            return true;
        };
        if (todo <= cap / 16) {
            for (int i0 = tid - lane; i0 < todo; i0 += nt) {
                const bool has = i0 + lane < todo;
                const int item = has ? src[i0 + lane] : 0;
                const bool left = has && !pair(item, true);
                const uint32_t m = __ballot_sync(0xffffffffu, left);
                if (m == 0) continue;
                int first = 0;
                if (lane == 0) first = atomicAdd(&cnt[1], __popc(m));
                first = __shfl_sync(0xffffffffu, first, 0);
                if (left) list2[first + __popc(m & ((1u << lane) - 1u))] = (uint16_t)item;
            }
            __syncthreads();
            todo = cnt[1];
            src = list2;
        }
        for (int i = tid; i < todo; i += nt) pair(src[i], false);
        __syncthreads();
    }
    for (int p = tid; p < npix; p += nt) {
        const int r = a.Ty == 1 ? 0 : p / W, x = p - r * W;
        for (int b = 0; b < nb; ++b) {
            const T* hp = Hs + (size_t)b * nt2 * tile + r * W;
            T A = T(0), V = T(0);
            int xv = wrap1(x + t2first, W);
            for (int jt = 0; jt < nt2; ++jt) {
                if (jt == gap) xv = xv + 1 == W ? 0 : xv + 1;
                A += hp[x];
                V += hp[xv];
                hp += tile;
                xv = xv + 1 == W ? 0 : xv + 1;
            }
            const size_t o = (size_t)(c0 + b) * 2 * side * n + (size_t)y0 * W + p;
            a.planes[o + (size_t)(t1 + S) * n] = A;
            a.planes[o + (size_t)(side + t1 + S) * n] = V;
        }
    }
}

// ---- the forms of the state -------------------------------------------------------------------
// The conversions are exact and in place: the thread of a (tau, pixel) reads every word of one
// (tau, c, m) before it writes any, and no other thread touches those words.  Each launch looks at the
// state on the device and does nothing where that does not call for it; `work` runs of window_run
// pixels of one kept offset are shared out over the blocks, a few per SM, so that such a launch costs a few
// microseconds whatever the problem's size.  The ranks of a thread lie in planes of their own, so a
// thread takes its entries through a column of shared memory, and the planes are read and written in
// whole rows.

// Blocks of a conversion per SM.  Bound by the latency of its scattered reads: the caps trade registers
// (unbounded 227 for 25 entries in FP32, two blocks) for blocks.
template <typename T, int K>
__host__ __device__ constexpr int window_resident() { return sizeof(T) == 8 ? 4 : (K == 1 ? 6 : 4); }

// Threshold codes of a window, ascending, each with its patch index in the low 5 bits.
template <typename T, typename WT, int K>
__device__ __forceinline__ void window_keys(const WT* __restrict__ om, int y, int x, int H, int W, T coef, T ig, T* mus,
                                            typename grid_code<T>::utype (&key)[(2 * K + 1) * (2 * K + 1)]) {
    constexpr int NP = (2 * K + 1) * (2 * K + 1);
    using U = typename grid_code<T>::utype;
    code_t<T> v[NP];
    window_codes<T, WT, K>(om, y, x, H, W, coef, ig, v, mus);
#pragma unroll
    for (int k = 0; k < NP; ++k) key[k] = ((U)v[k] << 5) | (U)k;
    sort_network<NP>(key);
}

// The pixels of a conversion: f(kept offset, pixel, tau, keys of its window); mus: see window_codes.
template <typename T, typename WT, int K, typename F>
__device__ __forceinline__ void each_window(const LevelArgs<T, WT>& a, int work, T* mus, F f) {
    constexpr int NP = (2 * K + 1) * (2 * K + 1);
    const size_t n = (size_t)a.H * a.W;
    constexpr int R = window_run<T, K>();
    const int runs = (int)((n + R - 1) / R);
    const TauMap tm{a.S, a.half};
    const T ig = a.grid->ig;
    for (int job = blockIdx.x; job < work; job += gridDim.x) {
        const int si = job / runs;
        const size_t p = (size_t)(job - si * runs) * R + threadIdx.x;
        if (p >= n) continue;
        int t1, t2;
        tau_of_state_index(si, a.S, a.half, &t1, &t2);
        ucode_t<T> key[NP];
        window_keys<T, WT, K>(a.omega + (size_t)tm.w_index(t1, t2) * n, (int)(p / a.W), (int)(p % a.W), a.H, a.W, a.coef,
                              ig, mus, key);
        f(si, p, t1, t2, key);
    }
}

// Entries s_k of levels, in the iterate type; a: the arguments that the levels were formed with.  out: the
// entries' planes, which may be those of the levels' values.
template <typename T, typename WT, int K>
__device__ __forceinline__ void write_entries(const LevelArgs<T, WT>& a, T* out, int work, T* col, T* mus) {
    using C = code_t<T>;
    using U = ucode_t<T>;
    constexpr int NP = (2 * K + 1) * (2 * K + 1), R = window_run<T, K>();
    const size_t n = (size_t)a.H * a.W, kst = (size_t)a.Ls * n, Wp = a.W + 2 * a.S, img = a.H * Wp;
    const T g = a.grid->g;
    each_window<T, WT, K>(a, work, mus, [&](int si, size_t p, int t1, int t2, const U (&key)[NP]) {
        const size_t y = p / a.W, x = p % a.W;
        const size_t po = y * Wp + a.S + x, ps = (size_t)wrap1((int)y - t1, a.H) * Wp + a.S + x - t2;
        for (int c = 0; c < a.Ls; ++c) {
            const size_t o = ((size_t)si * a.Ls + c) * n + p, e0 = (size_t)si * NP * kst + (size_t)c * n + p;
            const Levels l = levels_of<NP>(load_record(a.rec + o).meta, NP == 9 ? make_uint2(0u, 0u) : a.masks[o]);
            const U w = a.pt[c * img + ps].after - a.pt[c * img + po].after;
            C s[NP];
            int height = bits_set(l.E);
            C d = 0, sg = 0;
#pragma unroll
            for (int r = 0; r < NP; ++r) {
                if (r == 0 || ((l.E >> (r == 0 ? 0 : r - 1)) & 1u)) {
                    --height;
                    const int end = r + lowest_bit(l.E >> r) - 1;
                    sg = l.free && height == 0 ? 0 : (((l.G >> end) & 1u) ? 1 : -1);
                    d = r == 0 && l.q > 0 ? C(0) : (C)(w - a.e[e0 + (size_t)height * kst]);
                }
                s[r] = sg * (C)(key[r] >> 5) + d;
            }
#pragma unroll
            for (int r = 0; r < NP; ++r) col[(key[r] & 31u) * R] = (T)s[r] * g;
#pragma unroll
            for (int k = 0; k < NP; ++k)                  // see latent_bound::entry
                out[e0 + (size_t)k * kst] = SymBound<T>::of(mus[k * R]).clamp(col[k * R]);
        }
    });
}

// Levels -> entries in place, where the coming calls want entries (want below kStateLevels), the grid does
// not carry their inputs, or the weights have changed since the levels were formed (old: the arguments
// from before).  The entries are then those of a run on the current weights, or to be looked at; with
// want = kStateEntries or off the grid they go on in the iterate type's arithmetic.
template <typename T, typename WT, int K>
__global__ void __launch_bounds__(window_run<T, K>(), window_resident<T, K>())
levels_to_entries_kernel(LevelArgs<T, WT> now, LevelArgs<T, WT> old, int work, int want) {
    constexpr int NP = (2 * K + 1) * (2 * K + 1);
    constexpr int R = window_run<T, K>();
    __shared__ T stage[2 * NP * R];
    if (now.ctl->mode != kStateLevels || !(now.ctl->was || want < kStateLevels || !now.ctl->fit)) return;
    const LevelArgs<T, WT> a = now.ctl->was ? old : now;
    write_entries<T, WT, K>(a, reinterpret_cast<T*>(a.e), work, stage + threadIdx.x, stage + NP * R + threadIdx.x);
    if (last_block(now.ctl, gridDim.x) && threadIdx.x == 0) {
        now.ctl->mode = want == kStateEntries || !now.ctl->fit ? kStateEntries : now.ctl->was ? kStateGiven : kStateGrid;
        now.ctl->was = 0;
    }
}

// The state's entries to another buffer, whichever form it is in; it stays what it is.  words: entries.
template <typename T, typename WT, int K>
__global__ void __launch_bounds__(window_run<T, K>(), window_resident<T, K>())
save_entries_kernel(LevelArgs<T, WT> now, LevelArgs<T, WT> old, T* out, size_t words, int work) {
    constexpr int NP = (2 * K + 1) * (2 * K + 1);
    constexpr int R = window_run<T, K>();
    __shared__ T stage[2 * NP * R];
    if (now.ctl->mode == kStateLevels) {
        const LevelArgs<T, WT> a = now.ctl->was ? old : now;
        write_entries<T, WT, K>(a, out, work, stage + threadIdx.x, stage + NP * R + threadIdx.x);
        return;
    }
    const T* e = reinterpret_cast<const T*>(now.e);
#pragma unroll 8
    for (size_t i = (size_t)blockIdx.x * R + threadIdx.x; i < words; i += (size_t)gridDim.x * R) out[i] = e[i];
}

// The codes of the NP entries at eb, in the order of the keys (col: the thread's column of shared memory);
// false if one is above its threshold's code, or neither on the grid nor at its threshold (mus).
template <typename T, int NP, int R>
__device__ __forceinline__ bool entry_codes(const T* eb, size_t kst, T ig, const ucode_t<T> (&key)[NP], T* col,
                                            const T* mus, code_t<T> (&s)[NP]) {
    bool ok = true;
#pragma unroll
    for (int k = 0; k < NP; ++k) col[k * R] = eb[(size_t)k * kst];
#pragma unroll
    for (int r = 0; r < NP; ++r) {
        const T e = col[(key[r] & 31u) * R], v = e * ig, lim = (T)(key[r] >> 5);
        ok = ok && v >= -lim && v <= lim && (v == trunc(v) || (e < T(0) ? -e : e) == mus[(key[r] & 31u) * R]);
        s[r] = to_code(v);
    }
    return ok;
}

// Whether given entries are those of a run on the current weights, which the update on the grid and the
// levels need: on the grid, |s| <= mu, and 1-Lipschitz in mu, the state of a stop operator.
template <typename T, typename WT, int K>
__global__ void __launch_bounds__(window_run<T, K>(), window_resident<T, K>())
entries_check_kernel(LevelArgs<T, WT> a, int work) {
    using C = code_t<T>;
    using U = typename grid_code<T>::utype;
    constexpr int NP = (2 * K + 1) * (2 * K + 1);
    if (a.ctl->mode != kStateGiven) return;
    const size_t n = (size_t)a.H * a.W, kst = (size_t)a.Ls * n;
    const T ig = a.grid->ig;
    volatile int* off = &a.ctl->off;
    constexpr int R = window_run<T, K>();
    __shared__ T stage[2 * NP * R];
    T *col = stage + threadIdx.x, *mus = col + NP * R;
    each_window<T, WT, K>(a, work, mus, [&](int si, size_t p, int, int, const U (&key)[NP]) {
        for (int c = 0; c < a.Ls && !*off; ++c) {
            C s[NP];
            bool ok = entry_codes<T, NP, R>(reinterpret_cast<const T*>(a.e + (size_t)si * NP * kst + (size_t)c * n + p), kst, ig,
                                         key, col, mus, s);
#pragma unroll
            for (int r = 1; r < NP; ++r) {
                const C dm = (C)(key[r] >> 5) - (C)(key[r - 1] >> 5), ds = s[r] - s[r - 1];
                ok = ok && ds <= dm && -ds <= dm;
            }
            if (!ok) *off = 1;
        }
    });
    if (last_block(a.ctl, gridDim.x) && threadIdx.x == 0) {
        a.ctl->mode = *off ? kStateEntries : kStateGrid;
        *off = 0;
    }
}

// Entries of a run on the current weights -> levels.
template <typename T, typename WT, int K>
__global__ void __launch_bounds__(window_run<T, K>(), window_resident<T, K>())
entries_to_levels_kernel(LevelArgs<T, WT> a, int work) {
    using C = code_t<T>;
    using U = typename grid_code<T>::utype;
    constexpr int NP = (2 * K + 1) * (2 * K + 1);
    if (a.ctl->mode != kStateGrid) return;
    const size_t n = (size_t)a.H * a.W, kst = (size_t)a.Ls * n, Wp = a.W + 2 * a.S, img = a.H * Wp;
    const T ig = a.grid->ig;
    constexpr int R = window_run<T, K>();
    __shared__ T stage[2 * NP * R];
    T *col = stage + threadIdx.x, *mus = col + NP * R;
    each_window<T, WT, K>(a, work, mus, [&](int si, size_t p, int t1, int t2, const U (&key)[NP]) {
        const size_t y = p / a.W, x = p % a.W;
        const size_t po = y * Wp + a.S + x, ps = (size_t)wrap1((int)y - t1, a.H) * Wp + a.S + x - t2;
        for (int c = 0; c < a.Ls; ++c) {
            U* ob = a.e + (size_t)si * NP * kst + (size_t)c * n + p;
            C s[NP];
            entry_codes<T, NP, R>(reinterpret_cast<const T*>(ob), kst, ig, key, col, mus, s);
            U su[NP], mu[NP];
#pragma unroll
            for (int r = 0; r < NP; ++r) {
                su[r] = (U)s[r];
                mu[r] = key[r] >> 5;
            }
            const U w = a.pt[c * img + ps].after - a.pt[c * img + po].after;
            Levels l;
            LevelRecord<U> q;
            levels_from_entries<NP, U>(su, mu, w, l, q, [&](int pl, U e) { ob[(size_t)pl * kst] = e; });
            const size_t o = ((size_t)si * a.Ls + c) * n + p;
            store_record(a.rec + o, q);
            if constexpr (NP != 9) a.masks[o] = make_uint2(l.E, l.G);
        }
    });
    if (last_block(a.ctl, gridDim.x) && threadIdx.x == 0) a.ctl->mode = kStateLevels;
}

// Before the weights change (words: those of the weights, 16 bytes each): levels stay readable through
// the weights and the grid that they were formed with, kept in `was`; entries have to be looked at again.  The grid is then
// that for weights up to 1, which fuse_weights gives; given weights set their own.
template <typename T>
__global__ void __launch_bounds__(256)
weights_change_kernel(const uint4* __restrict__ omega, uint4* __restrict__ was, size_t words, LatentGrid<T>* grid,
                      LatentCtl* ctl) {
    const bool keep = ctl->mode == kStateLevels && !ctl->was;
    if (keep)
        for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < words; i += (size_t)gridDim.x * blockDim.x)
            was[i] = omega[i];
    if (last_block(ctl, gridDim.x) && threadIdx.x == 0) {
        if (keep) {
            grid[1] = grid[0];
            ctl->was = 1;
        }
        if (ctl->mode == kStateGrid) ctl->mode = kStateGiven;
        ctl->table = 0;
        grid[0] = grid[2];
    }
}

// The state that a solve starts with, and whether the grid carries its inputs: their size is the rms of
// the `count` samples of Y_l that S keeps (mask, over n pixels, or all), divided by `gain`, the most that B and E
// can have raised that of X.  Block row y of the launch is problem y.  The sums are formed in the same order
// on every device.  Latency-bound: a thread has its eight samples in flight at once, a problem of one block
// (8192 samples) needs no second round, and the problems of a batch share a launch (11 problems of 32
// to 360: 15 us of a call, 105 with a launch each).
template <typename T>
struct BeginArgs {
    const T* Y;
    const uint8_t* mask;
    size_t count, n;
    double gain, coef;
    const LatentGrid<T>* grid;
    LatentCtl* ctl;
    int cold, want;
};
template <typename T>
struct BeginBatch {
    static constexpr int kMost = 32;                  // problems of a launch: 2.6 KB of arguments
    BeginArgs<T> a[kMost];
};
inline __host__ __device__ int begin_blocks(size_t count) {
    const size_t need = (count + kBeginSamples - 1) / kBeginSamples;
    return (int)(need < 1 ? 1 : need < (size_t)kBeginBlocks ? need : (size_t)kBeginBlocks);
}
template <typename T>
__global__ void __launch_bounds__(1024) latent_begin_kernel(const __grid_constant__ BeginBatch<T> batch) {
    constexpr int R = kBeginSamples / 1024;
    __shared__ double red[2][32];
    const BeginArgs<T>& a = batch.a[blockIdx.y];
    const int blocks = begin_blocks(a.count), tid = threadIdx.x;
    if ((int)blockIdx.x >= blocks) return;
    const double g = (double)a.grid->g, wmax = (double)a.grid->wmax;
    const int mode = a.ctl->mode;
    double sq = 0.0, seen = 0.0;
    // the block's sums, in thread 0
    auto reduce = [&]() {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            sq += __shfl_down_sync(0xffffffffu, sq, o);
            seen += __shfl_down_sync(0xffffffffu, seen, o);
        }
        __syncthreads();
        if ((tid & 31) == 0) {
            red[0][tid >> 5] = sq;
            red[1][tid >> 5] = seen;
        }
        __syncthreads();
        if (tid < 32) {
            sq = red[0][tid];
            seen = red[1][tid];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                sq += __shfl_down_sync(0xffffffffu, sq, o);
                seen += __shfl_down_sync(0xffffffffu, seen, o);
            }
        }
    };
    for (size_t i0 = (size_t)blockIdx.x * kBeginSamples; i0 < a.count; i0 += (size_t)blocks * kBeginSamples) {
        T v[R], part = T(0);
        int kept = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const size_t i = i0 + r * 1024 + tid;
            const bool keep = i < a.count && (!a.mask || a.mask[i % a.n]);
            v[r] = keep ? a.Y[i] : T(0);
            kept += keep;
        }
#pragma unroll
        for (int r = 0; r < R; ++r) part += v[r] * v[r];
        sq += (double)part;
        seen += (double)kept;
    }
    reduce();
    if (blocks > 1) {
        if (tid == 0) {
            a.ctl->part[blockIdx.x] = sq;
            a.ctl->seen[blockIdx.x] = seen;
        }
        if (!last_block(a.ctl, blocks)) return;
        sq = tid < blocks ? __ldcg(&a.ctl->part[tid]) : 0.0;
        seen = tid < blocks ? __ldcg(&a.ctl->seen[tid]) : 0.0;
        reduce();
    }
    if (tid != 0) return;
    const double top = ldexp(g, grid_code<T>::B);
    // thresholds that are all zero leave the entries zero, on the grid of anything
    const bool fit = wmax <= 1e308 && (a.coef * wmax == 0.0 || top * a.gain <= sqrt(sq / seen));
    a.ctl->fit = fit;
    if (a.cold) {
        a.ctl->mode = fit || a.want == kStateGiven ? a.want : kStateEntries;
        a.ctl->was = 0;
    } else if (mode != kStateLevels && (a.want == kStateEntries || !fit)) {
        a.ctl->mode = kStateEntries;
    }
}

// grid->wmax = the largest of n weights, infinite if one is not a finite number >= 0 (zeroed before; the
// order of non-negative floating-point values is that of their bit patterns); then the grid from it.
template <typename T, typename WT>
__global__ void __launch_bounds__(256) wmax_kernel(const WT* __restrict__ w, size_t n, LatentGrid<T>* grid) {
    T m = T(0);
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const T v = (T)wload(w + i);
        if (v > m) m = v;
        if (!(v >= T(0))) m = (T)INFINITY;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = tmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) {
        if constexpr (sizeof(T) == 4) atomicMax(reinterpret_cast<int*>(&grid->wmax), __float_as_int(m));
        else atomicMax(reinterpret_cast<long long*>(&grid->wmax), __double_as_longlong(m));
    }
}
template <typename T>
__global__ void grid_kernel(LatentGrid<T>* grid, T coef) { *grid = latent_grid(coef, grid->wmax); }

template <typename T, typename WT, int K>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 8 : 6) latent_levels_kernel(LevelArgs<T, WT> a) {
    extern __shared__ __align__(16) unsigned char smem_levels[];
    latent_levels_body<T, WT, K>(a, blockIdx.x, blockIdx.y, blockIdx.z, smem_levels);
}

// Batched forms over the segment table (see latent_tma_batch_kernel): the points, the latent pass.
template <typename T, typename WT>
__global__ void __launch_bounds__(256)
points_batch_kernel(const LevelArgs<T, WT>* __restrict__ args, const Segment* __restrict__ seg, int nseg, int first) {
    int prob, bx, by, bz;
    segment_of_block(seg, nseg, blockIdx.x, &prob, &bx, &by, &bz);
    const LevelArgs<T, WT>& a = args[prob];
    const int row = bx * 8 + (threadIdx.x >> 5);
    if (row < a.H * a.Ls && a.ctl->mode == kStateLevels)
        points_row<T>(a.X, const_cast<LevelPoint<T>*>(a.pt), a.W, a.S, a.grid, first, row, threadIdx.x & 31);
}

template <typename T, typename WT, int K>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 8 : 6)
latent_levels_batch_kernel(const LevelArgs<T, WT>* __restrict__ args, const Segment* __restrict__ seg, int nseg) {
    extern __shared__ __align__(16) unsigned char smem_levels[];
    int prob, bx, by, bz;
    segment_of_block(seg, nseg, blockIdx.x, &prob, &bx, &by, &bz);
    const LevelArgs<T, WT> a = args[prob];
    latent_levels_body<T, WT, K>(a, bx, by, bz, smem_levels);
}

}  // namespace fuse
