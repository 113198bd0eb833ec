// Host check of the level arithmetic (latent_grid.cuh): random walks of w, each step against the
// entry-by-entry update of the same thresholds.  Compiled and run by test_levels_model.py.
#define FUSE_LEVEL_FN static inline
#include "latent_grid.cuh"

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <vector>

using namespace fuse;

#define REQUIRE(c)                                                                            \
    do {                                                                                      \
        if (!(c)) { printf("NP %d trial %d step %d: %s\n", NP, trial, it, #c); return 1; }    \
    } while (0)

template <int NP>
int walk(int seed) {
    std::mt19937 r(seed);
    long events = 0, grown = 0;
    for (int trial = 0; trial < 1500; ++trial) {
        // thresholds: uniform, decades apart, tiny, or few distinct values (0 among them)
        std::vector<int> mu(NP), P(NP + 1, 0);
        const int mode = r() % 4;
        for (int& m : mu)
            m = mode == 0 ? r() % (1 << 24) : mode == 1 ? (1 << 24) >> (r() % 25) : mode == 2 ? r() % 4 : (r() % 3) * 1000000;
        std::sort(mu.begin(), mu.end());
        for (int i = 0; i < NP; ++i) P[i + 1] = P[i] + mu[i];
        std::vector<int> s(NP, 0);
        std::vector<uint32_t> planes(NP, 0x55555555u);
        planes[0] = 0;
        Levels l{1u << (NP - 1), 0u, 0, true, true};
        LevelRecord<uint32_t> rec{0, 0, 0, levels_meta<NP>(l)};
        uint32_t w = r();                             // the running sums start anywhere modulo 2^32
        planes[0] = w;
        level_free_range<uint32_t>(rec, w, (uint32_t)mu[0]);
        rec.alpha = 0u - (uint32_t)NP * w;
        double scale = std::pow(2.0, r() % 27);
        const double decay = 0.5 + (r() % 100) / 150.0;
        for (int it = 0; it < 60; ++it) {
            // random, decaying oscillation, no move (with either sign of a tiny delta), big moves
            const int kind = r() % 10;
            int dq = 0;
            bool big = false;
            if (kind == 1 && r() % 4 == 0) {
                big = true;
                dq = r() % 2 ? 1 << 26 : -(1 << 26);
            } else if (kind > 0 && kind < 4) {
                dq = (int)(((int)(r() % 2000001) - 1000000) / 1e6 * scale);
            } else if (kind > 0) {
                dq = (int)((it % 2 ? 1 : -1) * scale * (0.5 + (r() % 100) / 200.0));
                scale *= decay;
                if (scale < 1 || scale > 6e7) scale = std::pow(2.0, r() % 26);
            }
            bool up = dq < 0, down = dq > 0;
            if (dq == 0) { const int z = r() % 3; up = z == 1; down = z == 2; }
            const uint32_t w0 = w, w1 = big ? r() : w - (uint32_t)dq;
            int s0 = 0, s1 = 0;
            for (int i = 0; i < NP; ++i) {
                s0 += s[i];
                s[i] = std::min(std::max(s[i] - dq, -mu[i]), mu[i]);
                s1 += s[i];
            }
            REQUIRE(signed_of(rec.alpha + (rec.meta & 31u) * w0) == s0);
            if (level_due<uint32_t>(rec, w0, w1, up, down, big)) {
                ++events;
                bool in_range = true;
                auto pre = [&](int q) { in_range = in_range && q >= 0 && q <= NP; return (uint32_t)P[in_range ? q : 0]; };
                auto ld = [&](int p) { in_range = in_range && p >= 0 && p < NP; return in_range ? planes[p] : 0u; };
                auto st = [&](int p, uint32_t e) { in_range = in_range && p >= 0 && p < NP; if (in_range) planes[p] = e; };
                l = levels_of<NP>(rec.meta, make_uint2(l.E, l.G));
                Levels lg = l;
                LevelRecord<uint32_t> rg = rec;
                const bool g = level_grow<NP, uint32_t>(lg, rg, w0, w1, big, pre);
                level_event<NP, uint32_t>(l, rec, w0, w1, up, big, pre, ld, st);
                REQUIRE(in_range);
                if (g) {
                    ++grown;
                    REQUIRE(lg.E == l.E && lg.G == l.G && lg.q == l.q && lg.up == l.up && lg.free == l.free);
                    REQUIRE(rg.alpha == rec.alpha && rg.trig == rec.trig && rg.half == rec.half && rg.meta == rec.meta);
                }
            }
            w = w1;
            if (r() % 8 == 0) {                       // the same state formed anew from its entries
                uint32_t su[NP], mm[NP];
                for (int i = 0; i < NP; ++i) { su[i] = (uint32_t)s[i]; mm[i] = (uint32_t)mu[i]; }
                bool fits = true;
                levels_from_entries<NP, uint32_t>(su, mm, w, l, rec, [&](int p, uint32_t e) {
                    fits = fits && p >= 0 && p < NP;
                    if (fits) planes[p] = e;
                });
                REQUIRE(fits);
            }
            REQUIRE(signed_of(rec.alpha + (rec.meta & 31u) * w1) == s1);
            // every entry from the levels
            int lo = 0, height = bits_set(l.E) - 1;
            for (uint32_t E = l.E; E; E &= E - 1, --height) {
                const int hi = lowest_bit(E);
                const int sg = l.free && (E & (E - 1)) == 0 ? 0 : ((l.G >> (hi - 1)) & 1u ? 1 : -1);
                const int d = l.q > 0 && lo == 0 ? 0 : signed_of(w - planes[height]);
                for (int i = lo; i < hi; ++i) REQUIRE(sg * mu[i] + d == s[i]);
                lo = hi;
            }
            REQUIRE(lo == NP);
        }
    }
    return events > 1000 && grown > 100 ? 0 : 2;
}

int main() {
    for (int s = 1; s < 5; ++s)
        if (walk<9>(s) || walk<25>(100 + s)) return 1;
    printf("ok\n");
    return 0;
}
