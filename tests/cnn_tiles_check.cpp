// Test program (built and run by tests/test_cnn_tiles.py, host only): the work
// items of the network's kernels over many shapes, dilations and numbers of
// resident CTAs.  Prints "name failures count" lines.
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "cnn_tiles.h"

using namespace gcmg_cnn_tiles;

int main() {
    long cover = 0, place = 0, bounds = 0, taps = 0, slow = 0, n = 0, flat = 0, chains = 0, split = 0;
    unsigned rng = 7;
    auto uni = [&](int lo, int hi) {
        rng = rng * 1664525u + 1013904223u;
        return lo + (int)((rng >> 8) % (unsigned)(hi - lo + 1));
    };
    for (int trial = 0; trial < 600; trial++) {
        const int H = uni(1, trial % 3 ? 40 : 150), W = trial % 4 ? uni(1, 60) : uni(100, 300);
        const int P = trial % 2 ? uni(1, 6) : uni(1, 96), dil = trial % 5 ? uni(1, P) : P, B = uni(1, 3);
        const int sms = trial % 3 ? 152 : 1, per_sm = trial % 3 == 2 ? 3 : 1;
        const double cta = trial % 2 ? 1.0 / 20 : 0.0;
        Geo g{B * (H + 2 * P) * (W + 2 * P), H + 2 * P, W + 2 * P, H, W, P, 0};
        const long guard = (long)P * g.Wp + P + kTile;   // rows before and after a channel group
        const Tiles t = make_tiles(g, B, dil, sms, per_sm, cta);
        std::vector<int> seen((size_t)g.npix, 0), pairs((size_t)9 * g.npix, 0);
        auto inside = [&](long q) {
            if (q < 0 || q >= g.npix) return false;
            const int i = (int)(q / g.Wp % g.Hp) - P, j = (int)(q % g.Wp) - P;
            return i >= 0 && i < H && j >= 0 && j < W;
        };
        for (int x = 0; x < t.items; x++) {
            TileItem it;
            if (!t.item(g, x, &it)) continue;
            for (int k = 0; k < it.cnt; k++) {
                const long q = it.q + (long)k * dil * g.Wp, lo = q - (long)dil * g.Wp - dil, hi = q + (long)dil * g.Wp + kTile - 1 + dil;
                bounds += lo < -guard || hi >= g.npix + guard || it.width < 1 || it.width > kTile;
                for (int r = 0; r < kTile; r++) {
                    int i = 0, j = 0;
                    if (!t.at(g, it, k, r, &i, &j)) continue;
                    place += q + r != ((long)it.b * g.Hp + P + i) * g.Wp + P + j || r >= it.width;
                    if (inside(q + r)) seen[q + r]++;
                }
                // the weight gradients' products: x at q + r + tap row, dz at q + r - tap column
                for (int r = 0; r < it.width; r++)
                    for (int tap = 0; tap < 9; tap++) {
                        const long o = q + r + (1 - tap % 3) * dil, xq = q + r + (long)(tap / 3 - 1) * dil * g.Wp;
                        bounds += o < -guard || o >= g.npix + guard;
                        if (inside(o) && inside(xq)) pairs[(size_t)tap * g.npix + o]++;
                    }
            }
        }
        for (long q = 0; q < g.npix; q++) {
            cover += seen[q] != (inside(q) ? 1 : 0);
            for (int tap = 0; tap < 9; tap++) {
                const long xq = q + (long)(tap / 3 - 1) * dil * g.Wp + (tap % 3 - 1) * dil;
                // same image: rows of neighbouring images are 2 P >= 2 dil apart
                taps += pairs[(size_t)tap * g.npix + q] != (inside(q) && inside(xq) ? 1 : 0);
            }
        }
        // no dearer than parts of four tiles on all SMs, than one tile an item and than the flattened rows
        const int nmax = (H + dil - 1) / dil;
        const int64_t slots = (int64_t)sms * per_sm, ch = (int64_t)B * ((W + kTile - 1) / kTile) * std::min(dil, H);
        auto time = [&](int64_t items, int len, double tiles) {
            return (double)((items + slots - 1) / slots * (len + 1)) + tiles / sms + cta * (double)std::min(items, slots);
        };
        const double rows = (double)B * ((W + kTile - 1) / kTile) * H;
        const int64_t rounds = (t.items + t.grid - 1) / t.grid, fl = B * (((int64_t)H * g.Wp - 2 * P + kTile - 1) / kTile);
        const double now = (double)(rounds * (t.len + 1)) + (t.flat ? (double)t.items : rows) / sms + cta * t.grid;
        const int64_t want = std::max<int64_t>(1, 3 * slots / ch);
        if ((nmax + want - 1) / want < 4) slow += now > time(ch * ((nmax + 3) / 4), 4, rows) || now > time(ch * nmax, 1, rows);
        slow += now > time(fl, 1, (double)fl);
        bounds += t.grid < 1 || t.grid > slots || t.grid > t.items;
        n++;
        (t.flat ? flat : t.len > 1 ? chains : split)++;
    }
    std::printf("cover %ld %ld\nplace %ld %ld\nbounds %ld %ld\ntaps %ld %ld\nslow %ld %ld\n", cover, n, place, n, bounds, n, taps, n,
                slow, n);
    std::printf("flat 0 %ld\nchains 0 %ld\nsingle 0 %ld\n", flat, chains, split);
    return cover + place + bounds + taps + slow ? 1 : 0;
}
