// Work items of the network's convolution and weight-gradient kernels: which
// tiles of 128 pixels a CTA takes in turn.  Shared by the kernels and the host.
#pragma once

#include <stdint.h>

#include <algorithm>

#if defined(__CUDACC__)
#define GCMG_HD __host__ __device__ __forceinline__
#else
#define GCMG_HD inline
#endif

namespace gcmg_cnn_tiles {

constexpr int kTile = 128;            // pixels of a tile (M of the MMAs)

struct Geo {
    int npix, Hp, Wp, H, W, P;
    int gs;        // rows between channel groups (npix plus zero guard rows on both sides)
};

// An item: cnt tiles, tile k's first pixel at q + k * dil * Wp; it reads the
// three pixel rows at that pixel and dil * Wp before and after it (dil more
// pixels at either end).
struct TileItem {
    long q;
    int b, row, col;   // image; flat: row 0, col = the tile's place in the image's flat range
    int cnt;           // tiles
    int width;         // pixels of a tile in use
};

// Chains (flat = 0): item = ((image * cols + column) * res + residue) * parts +
// part; its tiles are rows residue + (part * len + k) * dil of the image, 128
// columns each, and share their input rows.  Flat (flat = tiles an image): the
// image's rows one after the other, its borders' columns between them, in tiles of
// 128 pixels, one an item.
struct Tiles {
    int dil, cols, res, parts, len, items, flat;
    int grid;   // CTAs: CTA c takes items c, c + grid, ...
    // false: the part lies past the chain's end
    GCMG_HD bool item(const Geo &g, int t, TileItem *o) const {
        if (flat) {
            const int span = g.H * g.Wp - 2 * g.P;
            o->b = t / flat;
            o->row = 0;
            o->col = t % flat * kTile;
            o->cnt = 1;
            o->width = span - o->col < kTile ? span - o->col : kTile;
            o->q = ((long)o->b * g.Hp + g.P) * g.Wp + g.P + o->col;
            return true;
        }
        const int part = t % parts;
        t /= parts;
        const int r = t % res;
        t /= res;
        o->b = t / cols;
        o->col = t % cols * kTile;
        o->width = g.W - o->col < kTile ? g.W - o->col : kTile;
        const int n = (g.H - r + dil - 1) / dil, j0 = part * len;
        o->row = r + j0 * dil;
        o->cnt = n - j0 < len ? n - j0 : len;
        o->q = ((long)o->b * g.Hp + g.P + o->row) * g.Wp + g.P + o->col;
        return o->cnt > 0;
    }
    // image coordinates of pixel x of the item's tile k; false: none there
    GCMG_HD bool at(const Geo &g, const TileItem &o, int k, int x, int *i, int *j) const {
        if (flat) {
            *i = (o.col + x) / g.Wp;
            *j = (o.col + x) - *i * g.Wp;
            return *i < g.H && *j < g.W;
        }
        *i = o.row + k * dil;
        *j = o.col + x;
        return *j < g.W;
    }
};

// The items and the grid for at most per_sm CTAs on each of sms SMs.  A part of n
// tiles loads n + 2 segments, a CTA works through its items one after the other,
// an SM's CTAs share its tensor cores and a CTA costs `cta` tiles by itself, so a
// launch of `rounds` items a CTA takes about rounds x (n + 1) + tiles / sms + cta x
// CTAs tiles' time.  Chains cut into parts that give every CTA about three, of at
// least 4 tiles; where that is less (12 tiles a CTA or fewer), the length of 1 to
// 16 and the number of CTAs with the least such time.  Flat where that is less
// again: images much narrower than their last tile's end, whose chains compute
// columns that are not there.  Measured, us forward / backward, with parts of at
// least 4 tiles and no flat form against so: one image of 64^2, dilations 1, 86 /
// 227 -> 62 / 163; 129^2, default dilations, 83 / 224 -> 68 / 202; 16 of 128 x 16,
// dilations up to 5, 120 / 343 -> 71 / 228; 64 of 32^2, dilations 1, 120 / 340 -> 74 / 254.
inline Tiles make_tiles(const Geo &g, int batch, int dil, int sms, int per_sm, double cta) {
    Tiles h{};
    h.dil = dil;
    h.cols = (g.W + kTile - 1) / kTile;
    h.res = std::min(dil, g.H);
    const int nmax = (g.H + dil - 1) / dil;   // tiles of the longest chain
    const int64_t chains = (int64_t)batch * h.cols * h.res, slots = (int64_t)sms * per_sm;
    double best = 1e300;
    // parts of len tiles (flat: tiles an image), in as few rounds as the slots
    // allow, or more where CTAs cost something
    auto consider = [&](int len, int flat, bool fewer) {
        const int parts = flat ? 1 : (nmax + len - 1) / len;
        const int64_t items = flat ? (int64_t)batch * flat : chains * parts;
        const double tiles = flat ? (double)items : (double)batch * h.cols * g.H;
        const int64_t least = (items + slots - 1) / slots;
        for (int64_t r = least; r <= least + (fewer && cta > 0 ? 32 : 0); r++) {
            const int64_t grid = r == least ? std::min(items, slots) : (items + r - 1) / r;
            const double t = (double)(r * (len + 1)) + tiles / sms + cta * (double)grid;
            if (t >= best) continue;
            best = t;
            h.flat = flat;
            h.parts = parts;
            h.len = flat ? 1 : (nmax + parts - 1) / parts;
            h.items = (int)items;
            h.grid = (int)grid;
        }
    };
    const int64_t want = std::max<int64_t>(1, 3 * slots / chains);
    const int len = (int)((nmax + want - 1) / want);
    if (len >= 4) consider(len, 0, false);
    else
        for (int l = 1; l <= 16; l++) consider(l, 0, true);
    consider(1, (int)(((int64_t)g.H * g.Wp - 2 * g.P + kTile - 1) / kTile), true);
    return h;
}

}  // namespace gcmg_cnn_tiles
