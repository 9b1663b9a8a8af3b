// tilekey.cuh -- sort keys of the pairs: a tile's key within its view, and the
// counts of a record's lowest key digit.  Host and device code, plain C++.
#pragma once

#include <stdint.h>

#include "../../include/dashgs.h"

#ifdef __CUDACC__
#define DG_HD __host__ __device__ __forceinline__
#else
#define DG_HD inline
#endif

namespace dg {

struct TileGrid {
    int n;
    int TX[DG_MAX_VIEWS], TY[DG_MAX_VIEWS];
    int off[DG_MAX_VIEWS + 1];  // first global tile id of each view
};

constexpr int BIN_MAXPASS = 6;  // digits of a key

// Tile keys: tile row << xbits | tile column, so that the lowest digits are the
// column's and a record's counts of them take one addition per column of its
// mask (or two for a rect of any size, into a difference array).
// Linear keys, row * TX + column, take the grids of at most 256 tiles a view, which
// are one digit then, and those for which the other form fails: with every view one
// tile wide there is no column digit, and columns and rows whose maxima come from
// different views may need more than 31 bits together (a view's own grid has at
// most 2^30 tiles).  A record's lowest digits are then counted run by run, a row's
// tiles at once (tile by tile, by one thread per record, the counts took 40 of the 50
// us of the record kernel on 5k records and 120 tiles).
struct TileKey {
    int linear;
    int xbits, bits;
    int npass;
    int shift[BIN_MAXPASS], width[BIN_MAXPASS];  // digits
};

inline TileKey tile_key(const TileGrid& tg)
{
    TileKey k{};
    int yb = 0, lb = 0;
    for (int v = 0; v < tg.n; ++v) {
        while ((1ll << k.xbits) < tg.TX[v]) ++k.xbits;
        while ((1ll << yb) < tg.TY[v]) ++yb;
        while ((1ll << lb) < (long long)tg.TX[v] * tg.TY[v]) ++lb;
    }
    k.bits = k.xbits + yb;
    k.linear = lb <= 8 || k.xbits == 0 || k.bits > 31;
    if (k.linear) {
        k.bits = lb > 0 ? lb : 1;
        k.xbits = 0;
    }
    // the column's digits, then the row's (a grid of one row has none there), or the linear key's
    for (int part = 0; part < 2; ++part) {
        const int b = k.linear ? (part ? 0 : k.bits) : part ? yb : k.xbits, n = (b + 7) / 8, from = part ? k.xbits : 0;
        for (int i = 0, at = 0; i < n; ++i) {
            const int w = (b - at + (n - i) - 1) / (n - i);
            k.shift[k.npass] = from + at;
            k.width[k.npass++] = w;
            at += w;
        }
    }
    return k;
}

// Key distance of neighbouring tile rows.
DG_HD uint32_t key_row(int linear, int xbits, int TX) { return linear ? (uint32_t)TX : 1u << xbits; }
// Tile of a key within its view (row * TX + column).
DG_HD uint32_t key_tile(uint32_t key, int linear, int xbits, uint32_t TX)
{
    return linear ? key : (key >> xbits) * TX + (key & ((1u << xbits) - 1u));
}

// Counts of the lowest digit of `len` consecutive keys from `a` on, `times` each:
// cyclic through the digit's values, as a difference array with the full cycles apart.
template <class Diff, class Cycles>
DG_HD void count_run(uint32_t a, uint32_t len, uint32_t times, int width, Diff diff, Cycles cycles)
{
    const uint32_t dm = (1u << width) - 1u, rem = len & dm, lo = a & dm, hi = lo + rem;
    if (len > dm) cycles((len >> width) * times);
    if (rem) {
        diff(lo, (int)times);
        if (hi != dm + 1u) diff(hi & dm, -(int)times);
        if (hi > dm + 1u) diff(0u, (int)times);
    }
}

// Index of the lowest set bit of m (m != 0).
DG_HD int first_bit(uint32_t m)
{
#ifdef __CUDA_ARCH__
    return __ffs((int)m) - 1;
#else
    int i = 0;
    while (!((m >> i) & 1u)) ++i;
    return i;
#endif
}

// The same for a record's tiles under linear keys: the mask's bits row by row (lo,
// hi: eight rows of eight columns), or a rect of w x h tiles.
template <class Diff, class Cycles>
DG_HD void count_linear_mask(uint32_t key0, int TX, uint32_t lo, uint32_t hi, int width, Diff diff, Cycles cycles)
{
    for (int y = 0; lo | hi; ++y) {
        uint32_t m = lo & 255u;
        lo = (lo >> 8) | (hi << 24);
        hi >>= 8;
        while (m) {  // (a row of a tight mask is one run)
            const int x = first_bit(m), len = first_bit(~(m >> x));
            count_run(key0 + (uint32_t)(y * TX + x), (uint32_t)len, 1u, width, diff, cycles);
            m &= m + (1u << x);
        }
    }
}
template <class Diff, class Cycles>
DG_HD void count_linear_rect(uint32_t key0, int TX, uint32_t w, uint32_t h, int width, Diff diff, Cycles cycles)
{
    if (w == (uint32_t)TX) {  // whole rows follow one another
        count_run(key0, w * h, 1u, width, diff, cycles);
        return;
    }
    for (uint32_t y = 0; y < h; ++y) count_run(key0 + y * (uint32_t)TX, w, 1u, width, diff, cycles);
}

// A record's tiles in three words: the corner x0 | y0 << 16, then a mask of 8 x 8
// tiles (a whole rect that fits one, too) or a larger rect's size.  A mask's low word
// is never 0 (one with four empty rows starts four rows further down); with a low word
// of 0 the last word is (w - 1) | (h - 1) << bits of a column, which is 31 bits at
// most in a view's grid and 0 only where there are no tiles (1 x 1 is a mask).
// The record's index keeps all 32 bits of its own word.
struct RecTiles { uint32_t corner, lo, hi; };

DG_HD int column_bits(int TX)
{
    int b = 0;
#ifdef __CUDA_ARCH__
    b = TX > 1 ? 32 - __clz(TX - 1) : 0;
#else
    while ((1ll << b) < TX) ++b;
#endif
    return b;
}

DG_HD RecTiles pack_tiles(uint32_t x0, uint32_t y0, uint32_t w, uint32_t h, uint32_t lo, uint32_t hi, int TX)
{
    if ((lo | hi) == 0 && w <= 8 && h <= 8) {
        const uint32_t rows = 0x01010101u * ((1u << w) - 1u);
        lo = h >= 4 ? rows : rows & ((1u << (8 * h)) - 1u);
        hi = h <= 4 ? 0u : h == 8 ? rows : rows & ((1u << (8 * (h - 4))) - 1u);
    }
    RecTiles r;
    if ((lo | hi) != 0) {
        const bool down = lo == 0;
        r.corner = x0 | ((y0 + (down ? 4u : 0u)) << 16);
        r.lo = down ? hi : lo;
        r.hi = down ? 0u : hi;
    } else {
        r.corner = x0 | (y0 << 16);
        r.lo = 0;
        r.hi = w == 0 || h == 0 ? 0u : (w - 1u) | ((h - 1u) << column_bits(TX));
    }
    return r;
}
// Size of a rect from its last word (with a low word of 0).
DG_HD uint32_t rect_width(uint32_t hi, int TX) { return hi == 0 ? 0u : (hi & ((1u << column_bits(TX)) - 1u)) + 1u; }
DG_HD uint32_t rect_height(uint32_t hi, int TX) { return hi == 0 ? 0u : (hi >> column_bits(TX)) + 1u; }

}  // namespace dg
