"""The tile keys of the binning and the counts of their lowest digit, compiled
for the host from the library's own header: over grids of every form (one digit,
column and row digits, one column of more than 256 tiles, views whose columns and
rows need more than 31 bits together) the digits cover the key, a key leads back
to its tile, keys of one view are distinct, the counts equal an enumeration
of the record's tiles, and a record's three words lead back to its tiles."""
from __future__ import annotations

import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "tilekey.cuh"
using namespace dg;
static uint32_t rnd() { static uint32_t s = 12345u; s = s * 1664525u + 1013904223u; return s >> 8; }
int main(int argc, char** argv)
{
    TileGrid tg{};
    for (int i = 1; i + 1 < argc; i += 2) { tg.TX[tg.n] = atoi(argv[i]); tg.TY[tg.n] = atoi(argv[i + 1]); ++tg.n; }
    const TileKey k = tile_key(tg);
    if (k.npass < 1 || k.npass > BIN_MAXPASS || k.bits > 31) return 1;
    int at = 0;
    for (int p = 0; p < k.npass; ++p) {
        if (k.shift[p] != at || k.width[p] < 1 || k.width[p] > 8) return 2;
        at += k.width[p];
    }
    for (int v = 0; v < tg.n; ++v) {
        const int TX = tg.TX[v], TY = tg.TY[v];
        const uint32_t row = key_row(k.linear, k.xbits, TX);
        auto key = [&](uint32_t x, uint32_t y) { return y * row + x; };
        if ((unsigned long long)(TY - 1) * row + (TX - 1) >= (1ull << at)) return 3;  // the digits cover every key
        if (TX > 1 && row < (uint32_t)TX) return 4;
        for (int t = 0; t < 200; ++t) {
            const uint32_t x = rnd() % TX, y = rnd() % TY;
            if (key_tile(key(x, y), k.linear, k.xbits, TX) != y * (uint32_t)TX + x) return 5;
        }
        const int bins = 1 << k.width[0];
        const uint32_t dm = bins - 1u;
        // the form the record kernel counts: single digits per column, linear keys run by run
        if (k.npass > 1 && !k.linear && k.width[0] > k.xbits) return 6;  // the lowest digit is the column's
        for (int t = 0; t < 400; ++t) {
            std::vector<long long> want(bins, 0), diff(bins + 1, 0);
            long long cyc = 0;
            auto add = [&](uint32_t i, int n) { diff[i] += n; };
            auto full = [&](uint32_t n) { cyc += n; };
            const uint32_t x0 = rnd() % TX, y0 = rnd() % TY;
            const uint32_t wmax = TX - x0, hmax = TY - y0;
            const bool masked = t & 1;
            uint32_t w = 1 + rnd() % wmax, h = 1 + rnd() % (hmax < 600 ? hmax : 600);
            if (t % 8 == 0) w = wmax;
            if (w > 3000) w = 3000;
            if (masked) { w = wmax < 8 ? wmax : 8; h = hmax < 8 ? hmax : 8; }
            uint32_t lo = 0, hi = 0;
            for (uint32_t y = 0; y < h; ++y)
                for (uint32_t x = 0; x < w; ++x) {
                    if (masked) {
                        if (t % 3 == 0 ? rnd() % 3 == 0 : x >= y % 3 && x < w - y % 2) {
                            (y < 4 ? lo : hi) |= 1u << (8 * (y & 3) + x);
                        } else {
                            continue;
                        }
                    }
                    ++want[key(x0 + x, y0 + y) & dm];
                }
            {  // the record's words lead back to its tiles
                const uint32_t rw = masked ? 9 : w, rh = masked ? 9 : h;
                const RecTiles r = pack_tiles(x0 & 0xffffu, y0 & 0xffffu, rw, rh, lo, hi, TX);
                const RecTiles none = pack_tiles(x0 & 0xffffu, y0 & 0xffffu, t & 2 ? 0 : w, t & 2 ? h : 0, 0, 0, TX);
                if (none.lo || none.hi || rect_width(none.hi, TX) * rect_height(none.hi, TX)) return 8;
                const uint32_t px = r.corner & 0xffffu, py = r.corner >> 16;
                if (px != (x0 & 0xffffu)) return 9;
                unsigned long long m = (unsigned long long)lo | ((unsigned long long)hi << 32);
                if (!m && (rw > 8 || rh > 8)) {
                    if (masked && (rw > (uint32_t)TX || rh > (uint32_t)TY)) continue;  // (9 x 9 stands in, where it fits)
                    if (r.lo || rect_width(r.hi, TX) != rw || rect_height(r.hi, TX) != rh || py != (y0 & 0xffffu)) return 10;
                } else {
                    if (!m)
                        for (uint32_t y = 0; y < rh; ++y)
                            for (uint32_t x = 0; x < rw; ++x) m |= 1ull << (8 * y + x);
                    const unsigned long long got = (unsigned long long)r.lo | ((unsigned long long)r.hi << 32);
                    const uint32_t d = (py - y0) & 0xffffu;
                    if (!r.lo || (d != 0 && d != 4) || (d ? m >> 32 : m) != got || (d && (uint32_t)m)) return 11;
                }
            }
            if (k.linear) {
                if (masked) count_linear_mask(key(x0, y0), TX, lo, hi, k.width[0], add, full);
                else count_linear_rect(key(x0, y0), TX, w, h, k.width[0], add, full);
            } else if (k.npass > 1 && !masked) {
                count_run(x0, w, h, k.width[0], add, full);
            } else {
                continue;
            }
            long long run = 0;
            for (int d = 0; d < bins; ++d) {
                run += diff[d];
                if (run + cyc != want[d]) { printf("view %d record %d digit %d: %lld, not %lld\n", v, t, d, run + cyc, want[d]); return 7; }
            }
        }
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("tilekeys")
    src = d / "main.cpp"
    src.write_text(MAIN)
    exe = d / "main"
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2503_18402_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    return str(exe)


GRIDS = [
    [(1, 1)], [(15, 8)], [(16, 16)], [(17, 15)], [(155, 103)], [(300, 260)], [(263, 38)],
    [(500, 1)], [(1, 256)], [(1, 257)], [(1, 500)], [(1, 4000)], [(1, 70000)], [(1, 300), (1, 900)],
    [(1, 300), (2, 40)], [(65536, 1), (8, 8), (1, 65536)], [(65536, 1), (1, 40000)], [(32769, 1), (1, 16385)],
    [(20000, 3), (7, 40000)],
]


@pytest.mark.parametrize("grid", GRIDS, ids=[" ".join(f"{x}x{y}" for x, y in g) for g in GRIDS])
def test_keys_and_lowest_digit_counts(program, grid):
    r = subprocess.run([program, *(str(n) for xy in grid for n in xy)], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout)
