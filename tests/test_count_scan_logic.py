"""The arithmetic by which the count pass hands out tiles and the tile scan places records.

* Units of tiles: the count pass's own functions (CellWatch::split, unit), compiled for the
  host.  Whatever the step's size and the grid, the first units of all warps and those of the
  later tickets are disjoint and cover every tile, with and without early leaving.
* Places: a restatement of k_tile_scan on random tiles.  A warp takes 32 consecutive tiles, a
  segmented scan over runs of one cell numbers the passing records, a run that is its whole
  cell owns the child's counter, any other reserves its places with one addition, and tiles of
  pruned or left cells take part in nothing.  Over all warps, in any order, the places of every
  (cell, child) are a permutation of [0, count).
"""
import os
import re
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_2107_11810_gb300", "csrc", "gv_tile.cuh")

HOST = """
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <vector>
#define __device__
#define __forceinline__ inline
static void __syncwarp() {}
static struct { unsigned x; } gridDim;
struct Chunk { int early; };
struct Watch {
    enum { UNITS = 0, SIZE = 1, TILES = 2, RECORDS = 3 };
    uint32_t s[4];
FUNCTIONS
};
int main(int argc, char **argv) {
    for (int i = 1; i + 2 < argc; i += 3) {
        const unsigned nt = (unsigned)std::strtoul(argv[i], 0, 10), blocks = (unsigned)std::strtoul(argv[i + 1], 0, 10);
        const Chunk c = {std::atoi(argv[i + 2])};
        gridDim.x = blocks;
        std::vector<unsigned char> taken(nt, 0);
        unsigned long long sum = 0, twice = 0, later = 0;
        auto take = [&](unsigned tt, unsigned tb) {
            for (unsigned t = tt; t < tb; ++t) {
                if (t >= nt || taken[t]) ++twice;
                else taken[t] = 1, ++sum;
            }
        };
        Watch w;
        for (unsigned warp = 0; warp < blocks * 8; ++warp) {
            unsigned tt, tb;
            w.split(c, nt, warp, 0, tt, tb);
            take(tt, tb);
        }
        unsigned tt, tb;
        for (unsigned ticket = blocks * 8; w.unit(ticket, nt, tt, tb); ++ticket) take(tt, tb), ++later;
        std::printf("%llu %llu %llu\\n", sum, twice, later);
    }
}
"""


def member(text, name):
    m = re.search(r"^    __device__ __forceinline__ \w+ " + name + r"\(.*?^    }$", text, re.S | re.M)
    return m.group(0)


def test_units_cover_every_tile_once(tmp_path):
    text = open(SRC).read()
    src, exe = tmp_path / "units.cpp", tmp_path / "units"
    src.write_text(HOST.replace("FUNCTIONS", member(text, "split") + "\n" + member(text, "unit")))
    subprocess.run(["g++", "-std=c++17", "-O2", "-fsanitize=signed-integer-overflow,bounds",
                    "-fsanitize-undefined-trap-on-error", str(src), "-o", str(exe)], check=True)
    cases = []
    rng = np.random.default_rng(3)
    for blocks in (1, 2, 7, 152, 608, 1216):
        warps = blocks * 8
        per = [1, 2, 15, 16, 17, 31, 32, 33, 255, 256, 511, 512, 513]
        for nt in [1, 2, 31, 32, 33] + [warps * p + d for p in per for d in (-1, 0, 1)] + \
                rng.integers(1, 3_000_000, 8).tolist():
            if 0 < nt <= 4_000_000:
                cases += [(int(nt), blocks, e) for e in (0, 1, 64)]
    out = subprocess.run([str(exe)] + [str(x) for c in cases for x in c], capture_output=True, text=True)
    assert out.returncode == 0
    lines = out.stdout.splitlines()
    assert len(lines) == len(cases)
    tickets = 0
    for (nt, blocks, early), line in zip(cases, lines):
        covered, twice, later = map(int, line.split())
        assert (covered, twice) == (nt, 0), (nt, blocks, early)
        assert early or later == 0
        tickets += later
    assert tickets > 0


def scan_warp(cells, first, last, ballots, counters, whole_counts):
    """k_tile_scan's 32 lanes of one child slot: cells (-1: takes no part), first / last tile of
    its cell, passing lanes; counters: the children's, added to by runs that are a part of their
    cell.  Returns the first place of every lane's records."""
    n = len(cells)
    off = np.zeros(n, np.int64)
    i = 0
    while i < n:
        j = i
        while j + 1 < n and cells[j + 1] == cells[i]:
            j += 1
        if cells[i] >= 0:
            pops = [bin(b).count("1") for b in ballots[i:j + 1]]
            scan = np.cumsum(pops)
            base = 0
            if first[i] and last[j]:
                whole_counts[cells[i]] = int(scan[-1])
            else:
                base = counters.get(cells[i], 0)
                counters[cells[i]] = base + int(scan[-1])
            off[i:j + 1] = base + scan - pops
        i = j + 1
    return off


@pytest.mark.parametrize("seed", range(20))
def test_places_are_permutations(seed):
    rng = np.random.default_rng(seed)
    sizes = rng.integers(1, 40, 60) if seed % 2 else rng.integers(1, 4000, 25)
    out = rng.random(len(sizes)) < 0.25                      # pruned, or left by the count pass
    cells, first, last, ballots = [], [], [], []
    for c, n in enumerate(sizes):
        nt = (int(n) + 31) // 32
        for t in range(nt):
            valid = min(32, int(n) - 32 * t)
            cells.append(-1 if out[c] else c)
            first.append(t == 0)
            last.append(t == nt - 1)
            ballots.append(int(rng.integers(0, 2 ** 32)) & ((1 << valid) - 1) if rng.random() < 0.9 else 0)
    counters, whole, places = {}, {}, {}
    for w in rng.permutation((len(cells) + 31) // 32):       # warps in any order
        i, j = 32 * w, min(32 * w + 32, len(cells))
        before = dict(counters)
        off = scan_warp(cells[i:j], first[i:j], last[i:j], ballots[i:j], counters, whole)
        partial = {c for c in counters if counters[c] != before.get(c)}
        assert len(partial) <= 2                             # only a warp's first and last run
        for k in range(i, j):
            if cells[k] >= 0:
                places.setdefault(cells[k], []).extend(
                    off[k - i] + bin(ballots[k] & ((1 << l) - 1)).count("1") for l in range(32) if ballots[k] >> l & 1)
    for c, ps in places.items():
        assert sorted(ps) == list(range(len(ps)))
        assert whole.get(c, counters.get(c, 0)) == len(ps)
    assert not set(whole) & set(counters)
