"""Host rules of the engine (hot_plan.h), compiled on their own: no GPU."""
import ctypes
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2408_00598_gb300", "csrc")

WRAP = r"""
#include "hot_plan.h"
#include <cstring>
using namespace hot;
extern "C" int tile_table() { return kTileTable; }
extern "C" int max_group() { return kMaxGroup; }
// out: the entries, 4 ints each; start: used + 1 ints; returns used, *most
extern "C" int plan(int n, const int* tiles, const int* elems, int grid, int fp64, int* start, int* out, int* most) {
    std::vector<int> inst(n);
    for (int q = 0; q < n; ++q) inst[q] = q;
    const GroupPlan p = plan_groups(inst, std::vector<int>(tiles, tiles + n), std::vector<int>(elems, elems + n), grid, fp64);
    std::memcpy(start, p.start.data(), p.start.size() * sizeof(int));
    if (!p.entries.empty()) std::memcpy(out, p.entries.data(), p.entries.size() * sizeof(GroupEntry));
    *most = p.most;
    return p.used;
}
extern "C" int pick(int n, const int* rows, const double* single, const double* chain) {
    std::vector<HeightTime> t(n);
    for (int q = 0; q < n; ++q) t[q] = HeightTime{rows[q], single[q], chain[q]};
    return pick_height(t);
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src = d / "wrap.cpp"
    src.write_text(WRAP)
    out = str(d / "libplan.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I" + CSRC, str(src), os.path.join(CSRC, "hot_plan.cpp"),
                    "-o", out], check=True)
    return ctypes.CDLL(out)


def _plan(rules, tiles, elems, grid, fp64):
    n = len(tiles)
    ints = lambda v: (ctypes.c_int * max(1, len(v)))(*v)
    start, out, most = ints([0] * (grid + 1)), ints([0] * 4 * (grid + n)), ctypes.c_int()
    used = rules.plan(n, ints(tiles), ints(elems), grid, fp64, start, out, ctypes.byref(most))
    ctas = [[tuple(out[4 * e:4 * e + 3]) for e in range(start[c], start[c + 1])] for c in range(used)]
    return ctas, most.value


def _check(rules, tiles, elems, grid, fp64):
    """Every rank of every group is on one CTA; a CTA with a rank of a larger group has nothing else (its group waits
    for it); the plan fits the grid."""
    ctas, most = _plan(rules, tiles, elems, grid, fp64)
    assert len(ctas) <= grid and all(ctas)
    seen = {}
    for entries in ctas:
        for inst, rank, size in entries:
            assert size == 1 or len(entries) == 1
            assert seen.setdefault(inst, (size, set()))[0] == size
            assert rank not in seen[inst][1]
            seen[inst][1].add(rank)
    assert sorted(seen) == list(range(len(tiles)))
    for inst, (size, ranks) in seen.items():
        assert ranks == set(range(size)) and size <= rules.max_group()
    assert most == max([-(-tiles[q] // seen[q][0]) for q in seen], default=0)
    return ctas, most


def _tiles(m, n, fp64):
    """Tiles of an m x n pair and the elements of one (the rule of tile_rows without its balancing)."""
    long = max(m, n)
    pitch = (long + 3) & ~3
    rows = max(1, min(long, 4096 // pitch, 32 if pitch >= 96 else 64) if fp64 else min(long, 16384 // pitch, 128))
    tiles = n * -(-m // rows) + m * -(-n // rows)
    return tiles, m * n * (m + n) // tiles


@pytest.mark.parametrize("fp64", [0, 1])
@pytest.mark.parametrize("grid", [1, 7, 38, 152, 304])
def test_random_batches_up_to_the_tile_limit(rules, grid, fp64):
    rng = random.Random(grid)
    table = rules.tile_table()
    for _ in range(400):
        top = rng.choice([4, 16, 64, 128, 128 if fp64 else 256])
        tiles, elems, left = [], [], 4 * grid
        for _ in range(500):
            t, e = _tiles(rng.randint(2, top), rng.randint(2, top), fp64)
            if t <= left:
                left -= t
                tiles.append(t)
                elems.append(e)
        _, most = _check(rules, tiles, elems, grid, fp64)
        if not fp64:
            assert most <= table          # the dispatch's tile limit keeps plans below k_group32's table


def test_a_plan_above_the_tile_table_says_so(rules):
    """Beyond the dispatch's limit of four tiles per CTA: the host reads `most` and takes the chain."""
    _, most = _check(rules, [512], [16384], 4, 0)
    assert most == 128 > rules.tile_table()


@pytest.mark.parametrize("fp64,m,n,tiny", [(0, 256, 60, 150), (1, 64, 64, 200)])
def test_tiny_pairs_beside_a_larger_one_share_ctas(rules, fp64, m, n, tiny):
    """The batches of test_tiny_pairs_that_share_a_cta_equal_single_solves, on 304 CTAs."""
    sides = [(m, n)] + [(2, 2 + q % 2) for q in range(tiny)]
    work = [_tiles(a, b, fp64) for a, b in sides]
    ctas, _ = _check(rules, [t for t, _ in work], [e for _, e in work], 304, fp64)
    assert sum(t for t, _ in work) <= 4 * 304
    assert sum(1 for e in ctas if len(e) >= 2) >= 10


@pytest.mark.parametrize("times,want", [
    ([(64, 13.2, 26.1), (32, 12.7, 25.6), (16, 16.5, 28.0)], 32),
    # the chain loses more at the height that the group kernel likes best
    ([(48, 12.0, 25.0), (24, 11.8, 30.0)], 48),
    ([(128, 20.0, 35.0), (64, 22.7, 33.8)], 128),
    # heights at which a single solve runs the chain too
    ([(64, 111.5, 111.5), (32, 126.5, 126.5)], 64),
    ([(96, 18.3, 30.3), (48, 22.0, 30.2), (12, 41.5, 41.5)], 96),
    ([(16, 12.6, 25.2)], 16),
])
def test_tile_height_serves_both_forms(rules, times, want):
    n = len(times)
    col = lambda k, t: (t * n)(*[r[k] for r in times])
    assert rules.pick(n, col(0, ctypes.c_int), col(1, ctypes.c_double), col(2, ctypes.c_double)) == want
