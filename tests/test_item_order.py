"""Order in which the persistent CTAs take the items of a packed batch (csrc/item_order.h), on the host: every item once, heaviest
first, and where taking in turn is unbalanced no CTA has more than when each item goes to the one that has the least."""
import ctypes
import heapq
import random
import subprocess

import pytest

from paper_2609_09721_b200 import build

ITEM = 3        # tiles that an item costs beside its own
HARNESS = r"""
#include "item_order.h"
extern "C" int64_t order(const int32_t* tiles, const int32_t* counts, int n_runs, int64_t n_items, int ctas, int32_t* places)
{
    std::vector<efq::ItemRun> runs;
    for (int i = 0; i < n_runs; ++i) runs.push_back(efq::ItemRun{tiles[i], counts[i]});
    return efq::order_items(runs, n_items, ctas, places);
}
extern "C" int64_t room(int64_t n) { return efq::order_places(n); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("order")
    (d / "order.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I", build.CSRC, str(d / "order.cpp"), "-o", str(d / "order.so")], check=True)
    so = ctypes.CDLL(str(d / "order.so"))
    so.room.restype, so.room.argtypes = ctypes.c_int64, [ctypes.c_int64]
    so.order.restype = ctypes.c_int64
    so.order.argtypes = [ctypes.POINTER(ctypes.c_int32)] * 2 + [ctypes.c_int, ctypes.c_int64, ctypes.c_int, ctypes.POINTER(ctypes.c_int32)]
    return so


def _weights(lens, heads, causal):
    w = [(min(n, 128 * (t + 1)) + 127) // 128 if causal else (n + 127) // 128 for n in lens for t in range((n + 127) // 128) for _ in range(heads)]
    return sorted(w, reverse=True)


def _in_turn(w, ctas):
    load = [0] * ctas
    for i, x in enumerate(w):
        r, c = divmod(i, ctas)
        load[ctas - 1 - c if r & 1 else c] += x + ITEM
    return max(load)


def _least_first(w, ctas):
    load = [0] * ctas
    for x in w:
        heapq.heapreplace(load, load[0] + x + ITEM)
    return max(load)


def _rounds(w, ctas):
    """Items of the CTA that has the most of them when each goes to the one that has the least."""
    load = [(0, 0)] * ctas
    for x in w:
        heapq.heapreplace(load, (load[0][0] + x + ITEM, load[0][1] + 1))
    return max(n for _, n in load)


def _order(lib, w, ctas):
    """The items of every CTA, or None: in turn."""
    runs = []
    for x in w:
        if runs and runs[-1][0] == x:
            runs[-1][1] += 1
        else:
            runs.append([x, 1])
    array = lambda v: (ctypes.c_int32 * max(1, len(v)))(*v)
    places = array([-2] * (lib.room(len(w)) + 1))
    used = lib.order(array([r[0] for r in runs]), array([r[1] for r in runs]), len(runs), len(w), ctas, places)
    assert places[lib.room(len(w))] == -2
    if used == 0:
        return None
    lists = [[] for _ in range(ctas)]
    for p in range(used):
        k, c = divmod(p, ctas)
        items = lists[ctas - 1 - c if k & 1 else c]
        if places[p] >= 0:
            assert len(items) == k and (k == 0 or places[p] > items[-1])       # no empty place before it; heaviest first
            items.append(places[p])
    return lists


@pytest.mark.parametrize("lens,heads,causal", [
    ([3000] + [400] * 60, 2, False), ([6000] + [300] * 63, 4, False), ([12000] + [1000] * 30, 1, True), ([5000] * 3 + [1300] * 30, 1, True),
    ([8000, 8000] + [17 * n for n in range(1, 48)], 1, True), ([3000] + [130] * 100, 4, True), ([200000] + [500] * 40, 1, False),
])
def test_unbalanced_batches(lib, lens, heads, causal):
    w, ctas = _weights(lens, heads, causal), 148
    lists = _order(lib, w, ctas)
    assert lists is not None and sorted(i for items in lists for i in items) == list(range(len(w)))
    heaviest = max(sum(w[i] + ITEM for i in items) for items in lists)
    least = max(w[0] + ITEM, -(-sum(x + ITEM for x in w) // ctas))
    if w[0] + ITEM < 1024:
        assert heaviest == _least_first(w, ctas)
    assert heaviest < _in_turn(w, ctas) and heaviest <= 4 / 3 * least + 2        # the bound of that order; 2: steps coarser than a tile


def test_balanced_small_and_large_batches_are_taken_in_turn(lib):
    for w, ctas in [([16] * 444, 148), ([5] * 148, 148), ([9] + [1] * 100, 148), ([30] + [1] * (16 * 148), 148), ([], 148), ([1], 0)]:
        assert _order(lib, w, ctas) is None


def test_random_batches(lib):
    rng = random.Random(1)
    for _ in range(200):
        ctas = rng.choice([2, 7, 148])
        w = sorted((rng.choice([0, 1, rng.randint(1, 40), rng.randint(1, 900)]) for _ in range(rng.randint(ctas + 1, 16 * ctas))), reverse=True)
        lists = _order(lib, w, ctas)
        if lists is None:
            least = max(w[0] + ITEM, -(-sum(x + ITEM for x in w) // ctas))
            assert _in_turn(w, ctas) - least <= max(least / 50, len(w) / 64) or _rounds(w, ctas) * ctas > 3 * len(w) - ctas
            continue
        assert sorted(i for items in lists for i in items) == list(range(len(w)))
        assert max(sum(w[i] + ITEM for i in items) for items in lists) == _least_first(w, ctas)
