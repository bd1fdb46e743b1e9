"""CPU: the order in which the prefill attention hands out its query blocks (ham_order.cuh): every block
gets a place of its own, those that reach the farthest slot first, whatever the caches hold."""
import ctypes
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2505_20438_gb300", "csrc")


@pytest.fixture(scope="module")
def order(tmp_path_factory):
    d = tmp_path_factory.mktemp("order")
    src, lib = d / "order.cpp", d / "order.so"
    src.write_text(
        '#include "ham_order.cuh"\n'
        'extern "C" unsigned blocks(unsigned n, int s) { return ham::query_blocks(n, s); }\n'
        'extern "C" unsigned reach(unsigned L, unsigned n, unsigned j, int s) { return ham::block_reach(L, n, j, s); }\n'
        'extern "C" unsigned before(unsigned L, unsigned n, unsigned r, int first, int s) {\n'
        '  return ham::blocks_before(L, n, r, first != 0, s); }\n')
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)],
                   check=True)
    return ctypes.CDLL(str(lib))


@pytest.mark.parametrize("shift", [5, 6, 7, 8])  # rows a block at groups 8, 4, 2, 1
@pytest.mark.parametrize("most_rows,most_cached", [(1, 0), (40, 0), (300, 0), (40, 130), (700, 9000), (64, 64)])
def test_places_sort_the_blocks_by_reach(order, shift, most_rows, most_cached):
    rng = random.Random(most_rows * 1000 + most_cached + shift)
    for _ in range(40):
        B = rng.choice([1, 2, 3, 7, 40])
        n = [rng.choice([0, rng.randint(0, most_rows), most_rows]) for _ in range(B)]
        L = [rng.choice([0, rng.randint(0, most_cached), most_cached]) for _ in range(B)]
        want = sorted((-(L[b] + min(n[b], (j + 1) << shift)), b, j)
                      for b in range(B) for j in range(-(-n[b] >> shift)))
        got = {}
        for b in range(B):
            m = order.blocks(n[b], shift)
            assert m == -(-n[b] >> shift)
            for j in range(m):
                r = order.reach(L[b], n[b], j, shift)
                at = m - 1 - j + sum(order.before(L[c], n[c], r, int(c < b), shift) for c in range(B) if c != b)
                got[at] = (-r, b, j)
        assert [got[k] for k in range(len(want))] == want
