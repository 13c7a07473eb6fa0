"""Where the merged lists of 64- and 16-token blocks put their entries, formed on the CPU by the kernels' own index functions: every entry
a slot of its own, no more tiles than the blocks need, a kept block of every row group in the first tile, and (64-token blocks) at most
one block per row group in the tiles behind the shared ones."""
import ctypes
import itertools
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_10103_b200", "csrc")
SOURCE = """
#include "k_union.cuh"
template <int G> static int at(int n0, int n1, int n2, int what, int i) {
    UnionOrder<G> o; o.n0 = n0; o.n1 = n1; o.n2 = n2;
    return what < 3 ? o.slot(what, i) : what == 3 ? o.slots() : o.hole();
}
extern "C" int order2(int n0, int n1, int n2, int what, int i) { return at<2>(n0, n1, n2, what, i); }
extern "C" int order8(int n0, int n1, int n2, int what, int i) { return at<8>(n0, n1, n2, what, i); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("union")
    src, so = d / "union.cu", d / "union.so"
    src.write_text(SOURCE)
    subprocess.run([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-Xcompiler", "-fPIC",
                    "-shared", "-I", CSRC, str(src), "-o", str(so)], check=True, capture_output=True)
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("g", [2, 8])
def test_every_entry_has_a_slot(lib, g):
    order = lib.order2 if g == 2 else lib.order8
    sizes = [0, 1, 2, 3, 4, 7, 8, 9, 30]
    for n in itertools.product(sizes, sizes, sizes if g == 2 else [0]):
        if sum(n) == 0:
            continue
        where = {order(*n, x, i): x for x in range(3) for i in range(n[x])}
        slots, hole = order(*n, 3, 0), order(*n, 4, 0)
        assert len(where) == sum(n), "two entries share a slot"
        assert set(where) | ({hole} if hole >= 0 else set()) == set(range(slots)) and hole not in where
        assert -(-slots // g) == -(-sum(n) // g), "more tiles than the blocks fill"
        if g == 8:
            assert all(where[s] == 0 for s in range(n[0]))
            continue
        first = {where.get(0), where.get(1)}
        assert 0 in first or (n[1] == 0 or 1 in first) and (n[2] == 0 or 2 in first)
        if n[1] == n[2]:                 # lists of one length
            for t in range(-(-slots // 2)):
                pair = sorted(x for x in (where.get(2 * t), where.get(2 * t + 1)) if x is not None)
                assert pair in ([0, 0], [0], [1, 2])
