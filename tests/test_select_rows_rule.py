"""Query blocks per thread block of the selection at 129 to 256 key blocks: the form that is through in fewer rounds of the device (hf_dispatch.h)."""
import ctypes
import subprocess

import pytest

from tests.test_dispatch_rules import CSRC

SOURCE = """
#include "hf_dispatch.h"
extern "C" int rows_of(int G, int d, int Tn, int Tm, int BH) { return select_rows_of(select_kpl(Tn), G, d, Tn, Tm, BH, 148); }
extern "C" int uses_rows(int kpl, int rows, int G, int d, int n_b, int max_Tn, int Tm, int BH) { return select_uses_rows(kpl, rows, G, d, n_b, max_Tn, Tm, BH, 148); }
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rows")
    src, so = d / "rows.cpp", d / "rows.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-fPIC", "-shared", "-I", CSRC, str(src), "-o", str(so)], check=True, capture_output=True)
    return ctypes.CDLL(str(so))


# head dim, T_n, T_m, heads, rows of the form measured faster by more than 5 %
@pytest.mark.parametrize("d,Tn,Tm,heads,rows", [
    (64, 130, 65, 24, 4), (64, 148, 74, 16, 4), (64, 180, 90, 16, 4), (64, 208, 104, 12, 4), (64, 208, 104, 16, 4), (64, 208, 104, 24, 4),
    (64, 222, 74, 16, 4), (64, 250, 125, 12, 4), (64, 250, 125, 24, 4), (128, 130, 65, 24, 4),
    (64, 180, 90, 12, 8), (64, 180, 90, 24, 8), (64, 222, 74, 12, 8), (64, 250, 125, 8, 8), (64, 250, 125, 16, 8), (128, 130, 65, 12, 8),
    (128, 180, 90, 24, 8), (128, 208, 104, 8, 8), (128, 222, 74, 8, 8), (128, 222, 74, 24, 8), (128, 250, 125, 6, 8), (128, 250, 125, 24, 8)])
def test_fewer_rounds(rules, d, Tn, Tm, heads, rows):
    assert rules.rows_of(2, d, Tn, Tm, heads) == rows


def test_other_windows_and_kernels_a_context_touches(rules):
    for G in (1, 2, 8):
        for d in (64, 128):
            for n_b in (16, 37, 51, 74, 128):
                for heads in (1, 12, 24, 48):
                    seen = set()
                    for Tn in range(n_b, 8 * n_b + 1, n_b):
                        r, kpl = rules.rows_of(G, d, Tn, n_b, heads), 4 if Tn <= 128 else 8 if Tn <= 256 else 16 if Tn <= 512 else 32
                        assert r == 8 if G == 8 or Tn > 256 else r in (4, 8) if Tn > 128 else r == 4
                        seen.add((kpl, r))
                    for kpl in (4, 8, 16, 32):
                        for r in (4, 8):
                            assert bool(rules.uses_rows(kpl, r, G, d, n_b, 8 * n_b, n_b, heads)) == ((kpl, r) in seen)
