"""The rules by which a call takes one of two forms, as the library computes them (compiled for the CPU)."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_10103_b200", "csrc")
SOURCE = """
#include "hf_dispatch.h"
extern "C" int one_launch(int block, int Tm, int BH, int sm_count, int clusters) { return pool_select_one_launch(block, Tm, BH, sm_count, clusters); }
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    src, so = d / "rules.cpp", d / "rules.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-fPIC", "-shared", "-I", CSRC, str(src), "-o", str(so)], check=True, capture_output=True)
    return ctypes.CDLL(str(so))


def test_pooling_and_selection_without_room_for_a_cluster(rules):
    """Where no cluster of T_m thread blocks can be resident, a head's blocks are pooled and selected in two launches."""
    for Tm in range(1, 40):
        assert rules.one_launch(128, Tm, 1, 148, 0) == (Tm == 1)          # (one thread block is no cluster)
        assert rules.one_launch(128, Tm, 1, 148, 1) == (Tm <= 16)
        assert rules.one_launch(16, Tm, 1, 148, 0) == (Tm <= 8)           # no cluster in this form
        assert not rules.one_launch(64, Tm, 1, 148, 9)
