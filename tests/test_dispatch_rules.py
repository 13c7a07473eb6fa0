"""The rules by which a call takes one of two forms, as the library computes them (compiled for the CPU)."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_10103_b200", "csrc")
SOURCE = """
#include "hf_dispatch.h"
extern "C" int one_launch(int block, int d, int Tm, int BH, int clusters, int clusters16) {
    return pool_select_one_launch(block, d, Tm, BH, clusters, clusters16);
}
extern "C" int by_kernel(int context, int current, int given, int aligned, int device_memory, int device) {
    return kernel_instead_of_copy(context, current, CallerMemory{given != 0, aligned != 0, device_memory != 0, device});
}
extern "C" int kpl(int Tn) { return select_kpl(Tn); }
extern "C" int uses(int kpl, int n_b, int max_Tn) { return select_uses(kpl, n_b, max_Tn); }
extern "C" int rows(int kpl, int G, int Tm, int BH, int sms) { return select_rows(kpl, G, Tm, BH, sms); }
extern "C" int ahead(int block, int units, int selection_blocks, int sms) { return swa_history_ahead(block, units, selection_blocks, sms); }
extern "C" int teams(int d, int block, int tiles, int history) { return swa_teams(d, block, tiles, history != 0); }
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    src, so = d / "rules.cpp", d / "rules.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-fPIC", "-shared", "-I", CSRC, str(src), "-o", str(so)], check=True, capture_output=True)
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("d", [64, 128])
def test_pooling_and_selection_without_room_for_a_cluster(rules, d):
    """Where no cluster of T_m thread blocks can be resident, a head's blocks are pooled and selected in two launches."""
    for Tm in range(1, 40):
        assert rules.one_launch(128, d, Tm, 1, 0, 0) == (Tm == 1)          # (one thread block is no cluster)
        assert rules.one_launch(128, d, Tm, 1, 14, 14) == (Tm <= 16)
        assert rules.one_launch(16, d, Tm, 1, 0, 0) == (Tm <= 8)           # no cluster in this form
        assert not rules.one_launch(64, d, Tm, 1, 9, 9)


# query blocks a head, clusters that a B200 holds, most heads measured faster in one launch, fewest measured not faster (heads of 64; of 128)
LINE = [(2, 148, 130, 192, 130, 192), (3, 93, 81, 94, 81, 94), (4, 71, 61, 70, 61, 70), (5, 56, 49, 56, 49, 56), (6, 45, 40, 47, 40, 47),
        (7, 37, 32, 37, 32, 37), (8, 33, 28, 35, 28, 35), (9, 30, 27, 31, 27, 31), (10, 26, 22, 24, 22, 24), (11, 21, 16, 19, 13, 17),
        (12, 21, 16, 19, 14, 17), (13, 17, 14, 17, 14, 16), (14, 14, 13, 15, 13, 15), (15, 14, 14, 15, 14, 15), (16, 14, 14, 15, 14, 15)]


@pytest.mark.parametrize("Tm,clusters,fast64,slow64,fast128,slow128", LINE)
def test_one_launch_up_to_one_wave_of_clusters(rules, Tm, clusters, fast64, slow64, fast128, slow128):
    for d, fast, slow in ((64, fast64, slow64), (128, fast128, slow128)):
        assert all(rules.one_launch(128, d, Tm, BH, clusters, 14) for BH in range(1, fast + 1))
        assert not any(rules.one_launch(128, d, Tm, BH, clusters, 14) for BH in range(slow, 4096))


@pytest.mark.parametrize("d", [64, 128])
def test_a_single_block_and_small_blocks_on_any_grid(rules, d):
    for BH in (1, 148, 1024, 65535):
        assert rules.one_launch(128, d, 1, BH, 0, 0) and rules.one_launch(16, d, 8, BH, 0, 0) and not rules.one_launch(16, d, 9, BH, 0, 0)


def test_a_kernel_in_place_of_a_copy_only_at_home(rules):
    """The state leaves by a kernel where the context's device is current and the buffer is aligned memory of that device; a second device,
    current or under the buffer, takes the copy."""
    for context in (0, 1):
        for current in (-1, 0, 1):
            home = current == context
            for device in (-1, 0, 1):
                assert rules.by_kernel(context, current, 1, 1, 1, device) == (home and device == context)
                assert not rules.by_kernel(context, current, 1, 0, 1, device)         # not aligned
                assert not rules.by_kernel(context, current, 1, 1, 0, device)         # host, pinned or managed memory
            assert rules.by_kernel(context, current, 0, 1, 0, -1) == home             # this tensor is not wanted


def test_a_context_touches_the_selection_kernels_of_its_windows_only(rules):
    """Touching a kernel loads it: those for longer (or shorter) windows than the context can have stay out, and none that it launches."""
    for n_b in (1, 5, 37, 128, 129, 256, 300, 512, 1024):
        for chunks in range(1, 9):
            if n_b * chunks > 1024:
                continue
            launched = {rules.kpl(n_b * x) for x in range(1, chunks + 1)}
            touched = {k for k in (4, 8, 16, 32) if rules.uses(k, n_b, n_b * chunks)}
            assert launched <= touched and all(min(launched) <= k <= max(launched) for k in touched)
            assert all(32 * rules.kpl(n_b * x) >= n_b * x for x in range(1, chunks + 1))


def test_softmax_teams(rules):
    """Teams at head dim 64; at 128 for long lists of 128-token blocks, shorter ones without the history term (a context loads both kernels
    of the lists between, so that the rule must grow with the tiles and shrink with the history term)."""
    for tiles in range(1, 1025):
        for block in (16, 64, 128):
            assert rules.teams(64, block, tiles, 0) and rules.teams(64, block, tiles, 1)
            for history in (0, 1):
                t = rules.teams(128, block, tiles, history)
                assert t == (block == 128 and tiles >= (14 if history else 8))
                assert rules.teams(128, block, tiles + 1, history) >= t >= rules.teams(128, block, tiles, 1)


def test_history_term_ahead_of_the_selections_end(rules):
    """Where the selection leaves an SM for every thread block of the last round of units, and with one round of 64-token blocks."""
    for block in (16, 64, 128):
        assert rules.ahead(block, 12, 12, 148) and rules.ahead(block, 100, 48, 148)
        assert rules.ahead(block, 149, 147, 148) and not rules.ahead(block, 149, 148, 148)
        assert rules.ahead(block, 320, 80, 148) and not rules.ahead(block, 444, 1, 148) and not rules.ahead(block, 148, 1, 148)
        assert rules.ahead(block, 101, 48, 148) == (block == 64)
    assert rules.ahead(64, 132, 72, 148) and not rules.ahead(64, 1776, 76, 148)


def test_query_blocks_per_thread_block_of_the_selection(rules):
    for G in (1, 2, 8):
        for Tm in (1, 3, 4, 5, 37, 74, 100):
            for BH in (1, 4, 12, 48):
                assert rules.rows(4, G, Tm, BH, 148) == (8 if G == 8 else 4)
                assert rules.rows(16, G, Tm, BH, 148) == rules.rows(32, G, Tm, BH, 148) == 8
                assert rules.rows(8, G, Tm, BH, 148) == (8 if G == 8 or -(-Tm // 4) * BH > 148 else 4)
