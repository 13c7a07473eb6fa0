"""The rows of the temporal tables that the pooling pass reads, formed on the CPU by the kernel's own index function: every thread
of every block of a chunk, last blocks shorter than the sixteen rows of threads among them, at the cap of the rotation, where the
tables end with the chunk's last frame."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_10103_b200", "csrc")
SOURCE = """
#include "k_pool_select.cuh"
extern "C" int frame_of(int t0, int r, int n, int tokens_per_frame) { return turn_frame(t0, r, n, tokens_per_frame); }
"""


@pytest.fixture(scope="module")
def frame_of(tmp_path_factory):
    d = tmp_path_factory.mktemp("rows")
    src, lib = d / "rows.cu", d / "rows.so"
    src.write_text(SOURCE)
    subprocess.run([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-Xcompiler", "-fPIC",
                    "-shared", "-I", CSRC, str(src), "-o", str(lib)], check=True, capture_output=True)
    return ctypes.CDLL(str(lib)).frame_of


@pytest.mark.parametrize("tokens_per_frame,chunk_frames,block", [
    (20, 3, 16),        # 60 tokens: last block 12
    (130, 1, 128),      # last block 2
    (3, 1, 16),         # one block of 3
    (7, 11, 64),        # 77 tokens: last block 13, several frames in sixteen rows
    (96, 1, 64), (1560, 3, 128),
])
def test_no_row_past_the_tables(frame_of, tokens_per_frame, chunk_frames, block):
    tokens, cap = tokens_per_frame * chunk_frames, 2 * chunk_frames
    base = cap - chunk_frames + 1                       # index of the chunk's first frame once the cap is reached
    for t0 in range(0, tokens, block):
        n = min(block, tokens - t0)
        for r in range(block):                          # rows r + 16 i of the block, those past its end among them
            f = frame_of(t0, r, n, tokens_per_frame)
            if r < n:
                assert f == (t0 + r) // tokens_per_frame and 0 <= base + f <= cap
            else:
                assert f == -1, f"row {t0 + r} of {tokens} would read row {base + f} of tables that end at {cap}"
