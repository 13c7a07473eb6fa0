"""Softmax warps of the attention kernel in teams that take turns at the tiles: which team has a unit's first and last tile depends on all
the units before it on the same thread block.  Several units per thread block with one tile up to a few each, lists on both sides of the
line between teams and column groups, short last blocks around the edges of a half's columns.  Softmax branch with its row log-sums
against the warp-level kernel on the same lists, merged output against the oracle."""
import numpy as np
import pytest

from paper_2604_10103_b200 import inputs as gen
from tests import harness as hz

pytestmark = pytest.mark.gpu

f64 = gen.bf16_bits_to_f64


def check(w, chunks, rope=False):
    import torch
    gpu, ref, ora = hz.GpuStream(w, rope=rope), hz.GpuStream(w, swa_kernel=1, rope=rope), hz.make_oracle(w, rope=rope)
    try:
        for c in range(chunks):
            kc, vc = gen.clean_kv(w, 0, c)
            gpu.append(gpu.up(kc), gpu.up(vc)); ref.append(ref.up(kc), ref.up(vc)); ora.append(f64(kc), f64(vc))
        qb, kb, vb = gen.qkv(w, 0, chunks, 0)
        q, k, v = gpu.up(qb), gpu.up(kb), gpu.up(vb)
        m, idx, _ = gpu.select(q, k)
        o, lse = gpu.swa(q, k, v, want_lse=True)
        o_ref, lse_ref = ref.swa(q, k, v, idx=torch.from_numpy(idx).cuda(), want_lse=True)
        hz.assert_close_out(o, o_ref, "softmax branch")
        assert np.abs(lse - lse_ref).max() <= 1e-3          # fp32 sums of up to 3 072 terms in another order: below 1e-4
        out = gpu.forward(q, k, v)
        hz.assert_close_out(out, ora.forward(f64(qb), f64(kb), f64(vb), mask=m), "merged")
        for _ in range(3):
            assert np.array_equal(gpu.forward(q, k, v), out)
        assert gpu.ctx.hf_get_device_status() == (0, 0)
    finally:
        gpu.close(); ref.close()


@pytest.mark.parametrize("topk", [1, 2, 3, 4])
@pytest.mark.parametrize("d,block", [(64, 128), (64, 64), (64, 16)])
def test_several_units_of_few_tiles(d, block, topk):
    check(gen.Workload("teams", batch=2, heads=76, head_dim=d, tokens_per_frame=360, chunk_frames=1, window_frames=2, block=block, topk=topk,
                       keep_permille=0, seed=701 + topk), 3)


@pytest.mark.parametrize("topk", [7, 8, 13, 14, 15, 16])
def test_both_sides_of_the_line_at_head_dim_128(topk):
    check(gen.Workload("teams128", batch=1, heads=54, head_dim=128, tokens_per_frame=1000, chunk_frames=1, window_frames=2, block=128, topk=topk,
                       keep_permille=0, seed=709 + topk), 3, rope=topk == 15)


@pytest.mark.parametrize("d,topk", [(64, 3), (64, 6), (128, 14), (128, 23)])
@pytest.mark.parametrize("tail", [1, 32, 33, 64, 65, 97])
def test_short_last_blocks(d, topk, tail):
    check(gen.Workload("tails", batch=1, heads=2, head_dim=d, tokens_per_frame=7 * 128 + tail, chunk_frames=1, window_frames=3, block=128,
                       topk=topk, keep_permille=0, seed=719 + tail), 4)
