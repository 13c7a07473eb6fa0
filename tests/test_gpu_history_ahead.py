"""The history term of a thread block's first unit, formed ahead of the selection's end at head dim 128: grids that take it and grids that do not
(one unit, a wave, several units per thread block), units of one tile up to five, block sizes, rotated or not, behind a forward call that changed
nothing and behind commits that changed the state.  Merged output against the oracle, and every call the same bits."""
import numpy as np
import pytest

from paper_2604_10103_b200 import inputs as gen
from tests import harness as hz

pytestmark = pytest.mark.gpu

f64 = gen.bf16_bits_to_f64


@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("heads,tokens,block,topk", [(1, 100, 128, 1), (2, 129, 64, 2), (24, 330, 128, 2), (26, 600, 128, 3), (66, 300, 128, 1), (160, 100, 64, 2),
                                                     (58, 260, 128, 5), (3, 129, 16, 4), (60, 300, 16, 9)])
def test_first_unit(heads, tokens, block, topk, rope):
    w = gen.Workload("ahead", batch=1, heads=heads, head_dim=128, tokens_per_frame=tokens, chunk_frames=1, window_frames=2, block=block, topk=topk,
                     keep_permille=0, seed=811 + topk)
    gpu, ora = hz.GpuStream(w, rope=rope), hz.make_oracle(w, rope=rope)
    try:
        for c in range(4):
            qb, kb, vb = gen.qkv(w, 0, c, 0)
            q, k, v = gpu.up(qb), gpu.up(kb), gpu.up(vb)
            out = gpu.forward(q, k, v)
            if c in (0, 3):
                hz.assert_close_out(out, ora.forward(f64(qb), f64(kb), f64(vb)), f"chunk {c}")
            for _ in range(2):
                assert np.array_equal(gpu.forward(q, k, v), out)
            kc, vc = gen.clean_kv(w, 0, c)
            gpu.append(gpu.up(kc), gpu.up(vc)); ora.append(f64(kc), f64(vc))
        assert gpu.ctx.hf_get_device_status() == (0, 0)
    finally:
        gpu.close()
