"""The history term of a thread block's first unit ahead of the selection's end, on grids of several units per thread block: the unit behind the first finds the S buffers,
the buffer of S W^T and z, and the sums' buffers as that one left them.  Blocks of 128 and 64 tokens (16-token blocks have as many thread blocks in the
selection as units, so that the rule leaves them out there), one to five tiles and more, rotated or not.  Each case asserts which form it takes."""
import numpy as np
import pytest

from paper_2604_10103_b200 import inputs as gen
from tests import harness as hz
from tests.test_dispatch_rules import rules  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

f64 = gen.bf16_bits_to_f64


def takes_it(rules, heads, tokens, block, T_n):  # noqa: F811
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    units, T_m = -(-tokens // 128) * heads, -(-tokens // block)
    assert T_n <= 128 and T_m > 16          # (pooling and selection apart, four query blocks a thread block)
    return units > sms and bool(rules.ahead(block, units, -(-T_m // rules.rows(4, 128 // block, T_m, heads, sms)) * heads, sms))


@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("heads,tokens,block,topk", [(8, 2500, 128, 1), (8, 2500, 128, 2), (8, 2500, 128, 3), (8, 2433, 128, 5), (17, 2200, 128, 2), (8, 2500, 128, 13),
                                                     (8, 2500, 64, 1), (8, 2437, 64, 2), (8, 2500, 64, 5), (8, 2500, 64, 9)])
def test_several_units(rules, heads, tokens, block, topk, rope):  # noqa: F811
    w = gen.Workload("ahead_grids", batch=1, heads=heads, head_dim=128, tokens_per_frame=tokens, chunk_frames=1, window_frames=2, block=block, topk=topk,
                     keep_permille=0, seed=821 + topk)
    assert takes_it(rules, heads, tokens, block, 2 * -(-tokens // block))
    gpu, ora = hz.GpuStream(w, rope=rope), hz.make_oracle(w, rope=rope)
    try:
        for c in range(3):
            qb, kb, vb = gen.qkv(w, 0, c, 0)
            q, k, v = gpu.up(qb), gpu.up(kb), gpu.up(vb)
            out = gpu.forward(q, k, v)
            if c == 2:
                hz.assert_close_out(out, ora.forward(f64(qb), f64(kb), f64(vb)), f"chunk {c}")
            for _ in range(2):
                assert np.array_equal(gpu.forward(q, k, v), out)
            kc, vc = gen.clean_kv(w, 0, c)
            gpu.append(gpu.up(kc), gpu.up(vc)); ora.append(f64(kc), f64(vc))
        assert gpu.ctx.hf_get_device_status() == (0, 0)
    finally:
        gpu.close()


@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("block,topk", [(128, 1), (128, 2), (128, 4), (64, 1), (64, 3)])
def test_same_bits_where_the_term_is_not_ahead(rules, block, topk, rope):  # noqa: F811
    """On the same lists given by the caller, where no selection is in front, the term is formed behind the last tile."""
    import torch
    w = gen.Workload("ahead_bits", batch=1, heads=8, head_dim=128, tokens_per_frame=2500, chunk_frames=1, window_frames=2, block=block, topk=topk, keep_permille=0,
                     seed=827)
    assert takes_it(rules, 8, 2500, block, 2 * -(-2500 // block))
    gpu = hz.GpuStream(w, rope=rope)
    try:
        for c in range(3):
            gpu.append(*(gpu.up(x) for x in gen.clean_kv(w, 0, c)))
        q, k, v = (gpu.up(x) for x in gen.qkv(w, 0, 3, 0))
        o, given = torch.empty_like(q), torch.empty_like(q)
        gpu.ctx.hf_hybrid_forward(0, q, k, v, o)
        gpu.ctx.hf_block_select(0, q, k)
        gpu.ctx.hf_sparse_swa_merged(0, q, k, v, given)
        torch.cuda.synchronize()
        assert torch.equal(o, given) and gpu.ctx.hf_get_device_status() == (0, 0)
    finally:
        gpu.close()
