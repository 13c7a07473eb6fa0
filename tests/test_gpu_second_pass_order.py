"""Units that the attention kernel computes a second time, head dim 64 with five key blocks kept (four column groups): the numbers of the
first pass are not finite and on their way to the same rows, and must never be what stays there.  The last unit of twelve thread
blocks, behind a unit in range; with and without the history term, against the oracle, every call the same bits."""
import numpy as np
import pytest

from paper_2604_10103_b200 import inputs as gen
from tests import harness as hz

pytestmark = pytest.mark.gpu

f64 = gen.bf16_bits_to_f64


@pytest.mark.parametrize("rope", [False, True])
def test_the_second_pass_has_the_last_word(rope):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    d, n_b, heads = 64, 10, -(-(sms + 12) // 10)
    w = gen.Workload("second_pass", batch=1, heads=heads, head_dim=d, tokens_per_frame=128 * n_b - 30, chunk_frames=1, window_frames=1, block=128,
                     topk=5, keep_permille=0, seed=409)
    gpu, ora = hz.GpuStream(w, rope=rope), hz.make_oracle(w, rope=rope)
    try:
        kc, vc = gen.clean_kv(w, 0, 0)
        gpu.append(gpu.up(kc), gpu.up(vc)); ora.append(f64(kc), f64(vc))
        qb, kb, vb = gen.qkv(w, 0, 1, 0)
        one, a = np.ones((heads, d), np.float32), (180.0 / d ** 0.5) ** 0.5          # a^2 d / sqrt(d) = 180 nats
        kb = gen.shifted(kb, one, a, slice(128 * (n_b - 1), None))                   # the short last block, behind the first kept ones
        far = [u for u in range(sms, heads * n_b)]
        for u in far:
            h, i = divmod(u, n_b)
            head = np.zeros_like(one); head[h] = 1.0
            qb = gen.shifted(qb, head, a, slice(128 * i, 128 * (i + 1)))
        q, k, v = gpu.up(qb), gpu.up(kb), gpu.up(vb)
        m, _, _ = gpu.select(q, k)
        m_ref, _ = ora.select(f64(qb), f64(kb))
        assert np.array_equal(m, m_ref)
        o_ref, ol_ref, _ = ora.forward(f64(qb), f64(kb), f64(vb), mask=m_ref, parts=True)
        for call, ref in ((gpu.forward, o_ref), (gpu.swa, ol_ref)):
            before = gpu.ctx.hf_slow_path_units()
            first = call(q, k, v)
            assert gpu.ctx.hf_slow_path_units() - before == len(far)
            hz.assert_close_out(first, ref, call.__name__)
            for _ in range(10):
                assert np.array_equal(call(q, k, v), first)
        assert gpu.ctx.hf_get_device_status() == (0, 0)
    finally:
        gpu.close()
