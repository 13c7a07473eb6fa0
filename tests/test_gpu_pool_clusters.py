"""Pooling and selection by clusters of twelve to sixteen thread blocks (above the portable eight), up to the longest window they see
(T_n 128), and on both sides of the line between one launch and two: scores, masks and lists bit for bit against the oracle."""
import numpy as np
import pytest

from paper_2604_10103_b200 import inputs as gen
from tests import harness as hz
from tests.test_gpu_forward_lists import test_forward_equals_its_parts as check

pytestmark = pytest.mark.gpu

f64 = gen.bf16_bits_to_f64


@pytest.mark.parametrize("d,tokens,chunks,permille", [
    (128, 1500, 8, 120), (64, 1500, 1, 500),           # T_m 12
    (64, 1921, 8, 100), (128, 1793, 1, 1000),          # T_m 16 and 15 with a last block of one token
    (128, 1920, 8, 250), (64, 2048, 8, 60),            # T_m 15; T_m 16 and T_n 128
    (128, 2048, 8, 1000), (128, 2048, 1, 300),
])
def test_large_clusters(d, tokens, chunks, permille):
    check(128, d, tokens, chunks, permille)


@pytest.mark.parametrize("d,tokens,heads,launches", [
    (64, 500, 61, 1), (64, 500, 72, 2), (128, 500, 61, 1), (128, 500, 72, 2),            # T_m 4: 71 clusters resident on 148 SMs
    (64, 1300, 16, 1), (64, 1300, 19, 2), (128, 1300, 14, 1), (128, 1300, 15, 2),        # T_m 11: about the room of 16
    (64, 77, 600, 1),                                  # a single block a head: any grid
])
def test_both_sides_of_one_wave(d, tokens, heads, launches):
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the line is that of 148 SMs")
    w = gen.Workload("wave", batch=1, heads=heads, head_dim=d, tokens_per_frame=tokens, chunk_frames=1, window_frames=2, block=128, topk=0,
                     keep_permille=400, seed=421)
    gpu, ora = hz.GpuStream(w), hz.make_oracle(w)
    try:
        kc, vc = gen.clean_kv(w, 0, 0)
        gpu.append(gpu.up(kc), gpu.up(vc)); ora.append(f64(kc), f64(vc))
        qb, kb, _ = gen.qkv(w, 0, 1, 0)
        before = gpu.ctx.hf_launch_count()
        m, idx, sc = gpu.select(gpu.up(qb), gpu.up(kb))
        assert gpu.ctx.hf_launch_count() - before == launches
        m_ref, sc_ref = ora.select(f64(qb), f64(kb))
        assert np.array_equal(sc, sc_ref) and np.array_equal(m, m_ref)
        assert np.array_equal(idx, np.nonzero(m_ref)[3].reshape(idx.shape))
    finally:
        gpu.close()
