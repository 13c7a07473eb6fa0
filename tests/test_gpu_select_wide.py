"""Selection on both sides of 512 key blocks (ranking registers for 512, then 1 024) and with query blocks that do not fill a group of
eight: the checks of the narrower edges, bit for bit against the oracle."""
import pytest

from tests.test_gpu_select_edges import test_selection_at_tile_edges as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n_b,wf,topk", [(64, 64, 8, 100), (128, 65, 8, 519), (64, 65, 4, 1), (128, 33, 8, 264)])
@pytest.mark.parametrize("ties", [False, True])
def test_wide_windows(d, n_b, wf, topk, ties):
    check(d, n_b, wf, topk, ties)


@pytest.mark.parametrize("d,tokens,wf,topk", [(128, 300, 8, 10), (64, 640, 8, 33), (128, 640, 1, 2), (64, 100, 7, 6)])
def test_short_heads_with_equal_scores(d, tokens, wf, topk):
    """128-token blocks of heads that pool and select in one launch: every full key block of a chunk has the same mean, ties go to the
    lowest index."""
    import numpy as np
    from paper_2604_10103_b200 import inputs as gen
    from tests import harness as hz
    f64 = gen.bf16_bits_to_f64
    w = gen.Workload("sel_short", batch=1, heads=3, head_dim=d, tokens_per_frame=tokens, chunk_frames=1, window_frames=wf, block=128, topk=topk,
                     keep_permille=0, seed=359)
    gpu = hz.GpuStream(w); ora = hz.make_oracle(w)
    level = lambda bits, c: np.full_like(bits, gen.f32_to_bf16_bits(np.array([0.5 + (c % 2)], np.float32))[0])  # noqa: E731
    try:
        for c in range(wf - 1):
            kc, vc = gen.clean_kv(w, 0, c)
            gpu.append(gpu.up(level(kc, c)), gpu.up(vc)); ora.append(f64(level(kc, c)), f64(vc))
        qb, kb, _ = gen.qkv(w, 0, wf, 0)
        m, idx, sc = gpu.select(gpu.up(qb), gpu.up(level(kb, 1)))
        m_ref, sc_ref = ora.select(f64(qb), f64(level(kb, 1)))
        assert np.array_equal(sc, sc_ref) and np.array_equal(m, m_ref)
        assert np.array_equal(idx, np.nonzero(m_ref)[3].reshape(idx.shape))
    finally:
        gpu.close()
