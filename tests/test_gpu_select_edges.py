"""Block selection at the edges of its tiling: one score or two per thread (64 key blocks), one or several passes of 128 key
rows, 4 / 8 / 32 score images per lane of the ranking warp, query blocks that do not fill a group of four, one block kept and
all kept, equal scores.  Scores, masks and index lists bit for bit against the oracle."""
import numpy as np
import pytest

from paper_2604_10103_b200 import inputs as gen
from tests import harness as hz

pytestmark = pytest.mark.gpu

f64 = gen.bf16_bits_to_f64


@pytest.mark.parametrize("d,n_b,wf,topk", [
    (64, 1, 1, 1), (128, 3, 1, 3), (128, 32, 1, 1), (64, 33, 1, 32), (128, 64, 1, 20), (64, 65, 1, 65), (128, 32, 4, 127),
    (64, 43, 3, 1), (128, 43, 3, 60), (64, 64, 4, 255), (128, 37, 7, 64), (64, 128, 8, 300), (128, 128, 8, 1023),
])
@pytest.mark.parametrize("ties", [False, True])
def test_selection_at_tile_edges(d, n_b, wf, topk, ties):
    w = gen.Workload("sel", batch=1, heads=2, head_dim=d, tokens_per_frame=16 * n_b - 5 if n_b > 1 else 11, chunk_frames=1, window_frames=wf,
                     block=16, topk=topk, keep_permille=0, seed=307)
    gpu = hz.GpuStream(w); ora = hz.make_oracle(w)
    # equal scores: key tensors of one value per chunk give every full block of a chunk the same mean
    level = lambda bits, c: np.full_like(bits, gen.f32_to_bf16_bits(np.array([0.5 + (c % 2)], np.float32))[0]) if ties else bits  # noqa: E731
    try:
        for c in range(wf - 1):
            kc, vc = gen.clean_kv(w, 0, c)
            kc = level(kc, c)
            gpu.append(gpu.up(kc), gpu.up(vc)); ora.append(f64(kc), f64(vc))
        qb, kb, _ = gen.qkv(w, 0, wf, 0)
        kb = level(kb, 1)
        m, idx, sc = gpu.select(gpu.up(qb), gpu.up(kb))
        m_ref, sc_ref = ora.select(f64(qb), f64(kb))
        assert np.array_equal(sc, sc_ref) and np.array_equal(m, m_ref)
        assert np.array_equal(idx, np.nonzero(m_ref)[3].reshape(idx.shape))
    finally:
        gpu.close()
