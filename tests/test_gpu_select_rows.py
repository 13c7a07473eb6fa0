"""Selection over 129 to 256 key blocks with four and with eight query blocks a thread block on grids of more thread blocks than SMs, query blocks that fill neither,
head dims 64 and 128, equal scores.  Scores, masks and lists bit for bit against the oracle; the forms with merged lists by the forward call
against the warp-level kernel on the lists checked here."""
import numpy as np
import pytest

from paper_2604_10103_b200 import inputs as gen
from tests import harness as hz
from tests.test_select_rows_rule import rules  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

f64 = gen.bf16_bits_to_f64


@pytest.mark.parametrize("heads,d,n_b,wf,topk,block,rows", [
    (20, 64, 43, 3, 40, 16, 8), (20, 128, 43, 3, 129, 16, 8), (20, 64, 37, 6, 55, 16, 8), (20, 128, 37, 6, 111, 16, 8), (30, 64, 43, 3, 1, 16, 4), (32, 64, 37, 6, 100, 16, 4),
    (14, 128, 43, 3, 30, 64, 8), (28, 64, 43, 3, 30, 64, 4), (36, 128, 43, 3, 20, 64, 4)])
@pytest.mark.parametrize("ties", [False, True])
def test_rows(rules, heads, d, n_b, wf, topk, block, rows, ties):  # noqa: F811
    assert rules.rows_of(1, d, n_b * wf, n_b, heads) == rows and (block == 16 or rules.rows_of(2, d, n_b * wf, n_b, heads) == rows)
    w = gen.Workload("rows", batch=1, heads=heads, head_dim=d, tokens_per_frame=block * n_b - 5, chunk_frames=1, window_frames=wf, block=block, topk=topk,
                     keep_permille=0, seed=307)
    gpu, ref, ora = hz.GpuStream(w), hz.GpuStream(w, swa_kernel=1), hz.make_oracle(w)
    # equal scores: key tensors of one value per chunk give every full block of a chunk the same mean
    level = lambda bits, c: np.full_like(bits, gen.f32_to_bf16_bits(np.array([0.5 + (c % 2)], np.float32))[0]) if ties else bits  # noqa: E731
    try:
        for c in range(wf - 1):
            kc, vc = gen.clean_kv(w, 0, c)
            kc = level(kc, c)
            gpu.append(gpu.up(kc), gpu.up(vc)); ref.append(ref.up(kc), ref.up(vc)); ora.append(f64(kc), f64(vc))
        qb, kb, vb = gen.qkv(w, 0, wf, 0)
        kb = level(kb, 1)
        q, k, v = gpu.up(qb), gpu.up(kb), gpu.up(vb)
        m, idx, sc = gpu.select(q, k)
        m_ref, sc_ref = ora.select(f64(qb), f64(kb))
        assert np.array_equal(sc, sc_ref) and np.array_equal(m, m_ref)
        assert np.array_equal(idx, np.nonzero(m_ref)[3].reshape(idx.shape))
        hz.assert_close_out(gpu.forward(q, k, v), ref.forward(q, k, v), "forward")
        assert gpu.ctx.hf_get_device_status() == (0, 0)
    finally:
        gpu.close(); ref.close()
