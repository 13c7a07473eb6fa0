"""Selection over 129 to 256 key blocks, all key rows in shared memory at once: four query blocks a thread block, eight where the grid is large, numbers of
query blocks that fill neither, and the ends of the range; with the lists merged for blocks of 64 and 16 tokens.  Masks and scores bit for bit."""
import numpy as np
import pytest

from paper_2604_10103_b200 import inputs as gen
from tests import harness as hz
from tests.test_gpu_select_edges import test_selection_at_tile_edges as check

pytestmark = pytest.mark.gpu

f64 = gen.bf16_bits_to_f64


@pytest.mark.parametrize("d,n_b,wf,topk", [(128, 43, 3, 1), (64, 64, 4, 200), (128, 37, 6, 111), (64, 51, 5, 255)])
@pytest.mark.parametrize("ties", [False, True])
def test_windows(d, n_b, wf, topk, ties):
    check(d, n_b, wf, topk, ties)


@pytest.mark.parametrize("heads,d,tokens,block,wf,topk", [(2, 128, 43 * 64 + 5, 64, 4, 30), (40, 64, 43 * 64 - 1, 64, 3, 60), (3, 128, 43 * 16 + 1, 16, 3, 129),
                                                          (40, 64, 64 * 16, 16, 4, 40)])
def test_forward_on_merged_lists(heads, d, tokens, block, wf, topk):
    w = gen.Workload("sel256", batch=1, heads=heads, head_dim=d, tokens_per_frame=tokens, chunk_frames=1, window_frames=wf, block=block, topk=topk,
                     keep_permille=0, seed=823)
    gpu, ref = hz.GpuStream(w), hz.GpuStream(w, swa_kernel=1)
    try:
        for c in range(wf - 1):
            kc, vc = gen.clean_kv(w, 0, c)
            gpu.append(gpu.up(kc), gpu.up(vc)); ref.append(ref.up(kc), ref.up(vc))
        qb, kb, vb = gen.qkv(w, 0, wf, 0)
        q, k, v = gpu.up(qb), gpu.up(kb), gpu.up(vb)
        m, _, sc = gpu.select(q, k)
        m_ref, _, sc_ref = ref.select(q, k)
        assert np.array_equal(m, m_ref) and np.array_equal(sc, sc_ref) and (m.sum(-1) == topk).all()
        hz.assert_close_out(gpu.forward(q, k, v), ref.forward(q, k, v), "merged lists against the warp-level kernel")
        assert gpu.ctx.hf_get_device_status() == (0, 0)
    finally:
        gpu.close(); ref.close()
