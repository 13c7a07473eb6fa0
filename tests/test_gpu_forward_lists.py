"""A forward call in one piece against its parts: selection alone (masks against the oracle), then attention and history term on the
selected lists as a caller would hand them in.  Bit for bit, at the edges of the units that share a merged list and of the shapes
for which pooling and selection are one launch."""
import numpy as np
import pytest

from paper_2604_10103_b200 import inputs as gen
from tests import harness as hz

pytestmark = pytest.mark.gpu

f64 = gen.bf16_bits_to_f64


@pytest.mark.parametrize("block,d,tokens,chunks,permille", [
    (16, 64, 5, 1, 1000), (16, 128, 128, 8, 300), (16, 64, 77, 3, 300), (16, 128, 129, 3, 300), (16, 64, 1021, 3, 250), (16, 128, 520, 8, 330),
    (64, 64, 64, 1, 1000), (64, 128, 65, 3, 340), (64, 64, 1000, 3, 250), (64, 128, 1025, 2, 400), (64, 64, 2048, 4, 300), (64, 128, 2049, 2, 250),
    (128, 64, 1, 2, 500), (128, 128, 128, 8, 300), (128, 64, 300, 4, 250), (128, 128, 513, 3, 200), (128, 64, 640, 8, 60), (128, 128, 640, 1, 1000),
    (128, 64, 641, 2, 500), (128, 128, 1024, 8, 120), (128, 64, 1024, 1, 300), (128, 128, 1025, 8, 120),
])
def test_forward_equals_its_parts(block, d, tokens, chunks, permille):
    import torch
    w = gen.Workload("parts", batch=1, heads=2, head_dim=d, tokens_per_frame=tokens, chunk_frames=1, window_frames=chunks, block=block, topk=0,
                     keep_permille=permille, seed=311)
    gpu = hz.GpuStream(w); ora = hz.make_oracle(w)
    try:
        for c in range(chunks):
            kc, vc = gen.clean_kv(w, 0, c)
            gpu.append(gpu.up(kc), gpu.up(vc)); ora.append(f64(kc), f64(vc))
        qb, kb, vb = gen.qkv(w, 0, chunks, 0)
        q, k, v = gpu.up(qb), gpu.up(kb), gpu.up(vb)
        whole, parts = torch.full_like(q, float("nan")), torch.full_like(q, float("nan"))
        gpu.ctx.hf_hybrid_forward(0, q, k, v, whole)
        m, idx, sc = gpu.select(q, k)
        m_ref, sc_ref = ora.select(f64(qb), f64(kb))
        assert np.array_equal(sc, sc_ref) and np.array_equal(m, m_ref)
        gpu.ctx.hf_sparse_swa_merged(0, q, k, v, parts, idx=torch.from_numpy(idx).cuda())
        torch.cuda.synchronize()
        assert torch.isfinite(whole.float()).all() and torch.equal(whole, parts)
        assert gpu.ctx.hf_get_device_status() == (0, 0)
    finally:
        gpu.close()
