"""Two and four column groups of the softmax warps at head dim 64: on both sides of the line between them, short last blocks that end
inside, at and past the edges of a group's columns, whole windows of one kept block up to all of them.  Softmax branch with its row
log-sums against the warp-level kernel on the same lists, merged output against the oracle."""
import numpy as np
import pytest

from paper_2604_10103_b200 import inputs as gen
from tests import harness as hz

pytestmark = pytest.mark.gpu

f64 = gen.bf16_bits_to_f64


@pytest.mark.parametrize("topk", [1, 4, 5, 9])
@pytest.mark.parametrize("tail", [1, 31, 32, 33, 64, 65, 96, 97, 128])
def test_column_groups(topk, tail):
    import torch
    w = gen.Workload("groups", batch=1, heads=2, head_dim=64, tokens_per_frame=256 + tail, chunk_frames=1, window_frames=3, block=128, topk=topk,
                     keep_permille=0, seed=353)
    gpu, ref, ora = hz.GpuStream(w), hz.GpuStream(w, swa_kernel=1), hz.make_oracle(w)
    try:
        for c in range(4):
            kc, vc = gen.clean_kv(w, 0, c)
            gpu.append(gpu.up(kc), gpu.up(vc)); ref.append(ref.up(kc), ref.up(vc)); ora.append(f64(kc), f64(vc))
        qb, kb, vb = gen.qkv(w, 0, 4, 0)
        q, k, v = gpu.up(qb), gpu.up(kb), gpu.up(vb)
        m, idx, _ = gpu.select(q, k)
        o, lse = gpu.swa(q, k, v, want_lse=True)
        o_ref, lse_ref = ref.swa(q, k, v, idx=torch.from_numpy(idx).cuda(), want_lse=True)
        hz.assert_close_out(o, o_ref, "softmax branch")
        assert np.abs(lse - lse_ref).max() <= 1e-3          # fp32 sums of up to 1 152 terms in another order: below 1e-4
        hz.assert_close_out(gpu.forward(q, k, v), ora.forward(f64(qb), f64(kb), f64(vb), mask=m), "merged")
        assert gpu.ctx.hf_get_device_status() == (0, 0)
    finally:
        gpu.close(); ref.close()
