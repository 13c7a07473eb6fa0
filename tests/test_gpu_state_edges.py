"""The state update at the edges of its reduction: split counts around the batches in which partials are fetched and around the line
between the two forms of the fold (more than 2 splits at head_dim 64, more than 3 at 128), one split, the most splits, on both
head dimensions, onto a state that is not zero; against the oracle's Eq. 3, and with a merge matrix the read-out of the folded
state against Eq. 4."""
import numpy as np
import pytest

from oracle import hybrid_attention as oa
from paper_2604_10103_b200 import inputs as gen
from tests import harness as hz

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("merge", [False, True])
@pytest.mark.parametrize("d", [64, 128])
def test_state_update_over_split_counts(d, merge):
    w = gen.Workload("state_edges", batch=1, heads=2, head_dim=d, tokens_per_frame=64, chunk_frames=1, window_frames=2, block=64, topk=1,
                     keep_permille=0, seed=17)
    gpu = hz.GpuStream(w, merge=merge)
    W = bias = None
    if merge:
        Wb, bb = gen.merge_weights(w, 0)
        W, bias = gen.bf16_bits_to_f64(Wb), gen.bf16_bits_to_f64(bb)
    qb = gen.normal_bf16((1, 2, w.chunk_tokens, d), 17, 99, 0)
    try:
        S, z = np.zeros((2, d, d)), np.zeros((2, d))
        for i, splits in enumerate([1, 2, 3, 4, 5, 6, 7, 12, 13, 32]):       # one 64-token tile per split, the last one short
            n = 64 * splits - (i % 3) * 21
            kb, vb = gen.normal_bf16((1, 2, n, d), 17, i, 1), gen.normal_bf16((1, 2, n, d), 17, i, 2)
            gpu.ctx.hf_state_absorb(0, gpu.up(kb), gpu.up(vb), n)
            for h in range(2):
                S[h], z[h] = oa.absorb(S[h], z[h], gen.bf16_bits_to_f64(kb)[0, h], gen.bf16_bits_to_f64(vb)[0, h])
            Sg, zg = gpu.state()
            assert hz.rel_l2(Sg[0], S) <= hz.STATE_REL_L2 and hz.rel_l2(zg[0], z) <= hz.STATE_REL_L2
            if merge:
                out = gpu.linear(gpu.up(qb))
                ref = np.stack([oa.linear_readout(gen.bf16_bits_to_f64(qb)[0, h], S[h], z[h], W[h], bias[h], w.eps) for h in range(2)])
                hz.assert_close_out(out[0], ref, f"read-out after {splits} splits")
    finally:
        gpu.close()
