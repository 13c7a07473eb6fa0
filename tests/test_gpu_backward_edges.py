"""Backward kernels at the edges of their tiling: key blocks that no query block keeps between ones that some do, several units
per thread block, more than 32 query blocks (two words of the pair walk), chunks of one short block, one-block lists.  dq, dk and
dv against the oracle's gradients (bf16 P and dS operands: the tolerance of the other backward tests)."""
import numpy as np
import pytest

from oracle import hybrid_attention as oa
from paper_2604_10103_b200 import inputs as gen
from tests import harness as hz

pytestmark = pytest.mark.gpu

f64 = gen.bf16_bits_to_f64


@pytest.mark.parametrize("d,tpf,wf,topk,heads,batch", [
    (128, 1290, 2, 1, 16, 1),      # 176 units, most key blocks unkept
    (64, 1290, 2, 2, 16, 1),
    (128, 4300, 1, 3, 2, 1),       # 34 query blocks
    (64, 77, 2, 1, 3, 1),          # one short block per chunk
    (128, 200, 5, 9, 2, 1),        # 72-row last block; nine of ten blocks kept
    (64, 4300, 1, 33, 1, 1),
])
def test_gradients_at_tile_edges(d, tpf, wf, topk, heads, batch):
    import torch
    w = gen.Workload("bwd_edges", batch=batch, heads=heads, head_dim=d, tokens_per_frame=tpf, chunk_frames=1, window_frames=wf, block=128,
                     topk=topk, keep_permille=0, seed=401)
    gpu = hz.GpuStream(w); ora = hz.make_oracle(w)
    try:
        for c in range(wf):
            kc, vc = gen.clean_kv(w, 0, c)
            gpu.append(gpu.up(kc), gpu.up(vc)); ora.append(f64(kc), f64(vc))
        qb, kb, vb = gen.qkv(w, 0, wf, 0)
        gb = gen.normal_bf16(qb.shape, 401, 7, 7)
        q, k, v, g = gpu.up(qb), gpu.up(kb), gpu.up(vb), gpu.up(gb)
        m, _, _ = gpu.select(q, k)
        o = torch.empty(gpu.shape, dtype=torch.bfloat16, device="cuda")
        lse = torch.empty(gpu.shape[:3], dtype=torch.float32, device="cuda")
        gpu.ctx.hf_sparse_swa(0, q, k, v, o, lse=lse)
        dq, dk, dv = torch.empty_like(o), torch.full_like(o, 7.0), torch.full_like(o, 7.0)
        gpu.ctx.hf_sparse_swa_backward_dq(0, q, k, v, o, lse, g, dq)
        gpu.ctx.hf_sparse_swa_backward_dkv(0, q, k, v, o, lse, g, dk, dv)
        torch.cuda.synchronize()
        assert gpu.ctx.hf_get_device_status() == (0, 0)
        got = [gpu.f64(x) for x in (dq, dk, dv)]
        ref = [np.empty_like(got[0]) for _ in got]
        held = ora.sink + ora.past
        for bi in range(batch):
            for h in range(heads):
                kc_ = [kp[bi, h] for kp, _ in held] + [f64(kb)[bi, h]]
                vc_ = [vp[bi, h] for _, vp in held] + [f64(vb)[bi, h]]
                rq, rk, rv = oa.sparse_attention_backward(f64(qb)[bi, h], kc_, vc_, w.block, m[bi, h], f64(gb)[bi, h])
                ref[0][bi, h], ref[1][bi, h], ref[2][bi, h] = rq, rk[-1], rv[-1]
        for name, a, b in zip(("dq", "dk", "dv"), got, ref):
            rl, ma = hz.rel_l2(a, b), hz.max_abs(a, b)
            assert rl <= 1e-2 and ma <= 2e-2 * max(1.0, np.abs(b).max()), f"{name}: rel-L2 {rl:.3e}, max-abs {ma:.3e}"
        unkept = ~m[..., -w.blocks_per_chunk:].any(axis=2)
        for bi, h, jb in zip(*np.nonzero(unkept)):
            assert not got[1][bi, h, jb * 128:(jb + 1) * 128].any() and not got[2][bi, h, jb * 128:(jb + 1) * 128].any()
    finally:
        gpu.close()


@pytest.mark.parametrize("d", [64, 128])
def test_ds_is_rounded_with_its_factor(d):
    """dS = P (dP - delta) / sqrt(d) is rounded to bf16 as a whole.  The same products in 64 bits with that one rounding give the
    same bf16 numbers but for a few (float32 against 64-bit sums in front of a rounding: 2^-24 against 2^-9, a few per mille);
    with the factor applied after the rounding every other value of dq and dk is a neighbouring number at d = 128."""
    import torch
    w = gen.Workload("bwd_rounding", batch=1, heads=2, head_dim=d, tokens_per_frame=512, chunk_frames=1, window_frames=1, block=128, topk=4,
                     keep_permille=0, seed=409)
    gpu = hz.GpuStream(w)
    try:
        q, k, v = (gpu.up(x) for x in gen.qkv(w, 0, 0, 0))
        g = gpu.up(gen.normal_bf16((1, 2, 512, d), 409, 7, 7))
        gpu.select(q, k)
        o, dq, dk, dv = (torch.empty_like(q) for _ in range(4))
        lse = torch.empty(gpu.shape[:3], dtype=torch.float32, device="cuda")
        gpu.ctx.hf_sparse_swa(0, q, k, v, o, lse=lse)
        gpu.ctx.hf_sparse_swa_backward_dq(0, q, k, v, o, lse, g, dq)
        gpu.ctx.hf_sparse_swa_backward_dkv(0, q, k, v, o, lse, g, dk, dv)
        torch.cuda.synchronize()
        Q, K, V, G, O = (x.cpu().double() for x in (q, k, v, g, o))
        P = torch.exp(Q @ K.mT / d ** 0.5 - lse.cpu().double()[..., None])
        dS = (P * (G @ V.mT - (G * O).sum(-1, keepdim=True)) / d ** 0.5).to(torch.bfloat16).double()
        for name, got, ref in (("dq", dq, dS @ K), ("dk", dk, dS.mT @ Q)):
            differ = float((got.cpu() != ref.to(torch.bfloat16)).double().mean())
            assert differ < 0.05, f"{name}: {100 * differ:.1f} % of the values are other bf16 numbers"
    finally:
        gpu.close()


def test_more_units_than_are_put_in_order():
    """4 200 key blocks of the chunk: beyond the sort's capacity, each warp counts a unit's pairs itself.  A head's gradients do
    not depend on how many others there are, so they equal, bit for bit, those of a context with six heads."""
    import torch
    rng = torch.Generator(device="cuda").manual_seed(5)
    full = [torch.randn((2, 350, 700, 64), generator=rng, device="cuda").to(torch.bfloat16) for _ in range(4)]

    def gradients(batch, heads):
        w = gen.Workload("bwd_many", batch=batch, heads=heads, head_dim=64, tokens_per_frame=700, chunk_frames=1, window_frames=1, block=128,
                         topk=2, keep_permille=0, seed=402)
        gpu = hz.GpuStream(w)
        try:
            q, k, v, g = [x[:batch, :heads].contiguous() for x in full]
            gpu.append(k, v)
            gpu.select(q, k)
            o, lse = torch.empty_like(q), torch.empty(q.shape[:3], dtype=torch.float32, device="cuda")
            gpu.ctx.hf_sparse_swa(0, q, k, v, o, lse=lse)
            dk, dv = torch.full_like(q, 7.0), torch.full_like(q, 7.0)
            gpu.ctx.hf_sparse_swa_backward_dkv(0, q, k, v, o, lse, g, dk, dv)
            torch.cuda.synchronize()
            assert gpu.ctx.hf_get_device_status() == (0, 0)
            return dk[:1, :6].cpu(), dv[:1, :6].cpu()
        finally:
            gpu.close()

    for a, b in zip(gradients(2, 350), gradients(1, 6)):
        assert torch.equal(a, b) and float(b.float().abs().max()) > 0


@pytest.mark.parametrize("d,tpf,heads,batch", [
    (128, 2330, 24, 1),            # four tiles per thread block: every buffer used again; heads change within a range; 26-row last tile
    (64, 1025, 30, 2),             # the same at head_dim 64, one-row last tile
])
def test_read_out_and_its_gradient_at_tile_edges(d, tpf, heads, batch):
    import torch
    w = gen.Workload("bwdh_edges", batch=batch, heads=heads, head_dim=d, tokens_per_frame=tpf, chunk_frames=1, window_frames=1, block=128,
                     topk=1, keep_permille=0, seed=403)
    gpu = hz.GpuStream(w); ora = hz.make_oracle(w)
    try:
        for c in range(2):
            kc, vc = gen.clean_kv(w, 0, c)
            gpu.append(gpu.up(kc), gpu.up(vc)); ora.append(f64(kc), f64(vc))
        qb, _, _ = gen.qkv(w, 0, 2, 0)
        gb = gen.normal_bf16(qb.shape, 403, 7, 7)
        q, g = gpu.up(qb), gpu.up(gb)
        dq, y = torch.empty_like(q), torch.empty_like(q)
        gpu.ctx.hf_linear_attn(0, q, y)
        gpu.ctx.hf_linear_attn_backward_dq(0, q, g, dq)
        torch.cuda.synchronize()
        assert gpu.ctx.hf_get_device_status() == (0, 0)
        got, got_y, qf, gf = gpu.f64(dq), gpu.f64(y), f64(qb), f64(gb)
        for bi in range(batch):
            for h in range(heads):
                ref = oa.linear_readout_backward(qf[bi, h], ora.S[bi, h], ora.z[bi, h], gf[bi, h],
                                                 W=None if ora.W is None else ora.W[h], eps=ora.eps)[0]
                out = oa.linear_readout(qf[bi, h], ora.S[bi, h], ora.z[bi, h], W=None if ora.W is None else ora.W[h],
                                        bias=None if ora.bias is None else ora.bias[h], eps=ora.eps)
                for name, a, b in (("dq", got[bi, h], ref), ("y", got_y[bi, h], out)):
                    rl, ma = hz.rel_l2(a, b), hz.max_abs(a, b)
                    assert rl <= 1e-2 and ma <= 2e-2 * max(1.0, np.abs(b).max()), f"{name} ({bi}, {h}): rel-L2 {rl:.3e}, max-abs {ma:.3e}"
    finally:
        gpu.close()


@pytest.mark.parametrize("first,then", [("dq", "dkv"), ("dkv", "dq"), (None, "dq"), (None, "dkv")])
def test_backward_into_a_graph(first, then):
    """Neither backward call allocates: each can be captured, after the other or as the first, and the replay gives its bits."""
    import torch
    w = gen.Workload("bwd_graph", batch=1, heads=2, head_dim=128, tokens_per_frame=300, chunk_frames=1, window_frames=2, block=128, topk=2,
                     keep_permille=0, seed=419)
    gpu = hz.GpuStream(w)
    try:
        q, k, v = (gpu.up(x) for x in gen.qkv(w, 0, 0, 0))
        g = gpu.up(gen.normal_bf16(tuple(gpu.shape), 419, 7, 7))
        gpu.select(q, k)
        o, dq, dk, dv = (torch.empty_like(q) for _ in range(4))
        lse = torch.empty(gpu.shape[:3], dtype=torch.float32, device="cuda")
        gpu.ctx.hf_sparse_swa(0, q, k, v, o, lse=lse)
        calls = {"dq": (lambda: gpu.ctx.hf_sparse_swa_backward_dq(0, q, k, v, o, lse, g, dq), [dq]),
                 "dkv": (lambda: gpu.ctx.hf_sparse_swa_backward_dkv(0, q, k, v, o, lse, g, dk, dv), [dk, dv])}
        if first:
            calls[first][0]()
        torch.cuda.synchronize()
        call, outs = calls[then]
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            call()
        graph.replay()
        torch.cuda.synchronize()
        replayed = [t.clone() for t in outs]
        call()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(replayed, outs))
    finally:
        gpu.close()
