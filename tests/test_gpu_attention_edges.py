"""The attention kernel at the edges of its tiling: units of one tile (the history products share its S buffer), lists longer than
the 32 entries of one tail window, a chunk shorter than a tile, ragged last blocks, units on the same thread block with a new
head in between; forward (selection + both branches in one kernel) and softmax branch with lse, against the oracle."""
import numpy as np
import pytest

from paper_2604_10103_b200 import inputs as gen
from paper_2604_10103_b200.binding import HF_SWA_MMA
from tests import harness as hz

pytestmark = pytest.mark.gpu

f64 = gen.bf16_bits_to_f64


@pytest.mark.parametrize("d,block,tpf,wf,topk,heads,batch", [
    (128, 128, 1000, 2, 1, 10, 2),     # one tile per unit, 160 units: two units on some thread blocks
    (64, 128, 1000, 2, 1, 10, 2),
    (64, 128, 100, 2, 2, 3, 1),        # one short block per chunk: every tile is a tail
    (128, 128, 520, 7, 35, 2, 1),      # all 35 blocks kept (last one of each chunk 8 tokens): two tail windows
    (64, 64, 130, 4, 1, 3, 1),         # small blocks, lists of one
    (128, 64, 330, 3, 5, 2, 1),
    (128, 16, 200, 3, 1, 2, 1),        # up to eight one-entry lists in a unit; last block 8 tokens
    (64, 16, 90, 5, 7, 2, 2),
])
def test_forward_at_tile_edges(d, block, tpf, wf, topk, heads, batch):
    w = gen.Workload("edges", batch=batch, heads=heads, head_dim=d, tokens_per_frame=tpf, chunk_frames=1, window_frames=wf, block=block,
                     topk=topk, keep_permille=0, seed=211)
    gpu = hz.GpuStream(w); ora = hz.make_oracle(w)
    try:
        for c in range(wf + 1):
            kc, vc = gen.clean_kv(w, 0, c)
            gpu.append(gpu.up(kc), gpu.up(vc)); ora.append(f64(kc), f64(vc))
        qb, kb, vb = gen.qkv(w, 0, wf + 1, 0)
        q, k, v = gpu.up(qb), gpu.up(kb), gpu.up(vb)
        m_gpu, _, _ = gpu.select(q, k)
        m_ref, _ = ora.select(f64(qb), f64(kb))
        assert np.array_equal(m_gpu, m_ref)
        o_ref, ol_ref, _ = ora.forward(f64(qb), f64(kb), f64(vb), mask=m_ref, parts=True)
        hz.assert_close_out(gpu.forward(q, k, v), o_ref, "hybrid O")
        o_local, lse = gpu.swa(q, k, v, want_lse=True)
        hz.assert_close_out(o_local, ol_ref, "softmax branch")
        assert np.isfinite(lse).all()
        assert gpu.ctx.hf_get_device_status() == (0, 0)
    finally:
        gpu.close()


@pytest.mark.parametrize("d,block", [(128, 128), (64, 128), (128, 64), (64, 64), (64, 16)])
@pytest.mark.parametrize("rope", [False, True])
def test_units_of_one_tile_whatever_arrives_first(d, block, rope):
    """Lists of one block, several units per thread block, and keys that arrive late (caches flushed, the queries touched again,
    copies beside the call): the next unit's queries must not take the place of a unit's that are still to be read.  Every call
    gives the same bits, and the warp-level kernel's results."""
    import torch
    w = gen.Workload("late_keys", batch=1, heads=12, head_dim=d, tokens_per_frame=1560, chunk_frames=2, window_frames=6, block=block,
                     topk=1, keep_permille=0, seed=227)
    gpu, ref = hz.GpuStream(w, rope=rope), hz.GpuStream(w, rope=rope, swa_kernel=HF_SWA_MMA)
    rng = torch.Generator(device="cuda").manual_seed(3)
    rand = lambda: torch.randn(gpu.shape, generator=rng, device="cuda").to(torch.bfloat16)
    try:
        for _ in range(4):
            kc, vc = rand(), rand()
            gpu.append(kc, vc); ref.append(kc, vc)
        q, k, v, o = rand(), rand(), rand(), torch.empty(gpu.shape, dtype=torch.bfloat16, device="cuda")
        hz.assert_close_out(gpu.forward(q, k, v), ref.forward(q, k, v), "against the warp-level kernel")
        gpu.ctx.hf_sparse_swa_merged(0, q, k, v, o)
        torch.cuda.synchronize()
        first, side = o.clone(), torch.cuda.Stream()
        big = [torch.zeros(1 << 27, dtype=torch.int32, device="cuda") for _ in range(2)]
        wrong = 0
        for it in range(60):
            big[0].fill_(it)
            q.add_(0)
            torch.cuda.synchronize()
            if it % 2:
                with torch.cuda.stream(side):
                    big[1].copy_(big[0])
            gpu.ctx.hf_sparse_swa_merged(0, q, k, v, o)
            torch.cuda.synchronize()
            wrong += not torch.equal(o, first)
        assert wrong == 0, f"{wrong} of 60 calls gave other results"
        assert gpu.ctx.hf_get_device_status() == (0, 0)
    finally:
        gpu.close(); ref.close()


@pytest.mark.parametrize("d,block", [(128, 128), (64, 128), (128, 64), (64, 16)])
def test_rotated_history_in_both_passes(d, block):
    """The rotated numerator of the history term inside the attention kernel, in its tile stream and in the second pass (the
    newest keys rise ~180 nats above the first kept block for half of the queries)."""
    w = gen.Workload("rot_edges", batch=1, heads=2, head_dim=d, tokens_per_frame=300, chunk_frames=1, window_frames=2, block=block,
                     topk=0, keep_permille=600, seed=223)
    gpu = hz.GpuStream(w, rope=True); ora = hz.make_oracle(w, rope=True)
    u = gen.direction(w, 0)
    a = (180.0 / d ** 0.5) ** 0.5
    try:
        for c in range(4):
            kc, vc = gen.clean_kv(w, 0, c)
            gpu.append(gpu.up(kc), gpu.up(vc)); ora.append(f64(kc), f64(vc))
        qb, kb, vb = gen.qkv(w, 0, 4, 0)
        qb = gen.shifted(qb, u, a, slice(0, 128)); kb = gen.shifted(kb, u, a, slice(256, None))
        q, k, v = gpu.up(qb), gpu.up(kb), gpu.up(vb)
        m_gpu, _, _ = gpu.select(q, k)
        m_ref, _ = ora.select(f64(qb), f64(kb))
        assert np.array_equal(m_gpu, m_ref)
        hz.assert_close_out(gpu.forward(q, k, v), ora.forward(f64(qb), f64(kb), f64(vb), mask=m_ref), "hybrid O, rotated")
        assert gpu.ctx.hf_slow_path_units() > 0
        assert gpu.ctx.hf_get_device_status() == (0, 0)
    finally:
        gpu.close()


@pytest.mark.parametrize("d,tpf", [(128, 300), (64, 300), (128, 100)])
def test_an_entry_outside_the_window_is_block_0(d, tpf):
    """A list entry outside [0, T_n) is reported, and read as block 0, a full one or (one block per chunk) a short one: forward
    and dq give what the same list with 0 in its place gives.  -1, the entry behind the last block and one whose index + 1 is a
    multiple of the blocks per chunk are told apart from a chunk's short last block."""
    import torch
    w = gen.Workload("bad_entry", batch=1, heads=2, head_dim=d, tokens_per_frame=tpf, chunk_frames=1, window_frames=3, block=128,
                     topk=3, keep_permille=0, seed=229)
    gpu = hz.GpuStream(w)
    try:
        for c in range(3):
            kc, vc = gen.clean_kv(w, 0, c)
            gpu.append(gpu.up(kc), gpu.up(vc))
        q, k, v = (gpu.up(x) for x in gen.qkv(w, 0, 3, 0))
        g = gpu.up(gen.normal_bf16(tuple(gpu.shape), 229, 7, 7))
        tn, nb = gpu.ctx.hf_query(0, gpu.hf.HF_Q_KEY_BLOCKS), w.blocks_per_chunk
        _, idx0, _ = gpu.select(q, k)
        for bad in (-1, tn, tn + nb - 1, 2 ** 30):
            lists = {}
            for value in (0, bad):
                idx = idx0.copy()
                idx[0, :, :, 1] = value
                lists[value] = torch.from_numpy(idx).cuda()
            outs = {}
            for value, idx in lists.items():
                o, lse = gpu.swa(q, k, v, idx=idx, want_lse=True)
                ot, lt = torch.from_numpy(o).to(torch.bfloat16).cuda(), torch.from_numpy(lse).cuda()
                dq = torch.empty_like(q)
                gpu.ctx.hf_sparse_swa_backward_dq(0, q, k, v, ot, lt, g, dq, idx=idx)
                outs[value] = (o, lse, gpu.f64(dq))
                if value == 0:
                    assert gpu.ctx.hf_get_device_status() == (0, 0)
                else:
                    with pytest.raises(gpu.hf.HFError, match="HF_ERR_INVALID_ARG"):
                        gpu.ctx.hf_get_device_status()
            for a, b in zip(outs[0], outs[bad]):
                assert np.array_equal(a, b), f"entry {bad}"
    finally:
        gpu.close()


@pytest.mark.parametrize("units", [1, 5, 8, 9])
def test_only_the_listed_units_are_computed_again(units):
    """Ten units on one thread block, some with a block ~180 nats above the first kept one: up to eight of them are computed again
    and nothing else is; with a ninth all ten are.  Results are those of the warp-level kernel."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    d, n_b = 128, 21
    heads = -(-9 * sms // n_b) + 1
    w = gen.Workload("redo_list", batch=1, heads=heads, head_dim=d, tokens_per_frame=128 * n_b, chunk_frames=1, window_frames=1, block=128,
                     topk=2, keep_permille=0, seed=233)
    gpu = hz.GpuStream(w, merge=False)
    ref = hz.GpuStream(w, merge=False, swa_kernel=HF_SWA_MMA)
    rng = torch.Generator(device="cuda").manual_seed(7)
    rand = lambda: torch.randn(gpu.shape, generator=rng, device="cuda")
    try:
        q, k, v = rand(), rand(), rand().to(torch.bfloat16)
        a = (180.0 / d ** 0.5) ** 0.5               # a^2 d / sqrt(d) = 180
        k[:, :, -128:] += a                         # the last block: a few nats for queries that do not look for it
        total = heads * n_b
        mine = list(range(0, total, sms))           # units of the first thread block
        assert len(mine) == 10
        for u in mine[:units]:
            h, i = divmod(u, n_b)
            assert i != n_b - 1
            q[0, h, 128 * i:128 * (i + 1)] += a
        q, k = q.to(torch.bfloat16), k.to(torch.bfloat16)
        _, idx, _ = gpu.select(q, k); ref.select(q, k)
        o, r = gpu.swa(q, k, v), ref.swa(q, k, v)
        assert gpu.ctx.hf_slow_path_units() == (units if units <= 8 else len(mine))
        hz.assert_close_out(o, r, "against the warp-level kernel")
        assert gpu.ctx.hf_get_device_status() == (0, 0)
    finally:
        gpu.close(); ref.close()
