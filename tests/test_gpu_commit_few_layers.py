"""The layer-batched commit and state update with fewer (layer, head) items than SMs, on both sides of the line between one persistent
launch and a launch per layer: state, cache and forwards equal the per-layer calls bit for bit.  And the copy of the state out."""
import numpy as np
import pytest

from paper_2604_10103_b200 import inputs as gen

pytestmark = pytest.mark.gpu


def _same(a, b, w, chunk):
    import torch
    for layer in range(w.layers):
        st = []
        for ctx in (a, b):
            S = torch.empty(w.batch, w.heads, w.head_dim, w.head_dim, dtype=torch.float32, device="cuda")
            z = torch.empty(w.batch, w.heads, w.head_dim, dtype=torch.float32, device="cuda")
            ctx.hf_get_state(layer, S, z)
            o = torch.empty(w.batch, w.heads, w.chunk_tokens, w.head_dim, dtype=torch.bfloat16, device="cuda")
            ctx.hf_hybrid_forward(layer, *chunk, o)
            st.append((S, z, o))
        for x, y in zip(*st):
            assert torch.equal(x, y)


@pytest.mark.parametrize("d,heads,tokens,sink,layers", [
    (128, 8, 300, 0, 4), (64, 2, 63, 0, 2), (64, 5, 65, 1, 3), (128, 12, 1000, 0, 2), (128, 2, 4000, 0, 2), (64, 1, 1500, 0, 6),
])
def test_commit_of_few_layers(d, heads, tokens, sink, layers):
    import torch
    from paper_2604_10103_b200 import binding as hf
    w = gen.Workload("few", batch=1, heads=heads, head_dim=d, tokens_per_frame=tokens, chunk_frames=1, window_frames=2, block=128, topk=0,
                     keep_permille=500, layers=layers, seed=313)
    a, b = (hf.Context(hf.make_config(w, sink_frames=sink)) for _ in range(2))
    try:
        for ctx in (a, b):
            for layer in range(layers):
                Wb, bb = gen.merge_weights(w, layer)
                ctx.hf_set_merge_weights(layer, hf.bits_to_cuda(Wb), hf.bits_to_cuda(bb))
        for c in range(sink + 4):
            kv = [[hf.bits_to_cuda(x) for x in gen.clean_kv(w, layer, c)] for layer in range(layers)]
            a.hf_kv_append_layers(0, [k for k, _ in kv], [v for _, v in kv])
            for layer, (k, v) in enumerate(kv):
                b.hf_kv_append(layer, k, v)
        k_ev, v_ev = (torch.stack([x[i] for x in kv]).contiguous() for i in range(2))
        a.hf_state_absorb_layers(0, layers, k_ev, v_ev, w.chunk_tokens)
        for layer in range(layers):
            b.hf_state_absorb(layer, k_ev[layer], v_ev[layer], w.chunk_tokens)
        _same(a, b, w, [hf.bits_to_cuda(x) for x in gen.qkv(w, 0, 9, 0)])
        assert a.hf_get_device_status() == (0, 0)
    finally:
        a.close(); b.close()


def test_commit_of_few_layers_in_a_graph():
    """The first evicting commit of a context may be captured: nothing is allocated in it."""
    import torch
    from paper_2604_10103_b200 import binding as hf
    w = gen.Workload("few", batch=1, heads=8, head_dim=128, tokens_per_frame=300, chunk_frames=1, window_frames=2, block=128, topk=0,
                     keep_permille=500, layers=4, seed=317)
    a, b = (hf.Context(hf.make_config(w)) for _ in range(2))
    kv = [[[hf.bits_to_cuda(x) for x in gen.clean_kv(w, layer, c)] for layer in range(w.layers)] for c in range(2)]
    try:
        for ctx in (a, b):
            ctx.hf_kv_append_layers(0, [k for k, _ in kv[0]], [v for _, v in kv[0]])
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            a.hf_kv_append_layers(0, [k for k, _ in kv[1]], [v for _, v in kv[1]])
        g.replay()
        for layer, (k, v) in enumerate(kv[1]):
            b.hf_kv_append(layer, k, v)
        torch.cuda.synchronize()
        _same(a, b, w, [hf.bits_to_cuda(x) for x in gen.qkv(w, 0, 9, 0)])
    finally:
        del g
        a.close(); b.close()


def test_a_captured_commit_of_few_layers_outlives_an_update_of_many():
    """A graph holds the commit of two layers; an update of all fourteen (more items than SMs) then needs more scratch than the context was
    made with.  What the graph writes to must still be there."""
    import torch
    from paper_2604_10103_b200 import binding as hf
    w = gen.Workload("many", batch=1, heads=12, head_dim=64, tokens_per_frame=100, chunk_frames=1, window_frames=2, block=128, topk=0,
                     keep_permille=500, layers=14, seed=337)
    assert w.layers * w.heads > torch.cuda.get_device_properties(0).multi_processor_count
    a, b = (hf.Context(hf.make_config(w)) for _ in range(2))
    kv = [[[hf.bits_to_cuda(x) for x in gen.clean_kv(w, layer, c)] for layer in range(w.layers)] for c in range(3)]
    k, v = ([[x[i] for x in chunk] for chunk in kv] for i in range(2))
    k_ev, v_ev = torch.stack(k[2]), torch.stack(v[2])
    try:
        for ctx in (a, b):
            ctx.hf_kv_append_layers(0, k[0], v[0])
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            a.hf_kv_append_layers(0, k[1][:2], v[1][:2])
        for ctx in (a, b):
            ctx.hf_state_absorb_layers(0, w.layers, k_ev, v_ev, w.chunk_tokens)
        g.replay()
        b.hf_kv_append_layers(0, k[1][:2], v[1][:2])
        torch.cuda.synchronize()
        _same(a, b, w, [hf.bits_to_cuda(x) for x in gen.qkv(w, 0, 9, 0)])
        assert a.hf_get_device_status() == (0, 0)
    finally:
        del g
        a.close(); b.close()


@pytest.mark.parametrize("d,heads", [(64, 1), (128, 3)])
def test_state_copies(d, heads):
    """Either tensor or both, to this device's memory (a kernel) and to an address that is not 16-byte aligned (a copy)."""
    import torch
    from paper_2604_10103_b200 import binding as hf
    w = gen.Workload("state", batch=1, heads=heads, head_dim=d, tokens_per_frame=100, chunk_frames=1, window_frames=1, block=128, topk=0,
                     keep_permille=500, seed=331)
    ctx = hf.Context(hf.make_config(w))
    try:
        ctx.hf_kv_append(0, *[hf.bits_to_cuda(x) for x in gen.clean_kv(w, 0, 0)])
        n_S, n_z = heads * d * d, heads * d
        new = lambda n: torch.full((n + 5,), -7.0, dtype=torch.float32, device="cuda")  # noqa: E731
        S, z, S1, z1, S2, z2 = new(n_S), new(n_z), new(n_S), new(n_z), new(n_S), new(n_z)
        ctx.hf_get_state(0, S, z)
        ctx.hf_get_state(0, S=S1); ctx.hf_get_state(0, z=z1)
        ctx.hf_get_state(0, S2[1:], z2[3:])
        torch.cuda.synchronize()
        assert S[:n_S].abs().sum() > 0 and z[:n_z].min() > 0
        assert torch.equal(S, S1) and torch.equal(z, z1) and (S[n_S:] == -7).all() and (z[n_z:] == -7).all()
        assert torch.equal(S2[1:1 + n_S], S[:n_S]) and torch.equal(z2[3:3 + n_z], z[:n_z])
        assert (S2[:1] == -7).all() and (S2[1 + n_S:] == -7).all() and (z2[:3] == -7).all() and (z2[3 + n_z:] == -7).all()
    finally:
        ctx.close()


def test_state_copies_on_a_stream_and_in_a_graph():
    import torch
    from paper_2604_10103_b200 import binding as hf
    w = gen.Workload("state", batch=1, heads=3, head_dim=64, tokens_per_frame=100, chunk_frames=1, window_frames=1, block=128, topk=0,
                     keep_permille=500, seed=331)
    ctx = hf.Context(hf.make_config(w))
    try:
        ctx.hf_kv_append(0, *[hf.bits_to_cuda(x) for x in gen.clean_kv(w, 0, 0)])
        new = lambda: (torch.zeros(3, 64, 64, device="cuda"), torch.zeros(3, 64, device="cuda"))  # noqa: E731
        (S, z), (S1, z1), (S2, z2) = new(), new(), new()
        ctx.hf_get_state(0, S, z)
        torch.cuda.synchronize()
        n, side = ctx.hf_launch_count(), torch.cuda.Stream()
        with torch.cuda.stream(side):
            ctx.hf_get_state(0, S1, z1)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            ctx.hf_get_state(0, S2, z2)
        g.replay()
        torch.cuda.synchronize()
        assert ctx.hf_launch_count() - n == 2            # one kernel a call on either stream
        assert S.abs().sum() > 0 and torch.equal(S, S1) and torch.equal(S, S2) and torch.equal(z, z1) and torch.equal(z, z2)
    finally:
        del g
        ctx.close()
