"""Timed cases of the hybrid-attention path, through the entry points a streaming denoiser calls.

A case is a plain dict; its `kind` names what a program does with the library:

  forward  one `hf_hybrid_forward` call of one layer inside a stream that is already running (window filled as far as
           `committed` chunks fill it, older chunks folded into the state): what each layer of each denoising step costs
  stream   one chunk of a running stream: the previous chunk's clean K/V are committed (`hf_kv_append_layers`, or
           `hf_kv_append` with one layer), then `steps` denoising steps of `layers` forwards each
  train    the step with gradient: selection, both branches forward (softmax branch with its row log-sums), then dq, dk, dv of
           the softmax branch and dq of the history branch
  history  an old stretch of tokens is folded into the state and read: `hf_state_absorb` + `hf_linear_attn`

Shapes are those of `paper_2604_10103_b200.inputs` (tiny, the 832x480 layer, full depth, the sweep grid) and the tests' odd
sizes.  Values: unit normal noise plus a part that varies slowly over the tokens of a frame and comes back in every
chunk, so that neighbouring query blocks prefer related key blocks and attention rows are moderately peaked, as
they are in a video model.
"""
import math

import torch

from paper_2604_10103_b200 import binding as hf
from paper_2604_10103_b200 import inputs as gen

LAYER = dict(batch=1, heads=12, head_dim=128, tokens_per_frame=1560, chunk_frames=3, window_frames=9, block=128,
             keep_permille=250, topk=0, layers=1, steps=1, committed=5, merge="head", rope=False, temporal=0, sink_chunks=0,
             tokens=0)


def _case(name, kind, **kw):
    return dict(LAYER, name=name, kind=kind, **kw)


def listed():
    return [
        # the smallest call: the `tiny` workload (8x8 latent, 1-frame chunks, 16-token blocks, top-2); launches and host time
        _case("tiny", "forward", heads=2, head_dim=64, tokens_per_frame=64, chunk_frames=1, window_frames=3, block=16, topk=2,
              committed=4),
        # one layer of one denoising step at 832x480: the call a stream makes 120 times a chunk
        _case("layer_832x480", "forward"),
        # the same layer with 64-token blocks (sweep grid)
        _case("layer_64_token_blocks", "forward", block=64),
        # head_dim 64 with 1-frame chunks, 16-token blocks and a ragged last block: fine-grained selection on short chunks
        _case("short_chunks_16_token_blocks", "forward", head_dim=64, tokens_per_frame=1300, chunk_frames=1, window_frames=3, block=16),
        # window 21, half of the blocks kept, four streams in a batch: the large end of the sweep grid
        _case("window21_batch4", "forward", batch=4, window_frames=21, keep_permille=500, committed=7),
        # the first chunk of a stream at head_dim 64: nothing cached, rotation inside the history branch
        _case("first_chunk_rotated", "forward", head_dim=64, committed=0, rope=True),
        # one layer past the cap of the relative temporal rotation, with a sink chunk: commit (window re-rotated) + one forward
        _case("temporal_rope_sink", "stream", temporal=21, sink_chunks=1, committed=8),
        # short 1-frame chunks through a few layers: many small calls, where launches count (300 tokens: the tests' odd size)
        _case("small_stream", "stream", heads=8, tokens_per_frame=300, chunk_frames=1, window_frames=4, layers=4, steps=4, committed=6),
        # the whole model at 832x480: 30 layers x 4 denoising steps + the commit of all layers
        _case("full_depth_832x480", "stream", layers=30, steps=4),
        # the step with gradient of one layer at 832x480
        _case("train_832x480", "train"),
        # the step with gradient at head_dim 64, ragged, two streams, dense lists
        _case("train_small_ragged", "train", batch=2, heads=8, head_dim=64, tokens_per_frame=1300, chunk_frames=1, window_frames=2,
              keep_permille=500, committed=3),
        # seven chunks of history (32 760 tokens) folded into the state at once, then read by one chunk of queries
        _case("history_7_chunks", "history", tokens=32760, committed=0),
    ]


def draw(rng):
    log = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    kind = rng.choice(["forward"] * 5 + ["stream"] * 3 + ["train"] * 3 + ["history"])
    c = dict(LAYER, kind=kind)
    c["batch"] = rng.choice([1, 1, 1, 2, 4])
    c["heads"] = rng.choice([2, 5, 8, 12, 12, 16])
    c["head_dim"] = rng.choice([64, 128, 128])
    c["block"] = 128 if kind == "train" else rng.choice([16, 64, 128, 128, 128])
    c["chunk_frames"] = rng.choice([1, 2, 3, 3])
    c["tokens_per_frame"] = log(64, 1560)
    chunks = rng.choice([1, 2, 3, 3, 5, 7])
    n_b = -(-c["tokens_per_frame"] * c["chunk_frames"] // c["block"])
    while (chunks + 1) * n_b > 1000:            # the library's limit on key blocks a row spans is 1024
        if chunks > 1:
            chunks -= 1
        else:
            c["tokens_per_frame"] = (c["tokens_per_frame"] + 1) // 2
            n_b = -(-c["tokens_per_frame"] * c["chunk_frames"] // c["block"])
    c["window_frames"] = chunks * c["chunk_frames"]
    c["committed"] = rng.choice([0, 1, chunks + 1, chunks + 1, chunks + 2])
    c["keep_permille"] = log(100, 1000)
    if kind in ("forward", "stream"):
        c["merge"] = rng.choice(["head"] * 6 + ["identity", "full"])
        c["rope"] = rng.random() < 0.15
        c["sink_chunks"] = int(rng.random() < 0.25)
        if rng.random() < 0.2:
            c["temporal"] = max(c["chunk_frames"], 2 * c["window_frames"])
            c["committed"] += 2 * chunks
    if kind == "stream":
        c["layers"], c["steps"] = rng.choice([1, 2, 4, 14]), rng.choice([1, 2, 4])
    if kind == "history":
        c["tokens"] = log(500, 32760)
    while work(c)["flops"] > 5e12 or work(c)["bytes"] > 8e9:       # no more than the largest listed case costs
        if c["layers"] > 1:
            c["layers"] = (c["layers"] + 1) // 2
        elif c["batch"] > 1:
            c["batch"] = 1
        else:
            c["heads"] = (c["heads"] + 1) // 2
    return c


def _workload(c):
    return gen.Workload(c.get("name", "drawn"), batch=c["batch"], heads=c["heads"], head_dim=c["head_dim"], tokens_per_frame=c["tokens_per_frame"],
                        chunk_frames=c["chunk_frames"], window_frames=c["window_frames"], block=c["block"], topk=c["topk"],
                        keep_permille=c["keep_permille"], layers=c["layers"])


class _Values:
    """Seeded values on the GPU: unit normal noise, plus 0.5 x a slowly varying part per (layer, head) for q and k."""

    def __init__(self, w, seed):
        self.g = torch.Generator(device="cuda").manual_seed(seed)
        self.w = w

    def normal(self, *shape, scale=1.0):
        return (torch.randn(*shape, generator=self.g, device="cuda") * scale).to(torch.bfloat16)

    def slow(self, tokens):
        w = self.w
        pos = torch.arange(tokens, device="cuda") / max(8.0, w.tokens_per_frame / 12)
        left = pos.floor().long()
        a = torch.randn(w.batch, w.heads, int(left[-1]) + 2, w.head_dim, generator=self.g, device="cuda")
        f = (pos - left)[:, None]
        return 0.5 * (a[:, :, left] * (1 - f) + a[:, :, left + 1] * f)

    def tokens(self, n, slow=None):
        w = self.w
        x = torch.randn(w.batch, w.heads, n, w.head_dim, generator=self.g, device="cuda")
        return (x if slow is None else x + slow).to(torch.bfloat16)


def prepare(case, seed):
    w = _workload(case)
    val = _Values(w, seed)
    merge = {"head": hf.HF_MERGE_PER_HEAD, "identity": hf.HF_MERGE_IDENTITY, "full": hf.HF_MERGE_FULL_WIDTH}[case["merge"]]
    ctx = hf.Context(hf.make_config(w, merge=merge, sink_frames=case["sink_chunks"] * w.chunk_frames))
    d, n = w.head_dim, w.chunk_tokens
    for layer in range(w.layers):
        if case["merge"] == "head":
            ctx.hf_set_merge_weights(layer, val.normal(w.heads, d, d, scale=d ** -0.5), val.normal(w.heads, d, scale=0.1))
        elif case["merge"] == "full":
            hd = w.heads * d
            ctx.hf_set_merge_weights(layer, val.normal(hd, hd, scale=hd ** -0.5), val.normal(hd, scale=0.1))
    if case["rope"]:
        th = [torch.rand(n, d // 2, generator=val.g, device="cuda") * (2 * math.pi) for _ in range(2)]
        ctx.hf_set_rope(th[0].cos(), th[0].sin(), th[1].cos(), th[1].sin())
    if case["temporal"]:
        cos, sin, _ = gen.temporal_rope_tables(d, case["temporal"])
        ctx.hf_set_temporal_rope(case["temporal"], 0, cos.shape[1], torch.from_numpy(cos).cuda(), torch.from_numpy(sin).cuda())
    slow = [val.slow(n) for _ in range(w.layers)]
    # clean chunks: enough that the window never holds one twice
    window = w.past_chunks + case["sink_chunks"] + 2
    clean = [([val.tokens(n, s) for s in slow], [val.tokens(n) for _ in slow]) for _ in range(min(window, case["committed"] + 2))]
    for i in range(case["committed"]):
        ks, vs = clean[i % len(clean)]
        ctx.hf_kv_append_layers(0, ks, vs)
    st = {"case": case, "ctx": ctx, "clean": clean, "next": case["committed"]}
    st["q"] = [[val.tokens(n, s) for s in slow] for _ in range(w.steps if case["kind"] != "stream" else case["steps"])]
    st["k"] = [[val.tokens(n, s) for s in slow] for _ in st["q"]]
    st["v"] = [[val.tokens(n) for _ in slow] for _ in st["q"]]
    st["o"] = [torch.empty_like(x) for x in st["q"][0]]
    if case["kind"] == "train":
        st["g"] = val.tokens(n)
        st["lse"] = torch.empty(w.batch, w.heads, n, dtype=torch.float32, device="cuda")
        for name in ("o_hist", "dq", "dk", "dv", "dq_hist"):
            st[name] = torch.empty_like(st["o"][0])
    if case["kind"] == "history":
        st["k_ev"], st["v_ev"] = val.tokens(case["tokens"], val.slow(case["tokens"])), val.tokens(case["tokens"])
        st["S"] = torch.empty(w.batch, w.heads, d, d, dtype=torch.float32, device="cuda")
        st["z"] = torch.empty(w.batch, w.heads, d, dtype=torch.float32, device="cuda")
    return st


def run(st):
    ctx, kind = st["ctx"], st["case"]["kind"]
    q, k, v, o = st["q"], st["k"], st["v"], st["o"]
    if kind == "forward":
        ctx.hf_hybrid_forward(0, q[0][0], k[0][0], v[0][0], o[0])
        return o
    if kind == "stream":
        ks, vs = st["clean"][st["next"] % len(st["clean"])]
        st["next"] += 1
        if len(o) == 1:
            ctx.hf_kv_append(0, ks[0], vs[0])
        else:
            ctx.hf_kv_append_layers(0, ks, vs)
        for step in range(len(q)):
            for layer in range(len(o)):
                ctx.hf_hybrid_forward(layer, q[step][layer], k[step][layer], v[step][layer], o[layer])
        return o
    if kind == "train":
        q, k, v, o, g, lse = q[0][0], k[0][0], v[0][0], o[0], st["g"], st["lse"]
        ctx.hf_block_select(0, q, k)
        ctx.hf_sparse_swa(0, q, k, v, o, lse=lse)
        ctx.hf_linear_attn(0, q, st["o_hist"])
        ctx.hf_sparse_swa_backward_dq(0, q, k, v, o, lse, g, st["dq"])
        ctx.hf_sparse_swa_backward_dkv(0, q, k, v, o, lse, g, st["dk"], st["dv"])
        ctx.hf_linear_attn_backward_dq(0, q, g, st["dq_hist"])
        return [o, lse] + [st[name] for name in ("o_hist", "dq", "dk", "dv", "dq_hist")]
    ctx.hf_state_absorb(0, st["k_ev"], st["v_ev"], st["case"]["tokens"])
    ctx.hf_linear_attn(0, q[0][0], o[0])
    ctx.hf_get_state(0, st["S"], st["z"])
    return [o[0], st["S"], st["z"]]


def work(case):
    w = _workload(case)
    bh, d, tc, n_b = w.batch * w.heads, w.head_dim, w.chunk_tokens, w.blocks_per_chunk
    sink = min(case["committed"], case["sink_chunks"])
    cached = min(case["committed"] - sink, w.past_chunks)
    if case["kind"] == "stream":                # the pass commits a chunk first
        sink = min(case["committed"] + 1, case["sink_chunks"])
        cached = min(case["committed"] + 1 - sink, w.past_chunks)
    held = sink + cached
    t_n = (held + 1) * n_b
    keep = min(t_n, case["topk"] if case["topk"] else max(1, -(-case["keep_permille"] * t_n // 1000)))
    chunk = bh * tc * d * 2                                                 # bytes of one [B, H, T_c, d] bf16 tensor
    state = bh * (d * d + d) * 4
    pairs = bh * tc * (keep / t_n) * (held + 1) * tc                        # (query row, kept key)
    pairs_cur = bh * tc * (keep / t_n) * tc                                 # ... with the key in the current chunk
    full = 2 * (w.heads * d) ** 2 * w.batch * tc if case["merge"] == "full" else 0
    hist = 2 * d * d * bh * tc + full
    scores = 2 * d * bh * n_b * t_n
    fwd_bytes = 4 * chunk + 2 * held * min(chunk, n_b * keep * chunk / (held + 1)) + bh * held * n_b * d * 4 + state
    fwd_flops = 4 * d * pairs + hist + scores
    if case["kind"] == "history":
        return {"bytes": 2 * bh * case["tokens"] * d * 2 + 2 * chunk + 2 * state, "flops": 2 * d * d * bh * case["tokens"] + hist}
    if case["kind"] == "train":                 # g, and dq, dk, dv, dq of the history branch, on top of the forward
        return {"bytes": fwd_bytes + 7 * chunk + bh * tc * 4, "flops": fwd_flops + 6 * d * pairs + 4 * d * pairs_cur + 2 * d * d * bh * tc}
    if case["kind"] == "stream":
        leaves = case["committed"] - sink >= w.past_chunks or w.past_chunks == 0
        commit = 4 * chunk + (2 * chunk + 2 * state if leaves else 0)
        steps, layers = case["steps"], w.layers
        return {"bytes": layers * (steps * fwd_bytes + commit), "flops": layers * (steps * fwd_flops + (2 * d * d * bh * tc if leaves else 0))}
    return {"bytes": fwd_bytes, "flops": fwd_flops}


def tolerance(case):
    # Against the same path in 64 bits (masked softmax, its gradients, the state sums; d = 64 and 128, all block sizes) every bf16
    # output is off by rel 2.3e-3 to 2.6e-3 and max 0.9e-2 to 2.4e-2: bf16 results and one bf16 rounding of P / dS.  Four times that.
    return {"rel": 1e-2, "max": 0.1}
