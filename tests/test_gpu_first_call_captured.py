"""The first calls of a process under stream capture, one context for each device module of the attention kernels: creating the context has loaded what they launch
(a module that is first touched while a stream is being captured would end the capture)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = """
import torch
from paper_2604_10103_b200 import binding as hf, inputs as gen

for d, block, topk, wf in ((64, 128, 3, 2), (64, 16, 9, 2), (128, 128, 16, 3), (128, 128, 2, 2), (128, 64, 40, 8), (128, 16, 5, 2)):
    w = gen.Workload("capture", batch=1, heads=4, head_dim=d, tokens_per_frame=1100, chunk_frames=1, window_frames=wf, block=block, topk=topk, keep_permille=0)
    ctx = hf.Context(hf.make_config(w))
    q, k, v = (torch.randn(1, 4, 1100, d, device="cuda").to(torch.bfloat16) for _ in range(3))
    outs = [torch.empty_like(q) for _ in range(6)]
    def calls(o):
        ctx.hf_hybrid_forward(0, q, k, v, o[0]); ctx.hf_sparse_swa_merged(0, q, k, v, o[1]); ctx.hf_sparse_swa(0, q, k, v, o[2])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls(outs[:3])
    graph.replay()
    calls(outs[3:])
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(outs[:3], outs[3:])) and torch.equal(outs[0], outs[1])
    assert float(outs[2].float().abs().max()) > 0 and ctx.hf_get_device_status() == (0, 0)
    graph.reset()
    ctx.close()
print("captured")
"""


def test_first_calls():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "captured" in r.stdout, r.stdout + r.stderr
