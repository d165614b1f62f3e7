"""Calls whose inputs are made by the kernel right before them in the stream, on one workspace.  The first kernel of a call is
launched to overlap what comes before it, so it has to wait itself before it reads an input or writes the workspace."""
from __future__ import annotations

import pytest
import torch

from paper_2604_08077_b200 import inputs

import parity_util as pu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 9])
def test_decode_inputs_made_right_before(B):
    wl = inputs.small_decode(seed=91, B=B, T=64, H=8, W=8, cube=(1, 4, 4), n_text=40, Hq=8, Hkv=2, D=128)
    eng = pu.make_engine(wl, n_text_max=wl.n_text + 1)
    eng.forward(None, wl.k.cuda(), wl.v.cuda(), wl.n_text)
    steps = [(wl.q_new.cuda() * s, wl.k_new.cuda() * s, wl.v_new.cuda() * s) for s in (1.0, -0.5, 2.0)]
    tl = torch.full((B,), wl.n_text, dtype=torch.int32, device="cuda")
    want = []
    for q, k, v in steps:
        want.append(eng.decode(q, k, v, tl)[0].clone())
        torch.cuda.synchronize()
    q, k, v = (torch.empty_like(x) for x in steps[0])
    big, t = torch.empty(1 << 26, device="cuda"), torch.empty_like(tl)
    for _ in range(30):
        for (a, b, c), w in zip(steps, want):
            big.fill_(1.0)                                        # keeps the GPU busy while the host goes on
            q.copy_(a), k.copy_(b), v.copy_(c), t.copy_(tl)
            out, _ = eng.decode(q, k, v, t)
            t.fill_(-5), q.zero_()
            assert torch.equal(out, w)


@pytest.mark.parametrize("C", [(1, 4, 4), (2, 8, 8)])
def test_prefill_inputs_made_right_before(C):
    """The header and counters of the workspace are cleared on the stream, after the call before: outputs, counters and status
    of a call do not depend on what follows at once."""
    wl = inputs.make_prefill("order", seed=92, B=2, T=16, H=8, W=8, cube=C, n_text=21, Hq=8, Hkv=2, D=128, top_p=0.8, offset_std=1.5)
    eng = pu.make_engine(wl)
    steps = [(wl.q.cuda() * s, wl.k.cuda() * s, wl.v.cuda() * s) for s in (1.0, -0.5)]
    want = []
    for q, k, v in steps:
        out = eng.forward(q, k, v, wl.n_text)[0].clone()
        torch.cuda.synchronize()
        want.append((out, eng.header().executed_kv_blocks))
    q, k, v = (torch.empty_like(x) for x in steps[0])
    big = torch.empty(1 << 26, device="cuda")
    for _ in range(20):
        for (a, b, c), w in zip(steps, want):
            big.fill_(1.0)                                        # keeps the GPU busy while the host goes on
            q.copy_(a), k.copy_(b), v.copy_(c)
            out = eng.forward(q, k, v, wl.n_text)[0]
            q.zero_(), k.zero_(), v.zero_()
            assert torch.equal(out, w[0])
            hdr = eng.header()
            assert hdr.status == 0 and hdr.executed_kv_blocks == w[1]


def test_captured_behind_copies_and_memsets():
    """In a graph the node before a call's first kernel may be a copy or a memset instead of a kernel."""
    wl = inputs.make_prefill("graph", seed=93, B=1, T=8, H=8, W=8, cube=(1, 4, 4), n_text=21, Hq=8, Hkv=2, D=128, top_p=0.8, offset_std=1.5)
    eng = pu.make_engine(wl, n_text_max=wl.n_text + 1)
    src = [x.cuda() for x in (wl.q, wl.k, wl.v)]
    q, k, v = (torch.empty_like(x) for x in src)
    new = [torch.randn(1, 1, h, 128, device="cuda").to(torch.bfloat16) for h in (8, 2, 2)]
    tl = torch.full((1,), wl.n_text, dtype=torch.int32, device="cuda")
    want = eng.forward(*src, wl.n_text)[0].clone()
    want_new = eng.decode(*new, tl)[0].clone()
    out, out_new, q_new = torch.empty_like(want), torch.empty_like(want_new), torch.empty_like(new[0])
    torch.cuda.synchronize()
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):
        for a, b in zip((q, k, v), src):
            a.copy_(b)
        eng.forward(q, k, v, wl.n_text, out=out)
        q_new.copy_(new[0])
        eng.decode(q_new, new[1], new[2], tl, out=out_new)
        q.zero_()
        out_new.add_(0.0)
        eng.forward(*src, wl.n_text, out=out)
    for _ in range(10):
        out.zero_(), out_new.zero_()
        graph.replay()
        assert torch.equal(out, want) and torch.equal(out_new, want_new)
