"""Calls in the order of the stream, on one workspace.  The first kernel of a call is launched to overlap what comes before it, so it
has to wait itself before it reads an input or writes the workspace; most kernels of the library let the next one start early.  Calls right
behind one another, with nothing between them, are therefore what can go wrong (the last tests); behind copies, torch's kernels and memsets,
which let nothing in before they end, the first kernel only has to be ordered at all (the first tests)."""
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
    """Inputs that arrive by copies just before the call and are overwritten just behind it; the header is that of this call."""
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


def _right_behind_one_another(eng, calls, like, captured, rounds=12):
    """Runs `calls` (each writes the output it is given, shaped as in `like`; None: it has none) once in a while and then `rounds`
    times without anything between them: the same outputs, and the same header after the last."""
    for _ in range(2):                                            # the second time on the caches that every further round finds
        want = [None if x is None else torch.empty_like(x) for x in like]
        for call, out in zip(calls, want):
            torch.cuda.synchronize()
            call(out)
        hdr = bytes(eng.header())
    outs = [[None if x is None else torch.zeros_like(x) for x in like] for _ in range(rounds)]

    def all_rounds():
        for row in outs:
            for call, out in zip(calls, row):
                call(out)

    torch.cuda.synchronize()
    if captured:
        graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(graph, stream=stream):
            all_rounds()
        for _ in range(3):
            graph.replay()
    else:
        big = torch.empty(1 << 28, device="cuda")
        torch.cuda.synchronize()
        for _ in range(30):                                       # some 5 ms, for the host to get ahead
            big.fill_(1.0)
        all_rounds()
    torch.cuda.synchronize()
    for row in outs:
        for out, ref in zip(row, want):
            assert out is None or torch.equal(out, ref)
    assert bytes(eng.header()) == hdr and eng.header().status == 0


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("B", [1, 9])
def test_decode_steps_right_behind_one_another(B, captured):
    wl = inputs.small_decode(seed=94, B=B, T=64, H=8, W=8, cube=(1, 4, 4), n_text=40, Hq=8, Hkv=2, D=128)
    eng = pu.make_engine(wl, n_text_max=wl.n_text + 3)
    eng.forward(None, wl.k.cuda(), wl.v.cuda(), wl.n_text)
    calls = []
    for i, s in enumerate((1.0, -0.5, 2.0, -1.5)):
        new = [(x.roll(i, -1) * s).cuda() for x in (wl.q_new, wl.k_new, wl.v_new)]
        tl = torch.tensor([wl.n_text + (i + b) % 3 for b in range(B)], dtype=torch.int32, device="cuda")
        calls.append(lambda out, new=new, tl=tl: eng.decode(*new, tl, out=out))
    _right_behind_one_another(eng, calls, [wl.q_new.cuda()] * len(calls), captured)


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("cube,gather", [((4, 4, 4), 0.0), ((1, 4, 4), 0.0), ((4, 4, 4), pu.FORCE_GATHER), ((2, 8, 8), pu.FORCE_GATHER)])
def test_prefills_right_behind_one_another(cube, gather, captured):
    wl = inputs.make_prefill("behind", seed=95, B=2, T=16, H=8, W=8, cube=cube, n_text=21, Hq=8, Hkv=2, D=128, top_p=0.8, offset_std=1.5)
    eng = pu.make_engine(wl, gather=gather)
    calls = []
    for i, s in enumerate((1.0, -0.5, 3.0)):
        x = [(t.roll(i, -1) * s).cuda() for t in (wl.q, wl.k, wl.v)]
        calls.append(lambda out, x=x: eng.forward(*x, wl.n_text, out=out))
    _right_behind_one_another(eng, calls, [wl.q.cuda()] * 3, captured)
    assert (eng.header().gather_entries > 0) == (gather > 0)


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("gather", [0.0, pu.FORCE_GATHER])
def test_prefills_and_decode_steps_right_behind_one_another(gather, captured):
    """Prefill, decode, a prefill that only builds caches, decode: on other keys each time."""
    wl = inputs.make_prefill("mixed", seed=96, B=2, T=16, H=8, W=8, cube=(4, 4, 4), n_text=21, Hq=8, Hkv=2, D=128, top_p=0.8, offset_std=1.5)
    eng = pu.make_engine(wl, n_text_max=wl.n_text + 1, gather=gather)
    gen = torch.Generator().manual_seed(97)
    new = [[torch.randn(2, 1, h, 128, generator=gen).to(torch.bfloat16).cuda() for h in (8, 2, 2)] for _ in range(2)]
    tl = torch.full((2,), wl.n_text, dtype=torch.int32, device="cuda")
    a, b = ([(t.roll(i, -1) * s).cuda() for t in (wl.q, wl.k, wl.v)] for i, s in ((0, 1.0), (3, -0.5)))
    calls = [lambda out: eng.forward(*a, wl.n_text, out=out), lambda out: eng.decode(*new[0], tl, out=out),
             lambda out: eng.forward(None, *b[1:], wl.n_text), lambda out: eng.decode(*new[1], tl, out=out)]
    _right_behind_one_another(eng, calls, [a[0], new[0][0], None, new[1][0]], captured)


@pytest.mark.parametrize("captured", [False, True])
def test_calls_behind_calls_of_two_streams(captured):
    """A call behind the call before it on its own stream and one of another handle on another stream, which makes its queries."""
    wl = inputs.make_prefill("join", seed=98, B=1, T=16, H=8, W=8, cube=(4, 4, 4), n_text=21, Hq=8, Hkv=2, D=128, top_p=0.8, offset_std=1.5)
    mine, other = (pu.make_engine(wl, n_text_max=wl.n_text + 1) for _ in range(2))
    gen = torch.Generator().manual_seed(99)
    new = [torch.randn(1, 1, h, 128, generator=gen).to(torch.bfloat16).cuda() for h in (8, 2, 2)]
    tl = torch.full((1,), wl.n_text, dtype=torch.int32, device="cuda")
    a, b = ([(t.roll(i, -1) * s).cuda() for t in (wl.q, wl.k, wl.v)] for i, s in ((0, 1.0), (3, -0.5)))
    out = [torch.empty_like(a[0]) for _ in range(3)] + [torch.empty_like(new[0]) for _ in range(3)]
    side = torch.cuda.Stream()

    def chain(main):
        side.wait_stream(main)
        mine.forward(*a, wl.n_text, out=out[0])
        with torch.cuda.stream(side):
            other.forward(*b, wl.n_text, out=out[1])
        main.wait_stream(side)
        mine.forward(out[1], *b[1:], wl.n_text, out=out[2])
        side.wait_stream(main)
        mine.decode(*new, tl, out=out[3])
        with torch.cuda.stream(side):
            other.decode(*new, tl, out=out[4])
        main.wait_stream(side)
        mine.decode(out[4], *new[1:], tl, out=out[5])

    mine.forward(*a, wl.n_text, out=out[0])
    torch.cuda.synchronize()
    other.forward(*b, wl.n_text, out=out[1])
    torch.cuda.synchronize()
    mine.forward(out[1], *b[1:], wl.n_text, out=out[2])
    torch.cuda.synchronize()
    mine.decode(*new, tl, out=out[3])
    other.decode(*new, tl, out=out[4])
    torch.cuda.synchronize()
    mine.decode(out[4], *new[1:], tl, out=out[5])
    torch.cuda.synchronize()
    want = [x.clone() for x in out]
    main = torch.cuda.Stream()
    torch.cuda.synchronize()
    if captured:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=main):
            chain(main)
    for _ in range(20):
        for x in out:
            x.zero_()
        torch.cuda.synchronize()
        if captured:
            graph.replay()
        else:
            with torch.cuda.stream(main):
                chain(main)
        torch.cuda.synchronize()
        assert all(torch.equal(x, w) for x, w in zip(out, want))
