"""Decode step around the sizes at which its selection kernel changes shape: cubes dealt to the CTAs of a cluster in
rounds of 256, heads of a group dealt to them eight at a time; and the three kernels under graph capture, where each
may start before the one ahead of it has ended."""
from __future__ import annotations

import pytest
import torch

from paper_2604_08077_b200 import inputs
from test_gpu_decode import compare_decode, run_decode

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_cubes", [2, 64, 256, 258, 514])
@pytest.mark.parametrize("group", [1, 8, 9])
def test_cubes_and_heads_around_the_cluster(n_cubes, group):
    wl = inputs.small_decode(seed=50 + n_cubes, B=2, T=n_cubes, H=4, W=4, cube=(1, 4, 4), n_text=70, Hq=2 * group, Hkv=2,
                             D=64 if group == 8 else 128, top_p=0.8)
    text_len = [70, 3]
    _, out, bitmap = run_decode(wl, text_len)
    compare_decode(wl, text_len, out, bitmap, label=f"{n_cubes} cubes, {group} heads a group")


def test_repeated_steps_in_a_captured_graph():
    wl = inputs.small_decode(seed=61, B=4)
    text_len = [wl.n_text - b for b in range(wl.B)]
    eng, want, _ = run_decode(wl, text_len)
    q, k, v = wl.q_new.cuda(), wl.k_new.cuda(), wl.v_new.cuda()
    tl = torch.tensor(text_len, dtype=torch.int32, device="cuda")
    outs = [torch.zeros_like(q) for _ in range(3)]
    torch.cuda.synchronize()
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):
        for o in outs:
            eng.decode(q, k, v, tl, out=o)
    for _ in range(20):
        graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(o, want) for o in outs)
    hdr = eng.header()
    assert hdr.status == 0 and hdr.decode_kv_blocks > 0
    # a text_len out of range is reported, whatever the step before left in the header
    eng.decode(q, k, v, torch.tensor([wl.n_text + 1000] + text_len[1:], dtype=torch.int32, device="cuda"))
    torch.cuda.synchronize()
    assert eng.header().status == 1
    eng.decode(q, k, v, tl)
    torch.cuda.synchronize()
    assert eng.header().status == 0
