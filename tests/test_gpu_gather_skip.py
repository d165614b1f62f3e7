"""The query-gather kernels are left out where no selection could make them pay: around that size the outputs equal
those of a handle that has the path switched off, and where it can pay it is still decided on the device."""
from __future__ import annotations

import pytest
import torch

from paper_2604_08077_b200 import binding, inputs

pytestmark = pytest.mark.gpu


def _run(wl, threshold):
    eng = binding.AdaSAttn(cube=wl.cube, n_q_heads=wl.Hq, n_kv_heads=wl.Hkv, head_dim=wl.D, top_p=wl.top_p)
    eng.set_gather(threshold, 2 << 30)
    eng.partition(wl.B, wl.T, wl.H, wl.W, wl.n_text)
    out, _, _ = eng.forward(wl.q.cuda(), wl.k.cuda(), wl.v.cuda(), wl.n_text)
    torch.cuda.synchronize()
    assert eng.header().status == 0
    return out, eng.launches(), eng.header().gather_entries


@pytest.mark.parametrize("frames,expected", [(8, False), (40, False), (64, True)])
def test_small_calls_leave_the_gather_kernels_out(frames, expected):
    # 28 heads, pairs of tiles of 256 rows: (0 + 4 + .. + 36 + 40) x 28 = 6160 products lie below the bound of 6976, 64 frames above
    wl = inputs.make_prefill("skip", seed=91, B=1, T=frames, H=8, W=8, cube=(4, 4, 4), n_text=20, Hq=28, Hkv=4, D=64,
                             top_p=0.3, offset_std=3.0)
    off, launches_off, _ = _run(wl, 0.0)
    out, launches, _ = _run(wl, 30.0)
    assert (launches > launches_off) == expected
    if not expected:      # (the path rounds partial results to bf16: where it is taken the bits are its own)
        assert torch.equal(out, off)
    _, forced, entries = _run(wl, 1e30)
    assert forced > launches_off and entries > 0
