"""Selection from the tensor-core scores: bit by bit the selection of the fp64 kernel.

Rows whose boundary is nearer than fp32 can tell are handed to the fp64 kernel, all others are decided from fp32
scores, so no bit may differ.  The candidate counts are those at which the kernel changes its shape (rows per pass,
scores per row, buckets) and their neighbours."""
from __future__ import annotations

import math

import pytest
import torch

from paper_2604_08077_b200 import binding, inputs

pytestmark = pytest.mark.gpu


def _selection(wl, kernel, k=None, softmax_scale=0.0):
    eng = binding.AdaSAttn(cube=wl.cube, n_q_heads=wl.Hq, n_kv_heads=wl.Hkv, head_dim=wl.D, top_p=wl.top_p, top_k=wl.top_k,
                           softmax_scale=softmax_scale)
    binding.adaspark_attn_set_prefill_kernel(eng.handle, kernel)
    eng.set_gather(0.0, 0)
    eng.partition(wl.B, wl.T, wl.H, wl.W, wl.n_text + wl.n_prefix)
    k = wl.k if k is None else k
    _, bitmap, count = eng.forward(wl.q.cuda(), k.cuda(), wl.v.cuda(), wl.n_text, want_selection=True, n_prefix=wl.n_prefix)
    torch.cuda.synchronize()
    hdr = eng.header()
    assert hdr.status == 0
    return bitmap, count, hdr


def _equal(wl, k=None, softmax_scale=0.0):
    got, want = _selection(wl, 1, k, softmax_scale), _selection(wl, 0, k, softmax_scale)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    return got[2]


@pytest.mark.parametrize("n_cubes", [1, 2, 31, 33, 64, 65, 255, 257, 511, 513, 1023, 1025, 2047, 2049, 4096])
@pytest.mark.parametrize("rule", ["p", "k"])
def test_candidate_counts_around_every_shape(n_cubes, rule):
    # text rows have all the cubes as candidates, the video rows every smaller count
    wl = inputs.make_prefill("counts", seed=900 + n_cubes, B=1, T=n_cubes, H=4, W=4, cube=(1, 4, 4), n_text=129, Hq=2,
                             Hkv=1, D=64 if n_cubes % 2 else 128, top_p=0.9, offset_std=1.5)
    if rule == "k":
        wl.top_k = min(24, max(1, n_cubes // 3))
    _equal(wl)


@pytest.mark.parametrize("top_p", [1e-6, 0.3, 0.999])
@pytest.mark.parametrize("offset_std", [0.0, 0.05, 4.0])
def test_flat_and_sharp_scores(top_p, offset_std):
    wl = inputs.make_prefill("flat", seed=77, B=2, T=24, H=8, W=12, cube=(2, 4, 4), n_text=40, n_prefix=5, Hq=6, Hkv=2,
                             D=64, top_p=top_p, offset_std=offset_std)
    _equal(wl)


@pytest.mark.parametrize("rule", ["p", "k"])
@pytest.mark.parametrize("copies", [2, 8, 40])
def test_equal_scores(copies, rule):
    """Groups of identical cubes: the boundary falls among equal scores, which the cube index orders.  Only with more of
    them than the list holds do the rows need the fp64 kernel."""
    wl = inputs.make_prefill("ties", seed=78, B=1, T=80, H=8, W=8, cube=(2, 4, 4), n_text=33, Hq=4, Hkv=2, D=128,
                             top_p=0.8, offset_std=1.0)
    if rule == "k":
        wl.top_k = 13
    k = wl.k.clone()
    frames = k[:, :wl.S_v].view(1, 40, 2, 64, 2, 128)
    frames.copy_(frames[:, ::copies].repeat_interleave(copies, 1)[:, :40])
    rows = _equal(wl, k).fallback_rows
    assert rows > 0 if copies > 32 else rows < 0.002 * wl.S * wl.Hq


@pytest.mark.parametrize("copies", [2, 8])
def test_equal_scores_of_different_cubes(copies):
    """Cubes whose mean keys differ in an element that the queries leave out: their scores are equal too, their keys are not,
    and the fp64 kernel decides."""
    wl = inputs.make_prefill("ties", seed=81, B=1, T=80, H=8, W=8, cube=(2, 4, 4), n_text=33, Hq=4, Hkv=2, D=128,
                             top_p=0.8, offset_std=1.0)
    k = wl.k.clone()
    frames = k[:, :wl.S_v].view(1, 40, 2, 64, 2, 128)
    frames.copy_(frames[:, ::copies].repeat_interleave(copies, 1)[:, :40])
    frames[..., 5] = torch.arange(40).view(1, 40, 1, 1, 1).to(torch.bfloat16) / 16
    wl.q[..., 5] = 0.0
    assert _equal(wl, k).fallback_rows > 0.1 * wl.S * wl.Hq


@pytest.mark.parametrize("scale_k", [2.0 ** -70, 2.0 ** -20, 2.0 ** 40])
def test_sizes_whose_squares_leave_fp32(scale_k):
    """Mean keys far from 1 with a logit scale that makes up for it: same sets, and no row needs the fp64 kernel for it."""
    wl = inputs.make_prefill("sizes", seed=79, B=1, T=16, H=8, W=8, cube=(4, 4, 4), n_text=21, Hq=4, Hkv=2, D=128, top_p=0.9,
                             offset_std=1.5)
    k = (wl.k.float() * scale_k).to(torch.bfloat16)
    hdr = _equal(wl, k, softmax_scale=128 ** -0.5 / scale_k)
    assert hdr.fallback_rows < 0.01 * wl.S * wl.Hq


@pytest.mark.parametrize("shared", [(9.0, 3.0), (20.0, 0.0)])
def test_a_bias_that_all_keys_share(shared):
    """A vector added to all keys of a head moves a row's scores by a common offset (up to 300 here): same sets, and no more
    rows than without it are too near to call."""
    wl = inputs.make_prefill("bias", seed=82, B=1, T=64, H=8, W=8, cube=(1, 4, 4), n_text=31, Hq=4, Hkv=2, D=128, top_p=0.99,
                             offset_std=1.5)
    plain = _equal(wl).fallback_rows
    sign = torch.randint(0, 2, (128,), generator=torch.Generator().manual_seed(1)) * 2.0 - 1.0
    k = (wl.k.float() + shared[0] * sign).to(torch.bfloat16)
    wl.q = (wl.q.float() + shared[1] * sign).to(torch.bfloat16)
    assert _equal(wl, k).fallback_rows <= 2 * plain + 0.001 * wl.S * wl.Hq


@pytest.mark.parametrize("first", [0.0, 8.0])
@pytest.mark.parametrize("outlier", [0.0, 30.0])
@pytest.mark.parametrize("level", [False, True])
def test_first_cube_and_one_other_far_from_the_rest(first, outlier, level):
    """Scores are taken relative to cube 0, in the fixed point of the head's largest element: a first cube and one in the
    middle that are far larger than all others cost resolution, not correctness.  With queries whose elements are all of one
    size (level) a row's shift is the largest there is, 12."""
    wl = inputs.make_prefill("far", seed=83, B=1, T=40, H=8, W=8, cube=(1, 4, 4), n_text=31, Hq=4, Hkv=2, D=128, top_p=0.9,
                             offset_std=1.0)
    if level:
        wl.q = (torch.sign(wl.q.float()) * 1.984375).to(torch.bfloat16)
    k = wl.k.float()
    frames = k[:, :wl.S_v].view(1, 40, 2, 4, 2, 4, 2, 128)
    frames[:, 0, 0, :, 0] += first
    frames[:, 17, 1, :, 0] -= outlier
    _equal(wl, k.to(torch.bfloat16))


@pytest.mark.parametrize("top_p", [0.5, 0.99, 0.999, 0.9999, 0.99999, 0.9999999])
@pytest.mark.parametrize("n_cubes,offset_std", [(250, 1.5), (1000, 1.5), (1000, 0.3), (700, 3.0)])
def test_p_near_one(top_p, n_cubes, offset_std):
    """What is left out is 1 - p: the nearer p to 1, the smaller the sums that decide and their errors, so no more rows than
    at other p are too near to call (mass within eps of the target, eps = 5e-6 (1 - p) Z here, at boundary cubes that hold
    about 1 % of the rest)."""
    wl = inputs.make_prefill("rest", seed=84, B=1, T=n_cubes, H=4, W=4, cube=(1, 4, 4), n_text=200, Hq=2, Hkv=1, D=128, top_p=top_p,
                             offset_std=offset_std)
    assert _equal(wl).fallback_rows < 0.005 * wl.S * wl.Hq


@pytest.mark.parametrize("top_p", [0.3, 0.9])
def test_many_masses_that_are_nearly_equal(top_p):
    """4000 masses within a few per cent of each other, whose sums round to the same side again and again."""
    wl = inputs.make_prefill("level", seed=85, B=1, T=4000, H=4, W=4, cube=(1, 4, 4), n_text=300, Hq=1, Hkv=1, D=64, top_p=top_p,
                             offset_std=0.01)
    _equal(wl, wl.k * 0.125)


@pytest.mark.parametrize("n_cubes", [7, 9, 16, 57, 63, 119, 127, 249, 505, 1017])
@pytest.mark.parametrize("top_p", [0.2, 0.7, 0.99999])
def test_last_columns_of_a_row(n_cubes, top_p):
    """Candidate counts one off the 8 columns that a lane takes at a time, at the end of the kernel shapes for up to 1024, with a text prefix
    and a text that end inside the rows of a pass (rows without candidates beside rows with all of them) and cubes at the
    faces that hold no more than a few rows.  No more rows than elsewhere are left to the fp64 kernel, also where two lanes
    sum all buckets of a row."""
    wl = inputs.make_prefill("chunks", seed=86, B=1, T=n_cubes, H=4, W=3, cube=(1, 4, 4), n_text=139, n_prefix=13, Hq=3, Hkv=1,
                             D=128 if n_cubes % 2 else 64, top_p=top_p, offset_std=1.5)
    assert _equal(wl).fallback_rows < 0.005 * wl.S * wl.Hq + 2


@pytest.mark.parametrize("n_cubes", [2041, 4089])
@pytest.mark.parametrize("top_p", [0.2, 0.7, 0.99999])
def test_last_columns_of_the_largest_shapes(n_cubes, top_p):
    """The same for the shapes of one row a pass, where more rows are too near to call: the boundary cube holds less of the mass.  A row is
    handed over if the target lies within eps of the sum up to that cube or before it: eps <= 1e-5 q Z, q = min(p, 1 - p) (at most 88
    additions of 2^-24 and, with scores of up to 24 in log2 units, 2 (1 - q) times 2.4e-6), so a share of 2 eps / its mass, measured on the text
    rows, whose candidates are all cubes (the other rows have fewer, and larger masses).  Besides: 1e-3 of the rows whose last selected score
    is at the edge of a bucket, and those where it is within 4e-6 of the next one."""
    wl = inputs.make_prefill("chunks", seed=88, B=1, T=n_cubes, H=4, W=3, cube=(1, 4, 4), n_text=139, n_prefix=13, Hq=3, Hkv=1,
                             D=128 if n_cubes == 2041 else 64, top_p=top_p, offset_std=1.5)
    keys = wl.k[0, wl.n_prefix:wl.n_prefix + wl.S_v, 0].cuda().double().view(n_cubes, 12, wl.D).mean(1)
    scores = (wl.q[0, -wl.n_text:].cuda().double().flatten(0, 1) @ keys.T * wl.D ** -0.5).sort(descending=True).values
    probs = scores.softmax(1)
    last = ((probs.cumsum(1) < top_p).sum(1, keepdim=True)).clamp(max=n_cubes - 2)
    near = 2e-5 * min(top_p, 1 - top_p) / probs.gather(1, last)
    gap = (scores.gather(1, last) - scores.gather(1, last + 1)) / math.log(2.0)
    share = float(near.clamp(max=1.0).mean() + (gap < 4e-6).double().mean()) + 1e-3
    hdr = _equal(wl)
    print(f"{n_cubes} cubes, p {top_p}: {hdr.fallback_rows} rows of {wl.S * wl.Hq}, {share * wl.S * wl.Hq:.0f} allowed")
    assert share < 0.1 and hdr.fallback_rows < share * wl.S * wl.Hq + 2


@pytest.mark.parametrize("D,heads", [(128, 4), (64, 3)])
def test_rows_left_to_the_fp64_kernel_leave_nothing_in_the_union(D, heads):
    """Cubes whose scores differ by less than the fixed point can tell, ordered against their index: the kernel sets bits for such a
    row, finds that it cannot decide it and takes them back before the words enter the tile's union.  All rows of a head share one
    query, so that a tile selects few cubes; a bit too many would be a block visited more than with the fp64 kernel's selection
    (cubes are single key blocks here)."""
    wl = inputs.make_prefill("union", seed=87, B=1, T=160, H=8, W=8, cube=(4, 4, 4), n_text=33, Hq=heads, Hkv=1, D=D, top_p=0.8, offset_std=1.5)
    k = wl.k.clone()
    frames = k[:, :wl.S_v].view(1, 40, 4, 64, 1, D)
    frames.copy_(frames[:, ::8].repeat_interleave(8, 1))
    frames[..., 5] = torch.arange(40).view(1, 40, 1, 1, 1).to(torch.bfloat16) / 16
    q = (wl.q[:, :1] * 2).expand_as(wl.q).clone()
    q[..., 5] = 2.0 ** -22
    got = []
    for kernel in (1, 2):
        eng = binding.AdaSAttn(cube=wl.cube, n_q_heads=wl.Hq, n_kv_heads=wl.Hkv, head_dim=wl.D, top_p=wl.top_p)
        binding.adaspark_attn_set_prefill_kernel(eng.handle, kernel)
        eng.set_gather(0.0, 0)
        eng.partition(wl.B, wl.T, wl.H, wl.W, wl.n_text)
        out, bitmap, count = eng.forward(q.cuda(), k.cuda(), wl.v.cuda(), wl.n_text, want_selection=True)
        torch.cuda.synchronize()
        got.append((out, bitmap, count, eng.header()))
    assert all(torch.equal(a, b) for a, b in zip(got[0][:3], got[1][:3]))
    mine, want = got[0][3], got[1][3]
    assert mine.status == want.status == 0 and mine.fallback_rows > 0.1 * wl.S * wl.Hq
    assert mine.executed_kv_blocks == want.executed_kv_blocks and mine.max_tile_kv_blocks == want.max_tile_kv_blocks
    tiles = (wl.S + 127) // 128
    assert mine.executed_kv_blocks < 0.7 * wl.Hq * tiles * (tiles + 1)       # of the blocks of dense causal attention
