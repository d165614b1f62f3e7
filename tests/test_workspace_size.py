"""How large a forward workspace has to be at least: no larger than the library ever asked for.

The scores of the tensor-core selection lie in the place of the query-gather buffers and give way when the caller's
workspace is smaller than the library asks for: it is taken down to the size that held the fp64 kernel's score rows
instead (the sizes in SIZES), with the same results."""
from __future__ import annotations

import pytest
import torch

from paper_2604_08077_b200 import binding, inputs

# (B, T, H, W, cube, n_text, Hq, Hkv, D, top_p, top_k, gather budget): bytes with room for 1184 rows of fp64 scores, none for
# fp32 scores
SIZES = [
    ((1, 64, 16, 16, (4, 4, 4), 128, 28, 4, 128, 0.9, 0, 0), 19992832),
    ((1, 64, 16, 16, (4, 4, 4), 128, 28, 4, 128, 0.9, 0, 24 << 30), 1929398016),
    ((1, 64, 16, 16, (4, 4, 4), 128, 28, 4, 128, 0.9, 0, 100 << 20), 129479168),
    ((1, 256, 16, 16, (4, 4, 4), 256, 28, 4, 128, 0.9, 0, 0), 259025408),
    ((1, 8, 8, 8, (2, 4, 4), 32, 4, 4, 64, 0.9, 0, 0), 776448),
    ((2, 30, 14, 14, (4, 4, 4), 98, 16, 2, 128, 0.9, 0, 0), 6904832),
    ((1, 256, 16, 16, (1, 4, 4), 0, 4, 1, 64, 0.9, 0, 0), 177554432),
    ((16, 512, 16, 16, (4, 4, 4), 512, 28, 4, 128, 0.9, 0, 0), 15618092288),
    ((3, 8, 8, 8, (4, 4, 4), 5, 4, 4, 64, 0.9, 7, 0), 1082112),
]
# cubes of more than 64 tokens, whose partial results and local range are fp32: the bytes that the entries of single key blocks take, so
# that the budget bounds them too; and more heads than the words kept for each fill up to a multiple of 256 bytes
LARGE = [
    ((1, 64, 16, 16, (4, 8, 8), 128, 28, 4, 128, 0.7, 0, 100 << 20), 115393792),
    ((1, 256, 16, 16, (4, 8, 8), 256, 28, 4, 128, 0.7, 0, 100 << 20), 202591232),
    ((1, 512, 16, 16, (4, 8, 8), 0, 28, 4, 128, 0.7, 0, 100 << 20), 423151104),
    ((1, 512, 16, 16, (4, 8, 8), 0, 28, 4, 128, 0.7, 0, 24 << 30), 25366270976),
    ((1, 64, 16, 16, (2, 8, 8), 128, 16, 4, 64, 0.9, 0, 24 << 30), 585576192),
    ((2, 30, 14, 14, (8, 8, 8), 98, 16, 2, 128, 0.7, 0, 1 << 30), 586249472),
    ((1, 16, 8, 8, (16, 8, 8), 5, 4, 4, 64, 0.9, 3, 1 << 20), 930816),
    ((1, 384, 8, 8, (4, 8, 8), 201, 16, 2, 128, 0.7, 0, 24 << 30), 2499828480),
    ((5, 8, 8, 8, (4, 4, 4), 5, 4, 4, 64, 0.9, 0, 0), 1089792),
    ((21, 8, 8, 8, (4, 4, 4), 5, 8, 1, 64, 0.9, 0, 0), 1884160),
]


def _handle(B, T, H, W, cube, n_text, Hq, Hkv, D, top_p, top_k, budget):
    hd = binding.adaspark_attn_create(binding.Config(*cube, Hq, Hkv, D, top_p, 0.0, 0, top_k))
    binding.adaspark_attn_set_gather(hd, 30.0 if budget else 0.0, budget)
    binding.adaspark_attn_partition(hd, B, T, H, W, n_text)
    return hd, binding.adaspark_attn_get_layout(hd).forward_workspace_bytes


@pytest.mark.skipif(torch.cuda.is_available(), reason="looks at the order of the host's checks, with pointers that are none")
@pytest.mark.parametrize("sizes,nbytes", SIZES + LARGE)
def test_a_workspace_without_room_for_the_scores_is_taken(sizes, nbytes):
    hd, _ = _handle(*sizes)
    fake = 0x1000
    with pytest.raises(binding.AdasparkError) as e:
        binding.adaspark_attn_forward(hd, fake, fake, fake, 0, fake, fake, fake, fake, None, None, fake, nbytes)
    assert e.value.status == binding.ERR_CUDA             # no device: the size was accepted
    with pytest.raises(binding.AdasparkError) as e:
        binding.adaspark_attn_forward(hd, fake, fake, fake, 0, fake, fake, fake, fake, None, None, fake, nbytes // 2)
    assert e.value.status == binding.ERR_WORKSPACE_TOO_SMALL
    binding.adaspark_attn_destroy(hd)


def test_what_a_handle_asks_for():
    sizes = [64, 16, 16, (4, 4, 4), 128, 28, 4, 128]
    hd, with_gather = _handle(1, *sizes, 0.9, 0, 24 << 30)
    binding.adaspark_attn_destroy(hd)
    assert with_gather <= SIZES[1][1]                     # the scores lie inside the gather buffers
    hd, dense = _handle(1, *sizes, 1.0, 0, 0)
    binding.adaspark_attn_destroy(hd)
    assert dense <= SIZES[0][1]                           # p = 1 scores nothing
    hd, top_k = _handle(1, *sizes, 1.0, 8, 0)
    binding.adaspark_attn_destroy(hd)
    assert top_k > dense                                  # Top-K does, whatever top_p says


@pytest.mark.gpu
@pytest.mark.parametrize("kw", [dict(T=16, H=8, W=8, cube=(1, 4, 4), n_text=129, Hq=6, Hkv=2, D=128, top_p=0.9),
                                dict(T=80, H=4, W=4, cube=(1, 4, 4), n_text=70, Hq=4, Hkv=4, D=64, top_p=0.7, B=2),
                                dict(T=30, H=14, W=14, cube=(4, 4, 4), n_text=77, Hq=4, Hkv=2, D=128, top_p=0.9, n_prefix=21)])
@pytest.mark.parametrize("top_k", [0, 9])
def test_scores_of_few_tiles_at_a_time_give_the_same(kw, top_k):
    wl = inputs.make_prefill("few", **{"seed": 301, "offset_std": 1.5, "B": 1, **kw})
    wl.top_k = top_k
    got = []
    for short in (False, True):
        eng = binding.AdaSAttn(cube=wl.cube, n_q_heads=wl.Hq, n_kv_heads=wl.Hkv, head_dim=wl.D, top_p=wl.top_p, top_k=top_k)
        eng.set_gather(0.0, 0)
        eng.partition(wl.B, wl.T, wl.H, wl.W, wl.n_text + wl.n_prefix)
        if short:                                          # a guard behind the end that the call is told
            n_ld, tiles = (wl.N + 63) // 64 * 64, wl.B * wl.Hq * (eng.layout.s_cap // 128)
            assert tiles > 8
            eng.ws_bytes -= (tiles - 8) * 128 * (n_ld * 4 + 32)
            eng.workspace[eng.ws_bytes:] = 77
        out, bitmap, count = eng.forward(wl.q.cuda(), wl.k.cuda(), wl.v.cuda(), wl.n_text, want_selection=True, n_prefix=wl.n_prefix)
        torch.cuda.synchronize()
        assert eng.header().status == 0
        got.append((out, bitmap, count, eng.launches()))
        if short:
            assert bool((eng.workspace[eng.ws_bytes:] == 77).all())
    assert all(torch.equal(a, b) for a, b in zip(got[0][:3], got[1][:3]))
    assert got[1][3] > got[0][3]                           # in several launches


@pytest.mark.gpu
def test_nothing_is_written_behind_the_size_the_library_asks_for():
    """A workspace at the start of a larger buffer, whose whole size the call is told: what lies behind forward_workspace_bytes stays as it
    was, also where the scores of one more launch would fit there (4096 cubes, 513 query tiles; the size asked for holds those of 296)."""
    wl = inputs.make_prefill("behind", seed=302, B=1, T=4096, H=4, W=4, cube=(1, 4, 4), n_text=40, Hq=1, Hkv=1, D=64, top_p=0.9,
                             offset_std=1.5)
    eng = binding.AdaSAttn(cube=wl.cube, n_q_heads=1, n_kv_heads=1, head_dim=64, top_p=wl.top_p)
    eng.set_gather(0.0, 0)
    eng.partition(wl.B, wl.T, wl.H, wl.W, wl.n_text)
    asked = eng.layout.forward_workspace_bytes
    got = []
    for more in (0, 600 << 20):
        eng.ws_bytes = asked + more
        eng.workspace = torch.full((eng.ws_bytes + (1 << 20),), 77, dtype=torch.uint8, device="cuda")
        out, bitmap, _ = eng.forward(wl.q.cuda(), wl.k.cuda(), wl.v.cuda(), wl.n_text, want_selection=True)
        torch.cuda.synchronize()
        assert eng.header().status == 0
        touched = int((eng.workspace[asked:] != 77).sum())
        assert touched == 0
        got.append((out, bitmap))
    assert all(torch.equal(a, b) for a, b in zip(*got))
