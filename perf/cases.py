"""The work a user of this library has it do, as a set of measurable cases.

A case is one call through the public entry points of ``paper_2604_08077_b200.binding``: a prefill of a
sequence of video and text tokens (Eqs. 1-3 for every row), one chunk of a prefill that is fed frame by frame,
or a decode step of a batch of sequences whose caches a prefill has built.  The sizes are those of the
repository's configurations, tests and benchmark and of the range between them: from a video of 512 tokens,
where launches count, to 131072 tokens.  The inputs follow the recipe of ``inputs.py`` (normal draws, one shared
offset per cube on the keys, queries that are independent or cohere inside a cube), drawn on the GPU.
"""
from __future__ import annotations

import math
from statistics import NormalDist

import torch

from paper_2604_08077_b200 import binding, inputs

_NORMAL = NormalDist()

_BASE = {
    "kind": "prefill", "B": 1, "T": 64, "H": 16, "W": 16, "ct": 4, "ch": 4, "cw": 4, "n_text": 128, "n_prefix": 0,
    "Hq": 28, "Hkv": 4, "D": 128, "p": 0.9, "top_k": 0, "sigma": 1.5, "cohesive": False, "static_half": False,
    "selection": False, "frame_begin": 0, "frame_count": 0,
}


def _case(name, **kw):
    return {**_BASE, **kw, "name": name}


def listed():
    return [
        # A few seconds of video and a question: nothing but launches and one wave of blocks.
        _case("prefill_tiny", T=8, H=8, W=8, ct=2, n_text=32, Hq=4, Hkv=4, D=64, sigma=2.0),
        # A short clip behind a prompt, two sequences at once, a grid that the cube window does not divide, and the
        # selection handed to the caller (for a report of what was attended).
        _case("prefill_ragged_prefix", B=2, T=30, H=14, W=14, n_prefix=21, n_text=77, Hq=16, Hkv=2, selection=True),
        # The dense reference (p = 1) that a user compares with, at head_dim 64.
        _case("prefill_dense_8k", T=32, n_text=64, Hq=16, Hkv=4, D=64, p=1.0),
        # One layer at the ordinary length: the workload of the benchmark's headline.
        _case("prefill_16k"),
        # The method's default operating point (256-token cubes, p = 0.7) with queries that cohere inside a cube.
        _case("prefill_16k_cohesive", ch=8, cw=8, p=0.7, cohesive=True),
        # Minutes of video at 64 tokens a frame, GQA group of 8, independent queries, default operating point.
        _case("prefill_24k_default", T=384, H=8, W=8, ch=8, cw=8, n_text=201, Hq=16, Hkv=2, p=0.7),
        # A long video whose queries are sharp: each row keeps few of its 1024 cubes.
        _case("prefill_64k_sharp", T=256, n_text=256, p=0.7, sigma=3.0),
        # The same length with ordinary queries.
        _case("prefill_64k", T=256, n_text=256),
        # The longest video of the benchmark, half of it static.
        _case("prefill_128k_static_half", T=512, n_text=0, static_half=True),
        # The next eight seconds of a video that is fed as it arrives.
        _case("chunk_8k_of_64k", kind="chunk", T=256, frame_begin=160, frame_count=32),
        # One new token of a single conversation about a short video: latency.
        _case("decode_16k_b1", kind="decode"),
        # Serving: sixteen conversations about long videos.
        _case("decode_128k_b16", kind="decode", B=16, T=512, n_text=512, static_half=True),
    ]


# What a drawn case may cost: (query row, key) pairs of all heads, just below the largest listed case, and bytes of
# caches for a decode step, those of the largest listed one.
_MAX_PAIRS = 28 * 131072 ** 2 // 4
_MAX_CACHE_BYTES = 16 * 132096 * 4 * 128 * 4


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["prefill"] * 5 + ["chunk"] * 2 + ["decode"] * 3)
    Hq, Hkv, D = rng.choice([(4, 4, 64), (16, 4, 64), (8, 2, 128), (16, 2, 128), (28, 4, 128), (28, 4, 128)])
    H, W = rng.choice([(8, 8), (14, 14), (16, 16), (16, 16), (12, 20), (16, 24)])
    ct, ch, cw = rng.choice([(1, 4, 4), (2, 4, 4), (4, 4, 4), (4, 4, 4), (4, 4, 4), (2, 8, 8), (4, 8, 8), (8, 8, 8)])
    if kind == "chunk":          # a chunk needs a grid that the window divides and starts at a multiple of 256 tokens
        H, W = rng.choice([(8, 8), (16, 16), (16, 16), (16, 24)])
    B = rng.choice([1, 1, 1, 2, 4]) if kind != "decode" else rng.choice([1, 1, 2, 3, 4, 8, 16])
    while True:
        T = max(4, _log_uniform(rng, 512, 131072) // (H * W))
        if kind == "chunk":
            T = max(16, (T + 15) // 16 * 16)
        N = -(-T // ct) * -(-H // ch) * -(-W // cw)
        rows = T * H * W
        if N > 4096:
            continue
        if kind != "decode" and B * Hq * rows * rows // 2 > _MAX_PAIRS:
            continue
        if kind == "decode" and B * (rows + 1024) * Hkv * D * 4 > _MAX_CACHE_BYTES:
            continue
        break
    c = dict(_BASE, kind=kind, B=B, T=T, H=H, W=W, ct=ct, ch=ch, cw=cw, Hq=Hq, Hkv=Hkv, D=D,
             n_text=rng.choice([0, rng.randint(1, 64), rng.randint(65, 512)]),
             p=rng.choice([0.5, 0.7, 0.9, 0.9, 0.95, 1.0]), sigma=rng.choice([0.5, 1.5, 1.5, 3.0]),
             cohesive=kind == "prefill" and rng.random() < 0.3)
    if rng.random() < 0.15:
        c["top_k"] = rng.choice([1, 4, 8, 16, 32])
    if kind == "prefill" and rng.random() < 0.25:
        c["n_prefix"] = rng.randint(1, 96)
    if kind == "chunk":
        c["frame_count"] = max(8, T // rng.choice([2, 4, 8]) // 8 * 8)
        c["frame_begin"] = rng.randrange(0, T - c["frame_count"] + 1, 8)
        if c["frame_begin"] + c["frame_count"] < T:
            c["n_text"] = 0
    c["selection"] = kind == "prefill" and rows <= 16384 and rng.random() < 0.2
    return c


def _tensors(case, seed):
    """The tensors of the sequence(s): seeded draws on the GPU."""
    c = case
    kw = dict(seed=seed, B=c["B"], T=c["T"], H=c["H"], W=c["W"], cube=(c["ct"], c["ch"], c["cw"]), n_text=c["n_text"],
              Hq=c["Hq"], Hkv=c["Hkv"], D=c["D"], top_p=c["p"], offset_std=c["sigma"], device="cuda")
    if c["static_half"]:
        return inputs.make_heterogeneous("case", with_q=c["kind"] != "decode", **kw)
    return inputs.make_prefill("case", with_q=c["kind"] != "decode", n_prefix=c["n_prefix"],
                               q_offset_std=1.0 if c["cohesive"] else 0.0,
                               q_noise_std=0.25 if c["cohesive"] else 1.0, **kw)


def _new_tokens(case, seed):
    """A decode step's new token of every conversation, and how much text each of them holds."""
    c = case
    g = torch.Generator(device="cuda")
    g.manual_seed(seed + 7)
    new = lambda heads: torch.randn(c["B"], 1, heads, c["D"], generator=g, device="cuda").to(torch.bfloat16)  # noqa: E731
    q, k, v = new(c["Hq"]), new(c["Hkv"]), new(c["Hkv"])
    held = torch.randint(c["n_text"] // 2, c["n_text"] + 1, (c["B"],), generator=g, device="cuda")
    return q, k, v, held.to(torch.int32)


def prepare(case, seed):
    """The engine with its caches and workspace, the call's tensors, and an output buffer."""
    c = case
    cube = (c["ct"], c["ch"], c["cw"])
    decode, chunk = c["kind"] == "decode", c["kind"] == "chunk"
    wl = _tensors(c, seed)
    eng = binding.AdaSAttn(cube=cube, n_q_heads=c["Hq"], n_kv_heads=c["Hkv"], head_dim=c["D"], top_p=c["p"],
                           top_k=c["top_k"])
    if decode:
        eng.set_gather(0.0, 0)            # a decoding program has no use for the prefill's gather workspace
    eng.partition(c["B"], c["T"], c["H"], c["W"], c["n_text"] + c["n_prefix"] + (16 if decode else 0))
    state = {"case": c, "eng": eng}
    if decode:
        # the conversations of a batch hold texts of different lengths
        state["q"], state["k"], state["v"], state["text_len"] = _new_tokens(c, seed)
        eng.forward(None, wl.k, wl.v, c["n_text"])
    elif chunk:
        tok, t0, t1 = c["H"] * c["W"], c["frame_begin"], c["frame_begin"] + c["frame_count"]
        last = t1 == c["T"]
        for cache in (eng.k_cube, eng.v_cube, eng.cube_keys):
            cache.zero_()
        if t0:
            eng.forward_chunk(None, wl.k[:, :t0 * tok].contiguous(), wl.v[:, :t0 * tok].contiguous(), 0, t0, -1)
        end = wl.k.shape[1] if last else t1 * tok
        state.update({n: getattr(wl, n)[:, t0 * tok:end].contiguous() for n in "qkv"})
        state["n_text"] = c["n_text"] if last else -1
    else:
        state.update(q=wl.q, k=wl.k, v=wl.v)
    state["out"] = torch.empty_like(state["q"])
    return state


def run(state):
    """One call: the outputs, and the caches that it writes."""
    c, eng = state["case"], state["eng"]
    q, k, v, out = state["q"], state["k"], state["v"], state["out"]
    bitmap = count = None
    if c["kind"] == "decode":
        eng.decode(q, k, v, state["text_len"], out=out)
    elif c["kind"] == "chunk":
        eng.forward_chunk(q, k, v, c["frame_begin"], c["frame_count"], state["n_text"], out=out)
    else:
        _, bitmap, count = eng.forward(q, k, v, c["n_text"], out=out, want_selection=c["selection"],
                                       n_prefix=c["n_prefix"])
    got = {"out": out, "k_cube": eng.k_cube, "v_cube": eng.v_cube, "cube_keys": eng.cube_keys}
    if c["selection"]:
        got.update(bitmap=bitmap, count=count)
    return got


def _kept_share(c):
    """Share of its candidate cubes that a row keeps on average.  The scaled score of a cube is close to normal with
    the standard deviation of the cube offsets, so the probabilities are log-normal: the share of the cubes that
    carries the mass p is Phi(Phi^-1(p) - sigma)."""
    if c["p"] >= 1.0:
        return 1.0
    return _NORMAL.cdf(_NORMAL.inv_cdf(c["p"]) - c["sigma"])


def work(case):
    """Each input read once, each output written once; the scores of Eq. 1 and the attention over the kept cubes
    (4 D operations per query row and attended key)."""
    c = case
    cube = c["ct"] * c["ch"] * c["cw"]
    B, Hq, Hkv, D = c["B"], c["Hq"], c["Hkv"], c["D"]
    N = -(-c["T"] // c["ct"]) * -(-c["H"] // c["ch"]) * -(-c["W"] // c["cw"])
    kv_row, q_row = 2 * Hkv * D * 2, Hq * D * 2

    def kept(n):
        if n <= 0:
            return 0.0
        return float(min(c["top_k"], n)) if c["top_k"] else min(n, max(1.0, n * _kept_share(c)))

    if c["kind"] == "decode":
        share = kept(N) / N
        any_head = 1.0 - (1.0 - share) ** (Hq // Hkv)      # a cube is read once for the heads of a group
        keys = any_head * N * cube + 0.75 * c["n_text"] + 1
        nbytes = B * (keys * kv_row + N * Hkv * D * 4 * (c["p"] < 1.0 or c["top_k"] > 0) + 2 * q_row + 2 * kv_row)
        flops = B * Hq * (2 * D * N + 4 * D * (kept(N) * cube + 0.75 * c["n_text"] + 1))
        return {"bytes": nbytes, "flops": flops}
    tok = c["H"] * c["W"]
    n0, n1 = 0, c["T"] * tok
    n_text, n_prefix = c["n_text"], c["n_prefix"]
    if c["kind"] == "chunk":
        n0, n1 = c["frame_begin"] * tok, (c["frame_begin"] + c["frame_count"]) * tok
    rows = n1 - n0
    cand = (n0 + n1) / 2 / cube                            # candidate cubes of a video row on average
    pairs = rows * (kept(cand) * cube + cube / 2 + n_prefix) + n_prefix ** 2 / 2
    pairs += n_text * (kept(n1 / cube) * cube + n_prefix + n_text / 2)
    scores = rows * cand + n_text * n1 / cube
    seen = n0 if c["kind"] == "chunk" else 0               # keys of earlier calls, read from the caches
    total = rows + n_text + n_prefix
    nbytes = B * (total * (2 * q_row + 2 * kv_row) + seen * kv_row + (n1 // cube) * Hkv * D * 4)
    if c["selection"]:
        nbytes += B * Hq * total * (4 * -(-N // 32) + 4)
    return {"bytes": nbytes, "flops": B * Hq * (2.0 * D * scores + 4.0 * D * pairs)}


def tolerance(case):
    """bf16 outputs with fp32 sums and bf16 attention weights.  Two independent correct paths (tcgen05 with 64-bit fixed-point
    selection, mma.sync with fp64 selection) differ by a relative error of 3e-3 over all listed and drawn sizes, and
    in one place by up to 0.12 of the root mean square (a small element of an early row, whose few values are far
    above the mean square of the whole); the limits are about four times that.  The caches are copies and means
    rounded once.  The selection is exact up to ties (rows whose boundary lies within 1e-6 of the mass); no bit
    differed between the two paths."""
    return {"rel": 1.2e-2, "max": 0.4, "differ": 1e-5}


# What `exact` takes on in about ten seconds: (query row, key) pairs of all heads.
_MAX_EXACT_PAIRS = 28 * 70000 ** 2


def _cube_order(case):
    """For every raster video token its cube, and the tokens in cube order."""
    c = case
    t, y, x = torch.meshgrid(torch.arange(c["T"]), torch.arange(c["H"]), torch.arange(c["W"]), indexing="ij")
    nH, nW = -(-c["H"] // c["ch"]), -(-c["W"] // c["cw"])
    cube = ((t // c["ct"] * nH + y // c["ch"]) * nW + x // c["cw"]).reshape(-1)
    rank = (((t % c["ct"]) * c["ch"] + y % c["ch"]) * c["cw"] + x % c["cw"]).reshape(-1)
    order = torch.argsort(cube * (c["ct"] * c["ch"] * c["cw"]) + rank)
    return cube.cuda(), order.cuda()


def _kept_cubes(case, scores, candidates):
    """Eq. 2 for rows of scores: the shortest prefix of the descending order whose mass reaches p (Top-K: the K first)
    of the first `candidates[row]` cubes."""
    c = case
    N = scores.shape[-1]
    cand = torch.arange(N, device=scores.device) < candidates[:, None]
    if c["top_k"] == 0 and c["p"] >= 1.0:
        return cand
    prob = torch.nan_to_num(torch.softmax(scores.masked_fill(~cand, -math.inf), dim=-1), nan=0.0)
    prob = torch.where(cand, prob, -1.0)                       # what is no candidate comes last
    prob, at = torch.sort(prob, dim=-1, descending=True, stable=True)
    if c["top_k"]:
        first = (torch.arange(N, device=scores.device) < c["top_k"]).expand_as(prob)
    else:
        live = prob.clamp(min=0.0)
        first = torch.cumsum(live, dim=-1) - live < float(torch.tensor(c["p"], dtype=torch.float32))
    return torch.zeros_like(cand).scatter_(-1, at, first) & cand


def _attend(q, k, v, keep, column, causal_from):
    """Softmax attention of rows q [R, D] over keys [M, D]: key m is seen if keep[row, column[m]] and m <= causal_from + row."""
    s = q @ k.T / math.sqrt(q.shape[-1])
    seen = keep[:, column]
    if causal_from is not None:
        R, M = s.shape
        seen &= torch.arange(M, device=q.device) <= causal_from + torch.arange(R, device=q.device)[:, None]
    return torch.softmax(s.masked_fill_(~seen, -math.inf), dim=-1) @ v


def exact(case, seed):
    """Eqs. 1-3 in 64 bits with plain torch, in the layout of `run`.  The caches of keys and values are copies."""
    c = case
    Hq, Hkv, D, B = c["Hq"], c["Hkv"], c["D"], c["B"]
    G, vid, n_pre = Hq // Hkv, c["T"] * c["H"] * c["W"], c["n_prefix"]
    decode, chunk = c["kind"] == "decode", c["kind"] == "chunk"
    if not decode and B * Hq * vid ** 2 > _MAX_EXACT_PAIRS:
        return None
    wl = _tensors(c, seed)
    cube, order = _cube_order(c)
    N = int(cube.max()) + 1
    tok = c["H"] * c["W"]
    begin = c["frame_begin"] * tok if chunk else 0             # the call's tokens, in sequence order
    seen_video = (c["frame_begin"] + c["frame_count"]) * tok if chunk else vid
    end = wl.k.shape[1] if seen_video == vid else seen_video
    # rows and keys in the order [prefix][video by cube][text], where everything a token sees comes before it
    seq = torch.cat([torch.arange(n_pre, device="cuda"), order + n_pre, torch.arange(n_pre + vid, wl.k.shape[1], device="cuda")])
    column = torch.cat([torch.full((n_pre,), N, device="cuda"), cube[order], torch.full((wl.k.shape[1] - n_pre - vid,), N, device="cuda")])
    seq, column = seq[:end], column[:end]
    candidates = torch.where(column < N, column, N)            # preceding cubes; all cubes for the text,
    candidates[:n_pre] = 0                                     # none for the prefix
    held = torch.zeros(N, dtype=torch.float64, device="cuda").index_add_(0, cube, torch.ones(vid, dtype=torch.float64, device="cuda"))
    means = torch.zeros(B, Hkv, N, D, dtype=torch.float64, device="cuda")
    if decode:
        q_new, k_new, v_new, text_len = _new_tokens(c, seed)
    out = torch.zeros(B, 1 if decode else end - begin, Hq, D, dtype=torch.float64, device="cuda")
    rows_at_once = max(64, (1 << 26) // end)
    for b in range(B):
        for kv in range(Hkv):
            k, v = wl.k[b, seq, kv].double(), wl.v[b, seq, kv].double()
            n_vid = min(seen_video, vid)
            mean = means[b, kv].index_add_(0, column[n_pre:n_pre + n_vid], k[n_pre:n_pre + n_vid])
            mean /= held[:, None]
            for h in range(kv * G, kv * G + G):
                if decode:
                    n = n_pre + vid + int(text_len[b])
                    q = q_new[b, :, h].double()
                    keep = _kept_cubes(c, q @ mean.T / math.sqrt(D), torch.tensor([N], device="cuda"))
                    keep = torch.cat([keep, torch.ones_like(keep[:, :1])], dim=1)
                    ks, vs = torch.cat([k[:n], k_new[b, :, kv].double()]), torch.cat([v[:n], v_new[b, :, kv].double()])
                    out[b, :, h] = _attend(q, ks, vs, keep, torch.cat([column[:n], column.new_tensor([N])]), None)
                    continue
                for r0 in range(begin, end, rows_at_once):
                    r1 = min(r0 + rows_at_once, end)
                    q = wl.q[b, seq[r0:r1], h].double()
                    keep = _kept_cubes(c, q @ mean.T / math.sqrt(D), candidates[r0:r1])
                    keep = torch.cat([keep, torch.ones_like(keep[:, :1])], dim=1)          # text and prefix
                    keep.scatter_(1, column[r0:r1, None], True)                            # the own cube
                    out[b, seq[r0:r1] - begin, h] = _attend(q, k[:r1], v[:r1], keep, column[:r1], r0)
    return {"out": out, "k_cube": None, "v_cube": None, "cube_keys": means}
