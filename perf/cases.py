"""Timed work of the HeadCast attention path: what a program that serves attention layers with this library has it do.

A layer's life is: warm-up blocks with dense attention, one classification, one split of the cache, then for every
generated block one append and a few denoise steps of head-specific attention.  Each kind of case below is one of
these pieces, called through the public binding (``paper_2607_20125_b200.binding``):

    block      one generated block of the steady state: append + one headcast_attend per denoise step
    refresh    the same in the two-block Sink/Dummy mode, the newest block refreshed before every later denoise step
    dense      warm-up / dense baseline: refresh of the newest block + headcast_full_attend, per denoise step
    classify   the one-time classification (scores and labels come back to the host)
    host       one generated block whose tensors live in pinned host memory, until the outputs are there
    noalloc    one call of the allocation-free dense entry point
    start      a layer's whole start: create, two warm-up blocks, classification, split, the first sparse block, destroy

Inputs are seeded bf16 N(0, 1) draws with one planted pattern per head (first-frame keys scaled up, queries and keys of
a block sharing a direction, a positional code, nothing), the distributions of ``paper_2607_20125_b200.synth`` drawn
on the GPU.
"""
from __future__ import annotations

import math

import torch

from paper_2607_20125_b200 import binding, synth
from paper_2607_20125_b200.binding import DUMMY, GLOBAL, SINK, SPATIAL, HeadCast

RADIUS = 2  # of the Spatial proxy (the library's default)
HD = dict(heads=12, d=128, blocks=7, frames=3, cell=10)  # the layer of the 480P / 720P / 1080P configurations


def listed():
    return [
        # the smallest configuration of the repository: 192 queries, four heads of 64, launches and latency count
        dict(name="block-tiny", kind="block", gh=8, gw=8, heads=4, d=64, blocks=5, filled=5, frames=3, cell=10, mix="1/1/1/1", steps=4),
        # a low-resolution preview: ragged tiles, ragged cells, six heads
        dict(name="block-small", kind="block", gh=13, gw=22, heads=6, d=128, blocks=4, filled=4, frames=3, cell=6, mix="1/1/2/2", steps=4),
        # steady state at the 480P, 720P and 1080P grids, 7-block window, four denoise steps per block
        dict(name="block-480p", kind="block", gh=30, gw=52, filled=7, mix="2/3/4/3", steps=4, **HD),
        dict(name="block-720p", kind="block", gh=45, gw=80, filled=7, mix="0/3/6/3", steps=4, **HD),
        dict(name="block-1080p", kind="block", gh=68, gw=120, filled=7, mix="2/3/4/3", steps=4, **HD),
        # anchor + current block for Sink and Dummy heads, the newest block refreshed at every denoise step
        dict(name="refresh-480p", kind="refresh", gh=30, gw=52, filled=7, mix="2/3/4/3", steps=4, **HD),
        # second warm-up block: dense attention over two cached blocks
        dict(name="dense-480p-warmup", kind="dense", gh=30, gw=52, filled=2, mix="2/3/4/3", steps=4, **HD),
        # dense attention over the full window, what a layer without the split pays
        dict(name="dense-720p-full", kind="dense", gh=45, gw=80, filled=7, mix="2/3/4/3", steps=1, **HD),
        # classification right after the two warm-up blocks
        dict(name="classify-480p", kind="classify", gh=30, gw=52, filled=2, mix="2/3/4/3", steps=1, **HD),
        # a caller whose tensors live in host memory
        dict(name="host-480p", kind="host", gh=30, gw=52, filled=7, mix="2/3/4/3", steps=4, **HD),
        # dense attention without allocations, odd lengths, 64-wide heads
        dict(name="noalloc-odd-d64", kind="noalloc", gh=1, gw=1373, heads=16, d=64, blocks=1, filled=4, frames=1, cell=10, mix="0/0/0/16", steps=1),
        # a new video: context, warm-up, classification, split and the first sparse block
        dict(name="start-480p", kind="start", gh=30, gw=52, filled=2, mix="2/3/4/3", steps=4, **HD),
    ]


def draw(rng):
    """One more case of the same ranges; never more arithmetic or memory traffic than the largest listed one."""
    cap = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(["block", "block", "block", "refresh", "dense", "classify", "host", "noalloc", "start"])
        gh = int(round(8 * (68 / 8) ** rng.random()))
        gw = max(8, int(round(gh * rng.uniform(1.0, 1.85))))
        heads, d = rng.choice([4, 6, 8, 12, 12, 12, 16]), rng.choice([64, 128, 128, 128])
        blocks = rng.randint(3, 8)
        filled = blocks if kind in ("block", "refresh", "host") else rng.randint(2, blocks)
        cuts = sorted(rng.randint(0, heads) for _ in range(3))
        mix = "%d/%d/%d/%d" % (cuts[0], cuts[1] - cuts[0], cuts[2] - cuts[1], heads - cuts[2])
        case = dict(kind=kind, gh=gh, gw=gw, heads=heads, d=d, blocks=blocks, filled=filled, frames=3, cell=rng.randint(5, 12), mix=mix,
                    steps=4 if kind not in ("classify", "noalloc") else 1)
        if kind == "noalloc":
            case.update(gh=1, gw=int(round(100 * 60 ** rng.random())), blocks=1, frames=1, filled=rng.randint(1, 7))
        if kind == "start":
            case.update(filled=2)
        if _cost(case) <= cap and case["heads"] * -(-_tokens(case) // 256) <= 2048:
            return case


# ---------------------------------------------------------------------------------------------- inputs


def _tokens(case):
    return case["frames"] * case["gh"] * case["gw"]


def _labels(case):
    counts = [int(v) for v in case["mix"].split("/")]
    lab = [a for a in range(4) for _ in range(counts[a])]
    return tuple(lab[(7 * i) % len(lab)] if math.gcd(7, len(lab)) == 1 else lab[i] for i in range(len(lab)))  # interleaved


class _Inputs:
    """Seeded K, V and Q blocks of one layer, drawn on the GPU."""

    def __init__(self, case, seed):
        self.case, self.labels = case, _labels(case)
        self.gen = torch.Generator(device="cuda").manual_seed(seed)
        h, d, tf = case["heads"], case["d"], case["gh"] * case["gw"]
        lab = torch.tensor(self.labels, device="cuda")
        self.sink, self.dummy, self.spatial = (torch.nonzero(lab == a).flatten() for a in (SINK, DUMMY, SPATIAL))
        self.beta = math.sqrt(20.0 * math.sqrt(d))  # same-block keys of a Dummy head: 20 nats above the others
        ns = len(self.spatial)
        if ns:  # random Fourier features of a Gaussian kernel over grid positions, peak logit 32 nats
            omega = self._randn(ns, d, 2) / 1.25
            phase = torch.rand(ns, 1, d, device="cuda", generator=self.gen) * (2 * math.pi)
            pos = torch.stack([torch.arange(tf, device="cuda") // case["gw"], torch.arange(tf, device="cuda") % case["gw"]], 1).float()
            code = math.sqrt(2.0 / d) * torch.cos(torch.einsum("pc,sdc->spd", pos, omega) + phase)
            self.code = math.sqrt(32.0 * math.sqrt(d)) * code.permute(1, 0, 2).repeat(case["frames"], 1, 1)  # [L, ns, d]

    def _randn(self, *shape):
        return torch.randn(*shape, device="cuda", generator=self.gen)

    def _block(self, direction, first_keys=False):
        c = self.case
        x = self._randn(_tokens(c), c["heads"], c["d"])
        if first_keys and len(self.sink):
            x[: c["gh"] * c["gw"], self.sink] *= 6.0 if c["d"] == 128 else 10.0
        if direction is not None and len(self.dummy):
            x[:, self.dummy] += self.beta * direction
        if direction is not None and len(self.spatial):
            x[:, self.spatial] += self.code
        return x.to(torch.bfloat16)

    def block(self, index, n_q):
        """(K, V, [Q of n_q denoise steps]) of generated block `index`."""
        g = self._randn(1, len(self.dummy), self.case["d"])
        g = g / g.norm(dim=-1, keepdim=True).clamp_min(1e-6)
        return self._block(g, first_keys=index == 0), self._block(None), [self._block(g) for _ in range(n_q)]


def _context(case, **kw):
    return HeadCast(case["heads"], case["d"], case["gh"], case["gw"], case["blocks"], frames_per_block=case["frames"],
                    cell_h=case["cell"], cell_w=case["cell"], sd_mode=int(case["kind"] == "refresh"), **kw)


def prepare(case, seed):
    kind, steps, n = case["kind"], case["steps"], case["filled"]
    x = _Inputs(case, seed)
    s = dict(case=case, labels=x.labels, at=0)
    if kind == "noalloc":
        parts = [x.block(b, 0)[:2] for b in range(n)]
        k, v = (torch.cat([p[i] for p in parts]).contiguous() for i in (0, 1))
        return dict(s, k=k, v=v, q=x.block(n, 1)[2][0], out=torch.empty(_tokens(case), case["heads"], case["d"], dtype=torch.bfloat16, device="cuda"))
    if kind == "start":
        s["blocks"] = [x.block(b, steps) for b in range(n + 1)]
    elif kind == "classify":
        hc = _context(case)
        for b in range(n):
            k, v, q = x.block(b, 1)
            hc.append(k, v)
        return dict(s, hc=hc, q=q[0])
    else:
        hc = _context(case)
        for b in range(n):
            hc.append(*x.block(b, 0)[:2])
        if kind != "dense":
            hc.set_labels(x.labels)
            hc.split_cache()
        s["hc"] = hc
        # what the generator hands over next: two blocks, taken in turn
        s["blocks"] = [x.block(n + i, steps) for i in range(2)]
    s["outs"] = [torch.empty_like(s["blocks"][0][0]) for _ in range(steps)]
    if kind == "host":
        pin = lambda t: t.cpu().pin_memory()  # noqa: E731
        s["blocks"] = [(pin(k), pin(v), [pin(q) for q in qs]) for k, v, qs in s["blocks"]]
        s["outs"] = [torch.empty(o.shape, dtype=o.dtype, pin_memory=True) for o in s["outs"]]
    return s


# ---------------------------------------------------------------------------------------------- one pass


def run(state):
    kind = state["case"]["kind"]
    if kind == "noalloc":
        binding.dense_attend_noalloc(state["q"], state["k"], state["v"], state["out"])
        return state["out"]
    if kind == "classify":
        labels, scores = state["hc"].classify(state["q"])
        return {"labels": labels, "scores": scores}
    if kind == "start":
        return _start(state)
    hc, outs = state["hc"], state["outs"]
    k, v, qs = state["blocks"][state["at"]]
    state["at"] ^= 1
    if kind == "block":
        hc.append(k, v)
        for q, out in zip(qs, outs):
            hc.attend(q, out)
    elif kind == "refresh":
        for i, (q, out) in enumerate(zip(qs, outs)):
            (hc.overwrite_last if i else hc.append)(k, v)
            hc.attend(q, out)
    elif kind == "dense":
        for q, out in zip(qs, outs):
            hc.overwrite_last(k, v)
            hc.full_attend(q, out)
    else:
        hc.append_host(k, v)
        for q, out in zip(qs, outs):
            hc.attend_host(q, out)
        torch.cuda.current_stream().synchronize()  # the outputs are read on the host
    return outs


def _start(state):
    hc, outs = _context(state["case"]), state["outs"]
    result = {}
    for b, (k, v, qs) in enumerate(state["blocks"]):
        hc.append(k, v)
        if b < len(state["blocks"]) - 1:
            for q, out in zip(qs, outs):
                hc.full_attend(q, out)
            if b == len(state["blocks"]) - 2:
                result["warmup"] = [o.clone() for o in outs]
                result["labels"], result["scores"] = hc.classify(qs[0])
                hc.split_cache()
        else:
            for q, out in zip(qs, outs):
                hc.attend(q, out)
    result["outs"] = outs
    hc.destroy()
    return result


# ---------------------------------------------------------------------------------------------- work and tolerance


def _cell_squares(case):
    """Sum over the deployed cells of (tokens per frame)^2."""
    def sizes(n_grid):
        n = max(1, int(math.floor(n_grid / case["cell"] + 0.5)))
        e = [i * n_grid // n for i in range(n + 1)]
        return [b - a for a, b in zip(e, e[1:])]
    return sum((a * b) ** 2 for a in sizes(case["gh"]) for b in sizes(case["gw"]))


def _sparse(case, filled):
    """(flops, bytes of the keys and values read, kept blocks summed over the heads) of one headcast_attend."""
    l, d, lab = _tokens(case), case["d"], _labels(case)
    sd = 2 if case["kind"] == "refresh" else 1
    flops = kept = 0.0
    for a in lab:
        if a in (SINK, DUMMY):
            flops += 4.0 * l * sd * l * d
            kept += sd
        elif a == GLOBAL:
            flops += 4.0 * l * filled * l * d
            kept += filled
        else:
            flops += 4.0 * case["frames"] ** 2 * filled * _cell_squares(case) * d
            kept += filled
    return flops, 4.0 * kept * l * d, kept


def work(case):
    kind, l, h, d, steps, n = case["kind"], _tokens(case), case["heads"], case["d"], case["steps"], case["filled"]
    one = 2.0 * l * h * d  # bytes of one [L][H][d] tensor
    dense = lambda f: (4.0 * h * l * f * l * d, 2 * one + 2 * f * one)  # noqa: E731
    near = 4.0 * h * l * n * case["frames"] * min((2 * RADIUS + 1) ** 2, case["gh"] * case["gw"]) * d
    sf, sb, kept = _sparse(case, n)
    moved = sum(a != SINK or kind == "refresh" for a in _labels(case)) / h  # share of a block that an append keeps
    if kind in ("dense", "noalloc"):
        f, b = dense(n)
        return {"flops": steps * f, "bytes": steps * (b + (4 * one if kind == "dense" else 0))}
    if kind == "classify":
        return {"flops": dense(n)[0] + near, "bytes": one + 2 * n * one}
    if kind == "start":
        f = b = 0.0
        for i in range(1, n + 1):
            df, db = dense(i)
            f, b = f + steps * df, b + 4 * one + steps * db
        sf, sb, kept = _sparse(case, n + 1)
        f += dense(n)[0] + near + steps * sf
        b += one + 2 * n * one + 2 * 4.0 * kept * l * d + 2 * one * (1 + moved) + steps * (2 * one + sb)
        return {"flops": f, "bytes": b}
    appends = steps if kind == "refresh" else 1
    return {"flops": steps * sf, "bytes": appends * 2 * one * (1 + moved) + steps * (2 * one + sb)}


def _cost(case):
    w = work(case)
    return w["flops"] / 1.0e15 + w["bytes"] / (4.0e10 if case["kind"] == "host" else 5.0e12)


def tolerance(case):
    # bf16 probabilities, bf16 outputs, fp32 sums.  Measured against the same attention in 64 bits over the listed
    # sizes: rel 1.6e-3 to 2.4e-3, max 0.005 to 0.017; the scores of a classification against a float64 restatement:
    # rel 4.6e-5, max 2.0e-4.  About four times that; labels are exact (planted heads have wide margins).
    if case["kind"] == "classify":
        return {"rel": 2e-4, "max": 1e-3}
    return {"rel": 1e-2, "max": 0.07}


# ---------------------------------------------------------------------------------------------- the same in 64 bits


def _softmax64(q, k, v, *masks):
    """Attention of q [n, d] over k, v [m, d] in 64 bits; with masks (functions of a row range, or None for all keys) one
    output per mask and the share of the whole row's weight that it keeps."""
    n, scale = q.shape[0], 1.0 / math.sqrt(q.shape[1])
    q, k, v = q.double(), k.double(), v.double()
    outs = [torch.empty_like(q) for _ in masks or (None,)]
    shares = [torch.empty(n, dtype=torch.float64, device=q.device) for _ in outs]
    rows = max(1, (1 << 28) // k.shape[0])
    for a in range(0, n, rows):
        sel = slice(a, min(n, a + rows))
        logits = scale * (q[sel] @ k.T)
        whole = torch.logsumexp(logits, 1)
        for i, mask in enumerate(masks or (None,)):
            x = logits if mask is None else logits.masked_fill(~mask(sel), -math.inf)
            lse = whole if mask is None else torch.logsumexp(x, 1)
            outs[i][sel] = torch.exp(x - lse[:, None]) @ v
            shares[i][sel] = torch.exp(lse - whole)
    return (outs, shares) if masks else outs[0]


def _dense64(q, k, v):
    return torch.stack([_softmax64(q[:, h], k[:, h], v[:, h]) for h in range(q.shape[1])], 1)


def _cells(case, frames):
    """Index of the deployed cell of every token of `frames` frames."""
    def axis(n_grid):
        n = max(1, int(math.floor(n_grid / case["cell"] + 0.5)))
        edges = torch.tensor([i * n_grid // n for i in range(1, n)], dtype=torch.int64, device="cuda")
        return torch.bucketize(torch.arange(n_grid, device="cuda"), edges, right=True)
    return (axis(case["gh"])[:, None] * case["gw"] + axis(case["gw"])[None, :]).flatten().repeat(frames)


def _sparse64(case, labels, blocks, q):
    """headcast_attend over the logical window `blocks` of (K, V), Sink block first, newest block last."""
    both = case["kind"] == "refresh"
    cat = lambda part, h: tuple(torch.cat([b[i][:, h] for b in part]) for i in (0, 1))  # noqa: E731
    out = torch.empty(q.shape, dtype=torch.float64, device="cuda")
    for h, label in enumerate(labels):
        if label == SINK:
            k, v = cat([blocks[0], blocks[-1]] if both else blocks[:1], h)
        elif label == DUMMY:
            k, v = cat(blocks[-2:] if both else blocks[-1:], h)
        else:
            k, v = cat(blocks, h)
        if label != SPATIAL:
            out[:, h] = _softmax64(q[:, h], k, v)
            continue
        mine, theirs = _cells(case, case["frames"]), _cells(case, case["frames"] * len(blocks))
        for c in mine.unique():
            out[mine == c, h] = _softmax64(q[mine == c, h], k[theirs == c], v[theirs == c])
    return out


def _classify64(case, blocks, q):
    """(labels, scores [H, 10]): mean cosines of the proxies' outputs to the whole one, 5th percentile and squared error of
    the Spatial proxy, score, attention masses."""
    l, n = _tokens(case), len(blocks) * _tokens(case)
    pos, where = torch.arange(l, device="cuda") % (case["gh"] * case["gw"]), torch.arange(n, device="cuda")
    where_in = where % (case["gh"] * case["gw"])
    py, px, ky, kx = pos // case["gw"], pos % case["gw"], where_in // case["gw"], where_in % case["gw"]
    first, last = where < l, where >= n - l
    near = lambda s: ((ky - py[s, None]).abs() <= RADIUS) & ((kx - px[s, None]).abs() <= RADIUS)  # noqa: E731
    cosine = lambda a, b: (a * b).sum(1) / (a.norm(dim=1) * b.norm(dim=1)).clamp_min(1e-12)  # noqa: E731
    labels, scores = [], []
    for h in range(case["heads"]):
        k, v = (torch.cat([b[i][:, h] for b in blocks]) for i in (0, 1))
        outs, shares = _softmax64(q[:, h], k, v, None, lambda s: first[None], lambda s: last[None], near,
                                  lambda s: near(s) & ~first & ~last)
        cos = [cosine(o, outs[0]) for o in outs[1:4]]
        rank = 0.05 * (l - 1)
        low = cos[2].sort().values[[int(rank), min(int(rank) + 1, l - 1)]]
        p5 = low[0] + (rank - int(rank)) * (low[1] - low[0])
        mse = (outs[3] - outs[0]).square().mean()
        mass = [s.mean() for s in shares[1:4]]
        rest = (1.0 - shares[1] - shares[2] - shares[4]).mean()
        score = p5 - 5.0 * mse
        cs, cd, cp = (float(c.mean()) for c in cos)
        labels.append(SINK if cs >= 0.95 else DUMMY if cd >= 0.95 else SPATIAL if cp >= 0.95 and float(score) >= 0.755 else GLOBAL)
        scores.append(torch.stack([torch.as_tensor(x, dtype=torch.float64, device="cuda") for x in (cs, cd, cp, p5, mse, score, *mass, rest)]))
    return labels, torch.stack(scores).cpu()


def exact(case, seed):
    kind, steps, n = case["kind"], case["steps"], case["filled"]
    x = _Inputs(case, seed)
    if kind == "noalloc":
        parts = [x.block(b, 0)[:2] for b in range(n)]
        return _dense64(x.block(n, 1)[2][0], *(torch.cat([p[i] for p in parts]) for i in (0, 1)))
    if kind == "classify":
        blocks = [x.block(b, 1) for b in range(n)]
        return {"labels": None, "scores": _classify64(case, blocks, blocks[-1][2][0])[1]}
    if kind == "start":
        blocks = [x.block(b, steps) for b in range(n + 1)]
        whole = [torch.cat([b[i] for b in blocks[:n]]) for i in (0, 1)]
        labels, scores = _classify64(case, blocks[:n], blocks[n - 1][2][0])
        return {"warmup": [_dense64(q, *whole) for q in blocks[n - 1][2]], "labels": None, "scores": scores,
                "outs": [_sparse64(case, labels, blocks, q) for q in blocks[n][2]]}
    blocks = [x.block(b, 0) for b in range(n)]
    new = x.block(n, steps)
    if kind == "dense":  # the newest cached block was refreshed
        whole = [torch.cat([b[i] for b in blocks[:-1] + [new]]) for i in (0, 1)]
        return [_dense64(q, *whole) for q in new[2]]
    window = blocks + [new] if n < case["blocks"] else blocks[:1] + blocks[2:] + [new]
    return [_sparse64(case, x.labels, window, q) for q in new[2]]
