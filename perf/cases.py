"""Timed cases: what a user of this package has it compute, through its public calls.

listed()             the named cases
draw(rng)            one more case of the same ranges (rng: random.Random)
prepare(case, seed)  the inputs and handles a program holds before the call
run(state)           one pass, and its outputs
work(case)           bytes and operations no implementation can do without
exact(case, seed)    the computed numbers of run's outputs in 64 bits

A case holds the call it makes and its sizes:
  call "persistence"  the diagram of one image or volume
       "batched"      the diagrams of `n2` images and `n3` volumes of uneven sizes in one call
       "loss"         diagram, total-persistence loss and its gradient through autograd
       "step"         a BatchedPersistence step (forward, loss, gradient in one graph),
                      with the batch loaded first when `load` is set
       "full"         the whole diagram of a volume, H1 included
  filtration          "V" (pixels are vertices) or "T" (pixels are top cells)
  field               "noise" (independent uniform pixels), "smooth" (white noise blurred by
                      a Gaussian of `sigma` pixels) or "levels" (the same in 256 grey levels)
"""
import math
import random

import numpy as np
import torch

import paper_2606_04801_gb300 as cp

TAU = 0.05  # smallest persistence in the loss of a "step"


def _one(name, call, field, sigma, d, h, w, filtration="V", **kw):
    c = {"call": call, "filtration": filtration, "field": field, "sigma": sigma, "d": d, "h": h, "w": w}
    if name:
        c["name"] = name
    c.update(kw)
    return c


def _many(name, call, sigma2, sigma3, n2, lo2, hi2, n3, lo3, hi3, sizes, filtration="V", load=True):
    c = {"call": call, "filtration": filtration, "field": "smooth", "sigma": sigma2, "sigma3": sigma3, "n2": n2,
         "lo2": lo2, "hi2": hi2, "n3": n3, "lo3": lo3, "hi3": hi3, "sizes": sizes, "load": load}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a small noise image, looked at on its own: the smallest call
        _one("img_64_noise", "persistence", "noise", 0.0, 1, 64, 64),
        # a minibatch of small images of uneven sizes, as a feature extractor takes it
        _many("img_minibatch", "batched", 2.0, 0.0, 64, 32, 160, 0, 0, 0, 3, filtration="T"),
        # one step of an image optimised under a topological loss; odd sides
        _one("img_loss_769x1021", "loss", "smooth", 4.0, 1, 769, 1021),
        # an 8-bit photograph or micrograph: large, with heavy ties
        _one("img_2048_levels", "persistence", "levels", 8.0, 1, 2048, 2048),
        # the same size of use with the pixels as top cells; odd sides
        _one("img_t_1023x1537", "persistence", "smooth", 4.0, 1, 1023, 1537, filtration="T"),
        # noise in a volume, the paper's synthetic input: most survivors per voxel
        _one("vol_128_noise", "persistence", "noise", 0.0, 128, 128, 128),
        # a scan at its own odd size, under a topological loss
        _one("vol_loss_157x189x181", "loss", "smooth", 2.0, 157, 189, 181),
        # a scan with the voxels as top cells
        _one("vol_t_254x256x250", "persistence", "smooth", 3.0, 254, 256, 250, filtration="T"),
        # a large volume's training step, the volume already in the step's input buffer
        _one("vol_512_step", "step", "smooth", 3.0, 512, 512, 512, load=False),
        # a batch of 64 images and 8 volumes of uneven sizes: a training step on new inputs
        _many("batch_72_step", "step", 4.0, 2.0, 64, 128, 1024, 8, 64, 192, 0),
        # the whole diagram of a volume, loops included
        _one("vol_full_128", "full", "smooth", 2.0, 128, 128, 128),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["img", "img", "imgs", "vol", "vol", "vols", "full"])
    filt = rng.choice(["V", "V", "T"])
    call = rng.choice(["persistence", "loss", "step"])
    field = rng.choice(["noise", "smooth", "smooth", "levels"])
    if kind == "img":
        h = _log(rng, 32, 2048)
        w = max(24, min(2300, int(h * rng.uniform(0.6, 1.6))))
        c = _one(None, call, field, 0.0 if field == "noise" else round(rng.uniform(1.5, 8.0), 2), 1, h, w, filt)
    elif kind == "vol":
        d = _log(rng, 24, 128 if field == "noise" else 360)
        h, w = (max(16, min(400, int(d * rng.uniform(0.7, 1.4)))) for _ in range(2))
        c = _one(None, call, field, 0.0 if field == "noise" else round(rng.uniform(1.5, 4.0), 2), d, h, w, filt)
    elif kind == "imgs":
        hi = _log(rng, 48, 700)
        c = _many(None, rng.choice(["batched", "step"]), round(rng.uniform(1.5, 4.0), 2), 0.0, rng.randint(2, 64),
                  max(16, hi // 5), hi, 0, 0, 0, rng.randint(1, 10 ** 6), filt)
    elif kind == "vols":
        hi = _log(rng, 32, 160)
        c = _many(None, rng.choice(["batched", "step"]), 3.0, round(rng.uniform(1.5, 3.0), 2), rng.randint(0, 16), 64,
                  512, rng.randint(1, 8), max(16, hi // 3), hi, rng.randint(1, 10 ** 6), filt)
    else:
        s = _log(rng, 20, 96)
        h, w = (max(16, min(110, int(s * rng.uniform(0.7, 1.3)))) for _ in range(2))
        c = _one(None, "full", "smooth", round(rng.uniform(1.5, 2.2), 2), s, h, w)
    if c["call"] == "step":
        c["load"] = True
    return c


# ---------------------------------------------------------------- inputs
def _shapes(case):
    if "n2" not in case:
        d, h, w = case["d"], case["h"], case["w"]
        return [(h, w) if d == 1 else (d, h, w)]
    rng = np.random.default_rng(case["sizes"])
    s2 = [tuple(int(v) for v in rng.integers(case["lo2"], case["hi2"] + 1, 2)) for _ in range(case["n2"])]
    rng = np.random.default_rng(case["sizes"])
    s3 = [tuple(int(v) for v in rng.integers(case["lo3"], case["hi3"] + 1, 3)) for _ in range(case["n3"])]
    return s2 + s3


def _blur(a, sigma):
    """Separable Gaussian blur, truncated at 4 sigma, edges mirrored."""
    r = int(4.0 * sigma + 0.5)
    taps = np.exp(-0.5 * (np.arange(-r, r + 1) / sigma) ** 2)
    taps /= taps.sum()
    for ax in range(a.dim()):
        n = a.shape[ax]
        at = torch.arange(-r, n + r, device=a.device).remainder(2 * n)
        at = torch.where(at >= n, 2 * n - 1 - at, at)
        p = a.index_select(ax, at)
        a = torch.zeros_like(a)
        for i, t in enumerate(taps):
            a.add_(p.narrow(ax, i, n), alpha=float(t))
    return a


def _fields(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    out = []
    for s in _shapes(case):
        if case["field"] == "noise":
            out.append(torch.rand(s, generator=g, device="cuda"))
            continue
        x = _blur(torch.randn(s, generator=g, device="cuda"), case["sigma3"] if len(s) == 3 and "n2" in case else case["sigma"])
        lo, hi = x.min(), x.max()
        x = (x - lo) / (hi - lo)
        out.append(torch.floor(x * 255.0 + 0.5) if case["field"] == "levels" else x)
    return out


def prepare(case, seed):
    xs = _fields(case, seed)
    # room for every diagram of these sizes: twice the expected pairs (H1: about three times H0 and H2)
    pairs = _pairs(case) * (4 if case["call"] == "full" else 1)
    state = {"case": case, "x": xs, "rows": int(2 * pairs) + 512 * len(xs)}
    if case["call"] == "step":
        bp = cp.BatchedPersistence(_shapes(case), tau=TAU, filtration=case["filtration"])
        bp.load(xs)
        bp.capture()  # a program that steps many times captures its graph once
        state["bp"] = bp
        if not case["load"]:
            state["x"] = None
    return state


def _stacked(state, raw):
    """The pairs in a table of the case's row count (rows past the last pair
    are -1), so that the diagrams of several inputs stack."""
    out = raw.new_full((state["rows"], 8), -1)
    out[: raw.shape[0]] = raw
    return out


def run(state):
    case = state["case"]
    call, filt = case["call"], case["filtration"]
    if call == "step":
        bp = state["bp"]
        if case["load"]:
            bp.load(state["x"])
        loss, grad = bp.step()
        return {"loss": loss, "grad": grad}
    if call == "persistence":
        return _stacked(state, cp.persistence(state["x"][0], filtration=filt).raw)
    if call == "batched":
        return _stacked(state, cp.persistence_batched(state["x"], filtration=filt).raw)
    if call == "full":
        return _stacked(state, cp.persistence_full(state["x"][0]).raw)
    x = state["x"][0].detach().requires_grad_()
    birth, death, raw = cp.diagram(x, filtration=filt)
    loss = ((death - birth)[torch.isfinite(death)] ** 2).sum()
    loss.backward()
    return {"raw": _stacked(state, raw), "loss": loss.detach(), "grad": x.grad}


# ---------------------------------------------------------------- work
def _pairs_per_pixel(ndim, field, sigma):
    if field == "noise":  # minima under face neighbours, maxima under all neighbours
        return 1 / 5 + 1 / 9 if ndim == 2 else 1 / 7 + 1 / 27
    return 0.109 / sigma ** 2 if ndim == 2 else 0.034 / sigma ** 3


def _pairs(case):
    total = 0.0
    for s in _shapes(case):
        sigma = case["sigma3"] if len(s) == 3 and "n2" in case else case["sigma"]
        total += math.prod(s) * _pairs_per_pixel(len(s), case["field"], sigma) + 1
    return total


def work(case):
    """Every pixel read once and every pair (32 bytes) or gradient pixel written
    once; one comparison per edge and per facet of the grid."""
    shapes = _shapes(case)
    n = sum(math.prod(s) for s in shapes)
    nbytes = 4 * n
    if case["call"] != "step":
        nbytes += 32 * _pairs(case)
    if case["call"] in ("loss", "step"):
        nbytes += 4 * n
    ops = sum(2 * len(s) * math.prod(s) for s in shapes)
    return {"bytes": int(nbytes), "flops": int(ops)}


# ---------------------------------------------------------------- 64-bit values
def _half_offsets(ndim, faces):
    offs = []
    for k in range(3 ** ndim // 2 + 1, 3 ** ndim):
        o = [(k // 3 ** a) % 3 - 1 for a in reversed(range(ndim))]
        if not faces or sum(map(abs, o)) == 1:
            offs.append(o)
    return offs


def _slices(shape, off):
    a, b = [], []
    for n, o in zip(shape, off):
        a.append(slice(max(0, -o), n - max(0, o)))
        b.append(slice(max(0, o), n - max(0, -o)))
    return tuple(a), tuple(b)


def _merges(rank, faces, outside):
    """Elder-rule merges of the graph whose nodes enter in the order of their
    ranks (a permutation), over face neighbours or all neighbours; with
    `outside`, one more node, older than all, that touches the border.
    Returns the ranks (of the younger component's first node, of the merging
    node)."""
    shape, n = rank.shape, rank.numel()
    lab = rank.clone()  # each node's smallest neighbour by rank
    offs = _half_offsets(rank.dim(), faces)
    for off in offs:
        a, b = _slices(shape, off)
        lab[a] = torch.minimum(lab[a], rank[b])
        lab[b] = torch.minimum(lab[b], rank[a])
    border = torch.zeros(shape, dtype=torch.bool, device=rank.device)
    for ax in range(rank.dim()):
        border.select(ax, 0).fill_(True)
        border.select(ax, shape[ax] - 1).fill_(True)
    flat = rank.reshape(-1)
    nxt = torch.empty(n + 1, dtype=torch.int64, device=rank.device)  # by rank; n: the outside
    nxt[flat] = lab.reshape(-1)
    nxt[n] = n
    if outside:
        nxt[flat[border.reshape(-1)]] = n
    while True:
        two = nxt[nxt]
        if torch.equal(two, nxt):
            break
        nxt = two
    lab = nxt[rank]
    us, vs, ws = [], [], []
    for off in offs:
        a, b = _slices(shape, off)
        cut = lab[a] != lab[b]
        us.append(torch.minimum(lab[a], lab[b])[cut])
        vs.append(torch.maximum(lab[a], lab[b])[cut])
        ws.append(torch.maximum(rank[a], rank[b])[cut])
    u, v, w = torch.cat(us), torch.cat(vs), torch.cat(ws)
    order = torch.argsort(w, stable=True)
    pair = (u * (n + 1) + v)[order]
    first = torch.argsort(pair, stable=True)
    sp = pair[first]
    keep = torch.ones_like(sp, dtype=torch.bool)
    keep[1:] = sp[1:] != sp[:-1]
    order = order[torch.sort(first[keep]).values]  # the first edge of each pair of basins, in order
    parent = {}
    young, merge = [], []
    for a, b, k in zip(u[order].tolist(), v[order].tolist(), w[order].tolist()):
        while parent.get(a, a) != a:
            parent[a] = a = parent.get(parent[a], parent[a])
        while parent.get(b, b) != b:
            parent[b] = b = parent.get(parent[b], parent[b])
        if a == b:
            continue
        if a == n or (b != n and a < b):
            a, b = b, a
        parent[a] = b  # a: the younger class
        young.append(a)
        merge.append(k)
    return young, merge


def _loss_and_grad(x, filtration, tau):
    """Sum of squared persistence above tau over both dimensions, and its gradient."""
    vals = x.double().reshape(-1)
    n = vals.numel()
    grad = torch.zeros(n, dtype=torch.float64, device=x.device)
    loss = 0.0
    for up in (True, False):
        # ties by linear index; the top dimension is the components of the
        # superlevel sets and the outside, in the reversed order
        pix = torch.argsort(vals, stable=True)
        if not up:
            pix = pix.flip(0)
        rank = torch.empty_like(pix)
        rank[pix] = torch.arange(n, device=x.device)
        young, merge = _merges(rank.view(x.shape), faces=up == (filtration == "V"), outside=not up)
        if not young:
            continue
        first = pix[torch.tensor(young, device=x.device)]
        last = pix[torch.tensor(merge, device=x.device)]
        birth, death = (first, last) if up else (last, first)
        pers = vals[death] - vals[birth]
        pers = torch.where(pers > tau, pers, torch.zeros_like(pers))
        loss += float((pers * pers).sum())
        grad.index_add_(0, death, 2.0 * pers)
        grad.index_add_(0, birth, -2.0 * pers)
    return loss, grad


def exact(case, seed):
    """Loss and gradient; the diagrams are copies of pixels and indices.  None
    for diagrams with H1 and for volumes too large for the plain loop."""
    shapes = _shapes(case)
    cost = sum(math.prod(s) * (200 if case["field"] == "noise" else 4 if len(s) == 3 else 2) for s in shapes)
    if case["call"] not in ("loss", "step") or cost > 120e6:
        return None
    xs = _fields(case, seed)
    if case["call"] == "loss":
        loss, grad = _loss_and_grad(xs[0], case["filtration"], 0.0)
        return {"raw": None, "loss": torch.tensor(loss, dtype=torch.float64), "grad": grad.view(xs[0].shape).cpu()}
    parts = [_loss_and_grad(x, case["filtration"], TAU) for x in xs]
    return {"loss": torch.tensor([sum(p[0] for p in parts)], dtype=torch.float64),
            "grad": torch.cat([p[1] for p in parts]).cpu()}
