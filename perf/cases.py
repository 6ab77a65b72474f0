"""The work that users of this framework have it do, as timed cases.

Every case is one call (or one pair's calls) through the package's public entry points on
seeded synthetic feature maps: a piecewise-constant scene of Voronoi superpixels drawn from a
mixture, pixel noise and a ReLU, with a template resampled from it (rotation, scale, an
occluder, noise).  Everything here but ``run`` is plain torch; ``exact`` evaluates the method
in 64 bits without the package.

Kinds of case (``"op"``):

``pair``    the whole path for one template and one query, call by call
``assign``  the nearest-neighbour field of a query over a codebook
``fit``     a template's k-means codebook
``score``   the similarity heatmap and its maximum from a query's labels
``batch``   many templates of uneven size and k against several queries
``soft``    one training step: the soft-assignment heatmap and its gradients
"""
import math
import random

import torch

import paper_2306_15010_gb300 as vq

DEV = "cuda"


def listed():
    return [
        # the smallest whole job: a 256 x 256 map, a 32 x 32 template, five filters, FP32; one
        # pair is a chain of short launches
        dict(name="pair_small", op="pair", H=256, W=256, D=64, k=16, th=32, tw=32, iters=10, grid=2, prec="fp32"),
        # the high-resolution query against a kept codebook: a frame's nearest-neighbour field
        dict(name="assign_bf16_2048", op="assign", H=2048, W=2048, D=512, k=128, prec="bf16"),
        # a 720p frame with colour-patch features (27 values, padded to 32)
        dict(name="assign_bf16_colour", op="assign", H=720, W=1280, D=32, k=128, prec="bf16"),
        # the plain FP32 path on deep features
        dict(name="assign_fp32_1024", op="assign", H=1024, W=1024, D=512, k=128, prec="fp32"),
        # the FP8 path of the precision study: twice the depth, exact labels all the same
        dict(name="assign_fp8_d1024", op="assign", H=1024, W=1024, D=1024, k=128, prec="fp8"),
        # a new target: the codebook of a 128 x 128 template of deep features
        dict(name="fit_bf16_128", op="fit", th=128, tw=128, D=512, k=128, iters=10, prec="bf16"),
        # a small target of odd size, shallow features
        dict(name="fit_fp32_small", op="fit", th=45, tw=61, D=64, k=32, iters=10, prec="fp32"),
        # the heatmap of the high-resolution pair: full window and 3 x 3 cells
        dict(name="score_grid_2048", op="score", H=2048, W=2048, k=128, th=128, tw=128, D=512, grid=3),
        # the paper's filter bank (Gaussian and Haar filters at three sub-scales) on a 720p frame
        dict(name="score_paper_720p", op="score", H=720, W=1280, k=128, th=97, tw=82, D=512, grid=0),
        # a library of templates against several frames in one call
        dict(name="batch_3x10", op="batch", nq=3, nt=10, lo=512, hi=1024, tlo=16, thi=192, D=256, iters=10, grid=3, sizes=1),
        # the training workload: eight 512 x 512 maps, forward and backward
        dict(name="soft_train_8x512", op="soft", B=8, H=512, W=512, D=256, k=64, th=64, tw=64, grid=3, tau=0.1),
        # a training step on crops of odd size
        dict(name="soft_train_small", op="soft", B=2, H=121, W=150, D=64, k=32, th=33, tw=40, grid=3, tau=0.3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["pair", "assign", "assign", "assign", "fit", "fit", "score", "score", "batch", "soft"])
    prec = rng.choice(["fp32", "bf16", "bf16", "fp8"])
    if op == "pair":
        H, W = _log(rng, 128, 900), _log(rng, 128, 900)
        th, tw = _log(rng, 16, min(120, H // 2)), _log(rng, 16, min(120, W // 2))
        return dict(op=op, H=H, W=W, D=16 * _log(rng, 1, 32), k=min(_log(rng, 8, 128), th * tw // 4), th=th, tw=tw,
                    iters=10, grid=rng.choice([0, 2, 3]), prec=prec)
    if op == "assign":
        D = 16 * _log(rng, 1, 64)
        k = _log(rng, 8, 128 if prec == "fp8" or D > 512 else 256)
        most = {"fp32": 1 << 20, "fp8": 1 << 20, "bf16": 1 << 21}[prec] * 512 // max(D, 128)
        H = _log(rng, 96, 2048)
        return dict(op=op, H=H, W=max(64, min(_log(rng, 96, 2048), most // H)), D=D, k=k, prec=prec)
    if op == "fit":
        th, tw = _log(rng, 16, 160), _log(rng, 16, 160)
        return dict(op=op, th=th, tw=tw, D=16 * _log(rng, 1, 32), k=min(_log(rng, 8, 128), th * tw // 4),
                    iters=rng.choice([5, 10, 20]), prec=prec)
    if op == "score":
        H, W = _log(rng, 200, 2048), _log(rng, 200, 2048)
        return dict(op=op, H=H, W=W, k=_log(rng, 8, 128), th=_log(rng, 16, 180), tw=_log(rng, 16, 180), D=64,
                    grid=rng.choice([0, 2, 3, 3, 4]))
    if op == "batch":
        return dict(op=op, nq=rng.randint(1, 3), nt=rng.randint(2, 10), lo=300, hi=rng.randint(500, 1024), tlo=16,
                    thi=rng.randint(64, 192), D=16 * _log(rng, 2, 16), iters=10, grid=rng.choice([2, 3]), sizes=rng.randint(0, 1 << 20))
    H, W = _log(rng, 64, 512), _log(rng, 64, 512)
    return dict(op=op, B=rng.randint(1, 8), H=H, W=W, D=16 * _log(rng, 1, 16), k=_log(rng, 8, 64),
                th=_log(rng, 16, min(64, H // 2)), tw=_log(rng, 16, min(64, W // 2)), grid=rng.choice([2, 3]),
                tau=rng.choice([0.1, 0.3, 1.0]))


# ------------------------------------------------------------------ inputs (plain torch)
class _Scene:
    """Superpixel index of every pixel, and each superpixel's feature vector."""

    def __init__(self, H, W, D, g):
        M = max(8, min(128, H * W // 2048))
        n_sp = max(32, H * W // 210)
        mu = torch.rand((M, D), generator=g, device=DEV)
        cell = math.sqrt(H * W / n_sp)
        gy, gx = math.ceil(H / cell), math.ceil(W / cell)
        jit = torch.rand((gy, gx, 2), generator=g, device=DEV)
        cy = (torch.arange(gy, device=DEV)[:, None] + jit[..., 0]) * cell
        cx = (torch.arange(gx, device=DEV)[None, :] + jit[..., 1]) * cell
        py = (torch.arange(H, device=DEV) + 0.5)[:, None].expand(H, W)
        px = (torch.arange(W, device=DEV) + 0.5)[None, :].expand(H, W)
        iy, ix = (py / cell).long().clamp(0, gy - 1), (px / cell).long().clamp(0, gx - 1)
        best = torch.full((H, W), float("inf"), device=DEV)
        self.id = torch.zeros((H, W), dtype=torch.int64, device=DEV)
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                ny, nx = (iy + dy).clamp(0, gy - 1), (ix + dx).clamp(0, gx - 1)
                d = (cy[ny, nx] - py) ** 2 + (cx[ny, nx] - px) ** 2
                better = d < best
                best = torch.where(better, d, best)
                self.id = torch.where(better, ny * gx + nx, self.id)
        comp = torch.randint(0, M, (gy * gx,), generator=g, device=DEV)
        self.vec = mu[comp] + 0.05 * torch.randn((gy * gx, D), generator=g, device=DEV)
        self.mu, self.H, self.W, self.D = mu, H, W, D

    def rows(self, y0, y1, g):
        X = self.vec[self.id[y0:y1]]
        X.add_(torch.randn(X.shape, generator=g, device=DEV), alpha=0.02)
        return X.relu_()

    def chunks(self):
        n = max(1, (1 << 27) // (self.W * self.D))
        return [(y, min(self.H, y + n)) for y in range(0, self.H, n)]

    def features(self, g):
        X = torch.empty((self.H, self.W, self.D), device=DEV)
        for y0, y1 in self.chunks():
            X[y0:y1] = self.rows(y0, y1, g)
        return X

    def template(self, th, tw, g):
        """A th x tw patch: rotated, scaled, a quarter of it hidden, noisy."""
        u = torch.rand(6, generator=g, device=DEV).tolist()
        a, s = math.radians(60 * u[0] - 30), 0.8 + 0.45 * u[1]
        m = min(0.5 * math.hypot(th, tw) * 1.25 + 2, self.H / 2, self.W / 2)
        cy, cx = m + (self.H - 2 * m) * u[2], m + (self.W - 2 * m) * u[3]
        i = (torch.arange(th, device=DEV) - (th - 1) / 2)[:, None]
        j = (torch.arange(tw, device=DEV) - (tw - 1) / 2)[None, :]
        y = (cy + s * (math.cos(a) * i - math.sin(a) * j)).clamp(0, self.H - 1.001)
        x = (cx + s * (math.sin(a) * i + math.cos(a) * j)).clamp(0, self.W - 1.001)
        y0, x0 = y.long().clamp(max=self.H - 2), x.long().clamp(max=self.W - 2)
        fy, fx = (y - y0)[..., None], (x - x0)[..., None]
        v, ids = self.vec, self.id
        T = ((1 - fy) * ((1 - fx) * v[ids[y0, x0]] + fx * v[ids[y0, x0 + 1]])
             + fy * ((1 - fx) * v[ids[y0 + 1, x0]] + fx * v[ids[y0 + 1, x0 + 1]])).relu_()
        oh, ow = max(1, th // 2), max(1, tw // 2)
        oy, ox = int(u[4] * (th - oh)), int(u[5] * (tw - ow))
        occ = self.mu[int(u[4] * 997) % len(self.mu)] + 0.05 * torch.randn((oh, ow, self.D), generator=g, device=DEV)
        T[oy:oy + oh, ox:ox + ow] = occ.relu_()
        T.add_(torch.randn(T.shape, generator=g, device=DEV), alpha=0.05)
        return T.relu_().contiguous()


def _near(X, C):
    """Nearest codebook row of every row of X (the type of the inputs)."""
    cn = (C * C).sum(1)
    n = max(1, (1 << 26) // len(C))
    return torch.cat([(cn - 2 * (x @ C.T)).argmin(1) for x in X.split(n)])


def _codebook(T, k, g):
    """A k-means codebook to have in hand (not the method's seeded one)."""
    X = T.reshape(-1, T.shape[-1])
    C = X[torch.randperm(len(X), generator=g, device=DEV)[:k]].clone()
    for _ in range(8):
        one = torch.nn.functional.one_hot(_near(X, C), k).float()
        n = one.sum(0)[:, None]
        C = torch.where(n > 0, (one.T @ X) / n.clamp(min=1), C)
    return C.contiguous()


def _bank(th, tw, grid):
    """grid > 0: the full window and grid x grid cells.  grid = 0: the paper's Gaussian and
    Haar filters (equal bin weights) at three sub-scales, as integer-weighted rectangles."""
    if grid:
        bx, by = [i * tw // grid for i in range(grid + 1)], [i * th // grid for i in range(grid + 1)]
        rects = [(0, 0, tw, th)] + [(bx[c], by[r], bx[c + 1], by[r + 1]) for r in range(grid) for c in range(grid)]
        return [dict(rects=[(*r, 1)], w_f=1.0, area=float((r[2] - r[0]) * (r[3] - r[1]))) for r in rects]
    bank = []
    for s in (1, 2, 3):
        w, h = tw // s, th // s
        x0, y0 = (tw - w) // 2, (th - h) // 2
        bx, by = [x0 + i * w // 3 for i in range(4)], [y0 + i * h // 3 for i in range(4)]
        cols = lambda ws: [(bx[i], by[0], bx[i + 1], by[3], v) for i, v in enumerate(ws) if v]  # noqa: E731
        rows = lambda ws: [(bx[0], by[i], bx[3], by[i + 1], v) for i, v in enumerate(ws) if v]  # noqa: E731
        for rects, wf in (([(bx[0], by[0], bx[3], by[3], 1)], 1.0), (cols((1, 0, -1)), 0.25), (rows((1, 0, -1)), 0.25),
                          (cols((1, -2, 1)), 0.25), (rows((1, -2, 1)), 0.25)):
            bank.append(dict(rects=rects, w_f=wf / s, area=float(w * h)))
    return bank


def _counts(lab, k, bank):
    """F x k responses of the template labels `lab`."""
    out = torch.zeros((len(bank), k), dtype=torch.int64, device=DEV)
    for f, b in enumerate(bank):
        for x0, y0, x1, y1, w in b["rects"]:
            out[f] += w * torch.bincount(lab[y0:y1, x0:x1].reshape(-1).long(), minlength=k)
    return out


def _sizes(case):
    """The uneven sizes of a batch: queries, then templates with their k."""
    r = random.Random(case["sizes"])
    q = [(r.randint(case["lo"], case["hi"]), r.randint(case["lo"], case["hi"])) for _ in range(case["nq"])]
    t = [(r.randint(case["tlo"], case["thi"]), r.randint(case["tlo"], case["thi"]), r.choice([8, 16, 32, 64, 128, 256]))
         for _ in range(case["nt"])]
    return q, [(h, w, min(k, h * w)) for h, w, k in t]


def _inputs(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000 * int(seed) + 17)
    op, c = case["op"], case
    if op == "batch":
        q, t = _sizes(c)
        scenes = [_Scene(H, W, c["D"], g) for H, W in q]
        return dict(X=[s.features(g) for s in scenes],
                    T=[scenes[j % len(scenes)].template(h, w, g) for j, (h, w, _) in enumerate(t)], ks=[k for _, _, k in t])
    if op == "fit":
        return dict(T=_Scene(2 * c["th"] + 8, 2 * c["tw"] + 8, c["D"], g).template(c["th"], c["tw"], g))
    if op == "soft":
        scenes = [_Scene(c["H"], c["W"], c["D"], g) for _ in range(c["B"])]
        X = torch.stack([s.features(g) for s in scenes])
        T = scenes[0].template(c["th"], c["tw"], g)
        H, W = c["H"] - c["th"] + 1, c["W"] - c["tw"] + 1
        return dict(X=X, T=T, C=_codebook(T, c["k"], g), wf=torch.ones(c["grid"] ** 2, device=DEV),
                    dheat=torch.randn((c["B"], H, W), generator=g, device=DEV))
    scene = _Scene(c["H"], c["W"], c["D"], g)
    if op == "pair":
        return dict(T=scene.template(c["th"], c["tw"], g), X=scene.features(g))
    if op == "assign":
        C = _codebook(scene.template(min(128, c["H"]), min(128, c["W"]), g), c["k"], g)
        return dict(X=scene.features(g), C=C)
    T = scene.template(c["th"], c["tw"], g)  # score: the labels that the path's earlier steps leave
    k = min(c["k"], c["th"] * c["tw"])
    C = _codebook(T, k, g)
    lab = torch.empty((c["H"], c["W"]), dtype=torch.uint8, device=DEV)
    for y0, y1 in scene.chunks():
        lab[y0:y1] = _near(scene.rows(y0, y1, g).reshape(-1, c["D"]), C).reshape(y1 - y0, -1).to(torch.uint8)
    bank = _bank(c["th"], c["tw"], c["grid"])
    tl = _near(T.reshape(-1, c["D"]), C).reshape(c["th"], c["tw"])
    return dict(q=lab, k=k, bank=bank, counts=_counts(tl, k, bank).int())


# ------------------------------------------------------------------ the calls
def prepare(case, seed):
    c, s = case, _inputs(case, seed)
    s["case"] = c
    size = lambda op, H, W, **a: vq.Workspace(vq.vqnnf_workspace_bytes(op, H, W, **a))  # noqa: E731
    FIT, ASSIGN, SCORE = 0, 1, 3
    if c["op"] == "pair":
        s["bank"] = vq.Bank(_bank(c["th"], c["tw"], c["grid"]))
        p = dict(D=c["D"], k=c["k"], prec=c["prec"])
        s["ws"] = (size(FIT, c["th"], c["tw"], **p), size(ASSIGN, c["H"], c["W"], **p),
                   size(SCORE, c["H"], c["W"], k=c["k"], th=c["th"], tw=c["tw"], F=s["bank"].F))
    elif c["op"] == "assign":
        s["ws"] = size(ASSIGN, c["H"], c["W"], D=c["D"], k=c["k"], prec=c["prec"])
    elif c["op"] == "fit":
        s["ws"] = size(FIT, c["th"], c["tw"], D=c["D"], k=c["k"], prec=c["prec"])
    elif c["op"] == "score":
        s["bank"] = vq.Bank(s["bank"])
        s["ws"] = size(SCORE, c["H"], c["W"], k=s["k"], th=c["th"], tw=c["tw"], F=s["bank"].F)
    elif c["op"] == "batch":
        s["ws"] = vq.Workspace(vq.vqnnf_batch_workspace_bytes(s["X"], s["T"], s["ks"], c["grid"]))
    else:
        for n in ("X", "C", "wf"):
            s[n].requires_grad_(True)
    return s


def run(s):
    c = s["case"]
    op = c["op"]
    if op == "pair":
        wf, wa, wsc = s["ws"]
        C = vq.vqnnf_fit_codebook(s["T"], c["k"], c["iters"], 7, c["prec"], ws=wf)
        tl = vq.vqnnf_assign(s["T"], C, c["prec"], ws=wa)
        counts = vq.vqnnf_filter_responses(tl, c["k"], s["bank"])
        ql = vq.vqnnf_assign(s["X"], C, c["prec"], ws=wa)
        heat, yx = vq.vqnnf_score(ql, c["k"], c["th"], c["tw"], s["bank"], counts, ws=wsc)
        return dict(C=C, counts=counts, heat=heat, ql=ql, tl=tl, yx=yx)
    if op == "assign":
        return vq.vqnnf_assign(s["X"], s["C"], c["prec"], ws=s["ws"])
    if op == "fit":
        return vq.vqnnf_fit_codebook(s["T"], c["k"], c["iters"], 7, c["prec"], ws=s["ws"])
    if op == "score":
        heat, yx = vq.vqnnf_score(s["q"], s["k"], c["th"], c["tw"], s["bank"], s["counts"], ws=s["ws"])
        return dict(heat=heat, yx=yx)
    if op == "batch":
        heats, yx = vq.vqnnf_match_batch(s["X"], s["T"], s["ks"], c["iters"], 7, c["grid"], ws=s["ws"])
        return dict(heat=[h for row in heats for h in row], yx=yx)
    for n in ("X", "C", "wf"):
        s[n].grad = None
    heat = vq.soft_heatmap(s["X"], s["T"], s["C"], s["wf"], c["tau"], c["grid"])
    heat.backward(s["dheat"])
    return dict(heat=heat.detach(), dX=s["X"].grad, dC=s["C"].grad, dwf=s["wf"].grad)


# ------------------------------------------------------------------ work and exact values
def work(case):
    c, op = case, case["op"]

    def assign(px, D, k):
        return 4 * px * D + px + 4 * k * D, 2 * px * k * D

    def fit(px, D, k, iters):  # the template is read once; every step needs every distance
        return 4 * px * D + 4 * k * D, iters * (2 * px * k * D + px * D)

    def score(H, W, th, tw, k, F):  # labels in, heatmap out; |t - n| for every filter and cluster
        wins = (H - th + 1) * (W - tw + 1)
        return H * W + 4 * wins, 2 * wins * F * k

    if op == "assign":
        parts = [assign(c["H"] * c["W"], c["D"], c["k"])]
    elif op == "fit":
        parts = [fit(c["th"] * c["tw"], c["D"], c["k"], c["iters"])]
    elif op == "score":
        parts = [score(c["H"], c["W"], c["th"], c["tw"], c["k"], c["grid"] ** 2 + 1 if c["grid"] else 15)]
    elif op == "pair":
        F = c["grid"] ** 2 + 1 if c["grid"] else 15
        parts = [fit(c["th"] * c["tw"], c["D"], c["k"], c["iters"]), assign(c["th"] * c["tw"], c["D"], c["k"]),
                 assign(c["H"] * c["W"], c["D"], c["k"]), score(c["H"], c["W"], c["th"], c["tw"], c["k"], F)]
    elif op == "batch":
        q, t = _sizes(c)
        parts = [fit(h * w, c["D"], k, c["iters"]) for h, w, k in t]
        for H, W in q:
            parts.append((4 * H * W * c["D"], 2 * H * W * c["D"] * sum(k for _, _, k in t)))
            parts += [(4 * (H - h + 1) * (W - w + 1), 2 * (H - h + 1) * (W - w + 1) * (c["grid"] ** 2 + 1) * k)
                      for h, w, k in t]
    else:
        px, wins = c["B"] * c["H"] * c["W"], c["B"] * (c["H"] - c["th"] + 1) * (c["W"] - c["tw"] + 1)
        # features in, their gradient out, heatmap out and its gradient in; distances and two
        # gradient contractions, and |T - Q| with its sign for every cell and cluster
        parts = [(8 * px * c["D"] + 8 * wins, 7 * px * c["D"] * c["k"] + 4 * wins * c["grid"] ** 2 * c["k"])]
    return dict(bytes=sum(p[0] for p in parts), flops=sum(p[1] for p in parts))


def _fit64(T, k, iters, seed):
    """The method's k-means: k distinct pixels of a seeded shuffle (SplitMix64), `iters` steps of
    nearest centroid and mean, each mean rounded to float32 as the codebook's type."""
    X = T.reshape(-1, T.shape[-1]).double()
    order, state, mask = list(range(len(X))), seed, (1 << 64) - 1
    for i in range(k):
        state = (state + 0x9E3779B97F4A7C15) & mask
        z = state
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        z ^= z >> 31
        j = i + z % (len(X) - i)
        order[i], order[j] = order[j], order[i]
    C = X[torch.tensor(order[:k], device=DEV)]
    for _ in range(iters):
        one = torch.nn.functional.one_hot(_near(X, C.float().double()), k).double()
        n = one.sum(0)[:, None]
        C = torch.where(n > 0, (one.T @ X) / n.clamp(min=1), C.float().double())
    return C


def _heat64(q, k, th, tw, bank, counts):
    H, W = q.shape
    out = torch.zeros((H - th + 1, W - tw + 1), dtype=torch.float64, device=DEV)
    l1 = torch.zeros((len(bank), *out.shape), dtype=torch.int32, device=DEV)
    for j in range(k):
        S = torch.zeros((H + 1, W + 1), dtype=torch.int32, device=DEV)
        S[1:, 1:] = (q == j).cumsum(0, dtype=torch.int32).cumsum(1, dtype=torch.int32)
        at = lambda y, x: S[y:y + H - th + 1, x:x + W - tw + 1]  # noqa: E731
        for f, b in enumerate(bank):
            n = sum(w * (at(y1, x1) - at(y0, x1) - at(y1, x0) + at(y0, x0)) for x0, y0, x1, y1, w in b["rects"])
            l1[f] += (n - counts[f, j]).abs().int()
    for f, b in enumerate(bank):
        out -= b["w_f"] / b["area"] * l1[f].double()
    return out


def _near64(X, C):
    X, C = X.reshape(-1, X.shape[-1]), C.float().double()
    return torch.cat([_near(x.double(), C) for x in X.split(1 << 18)])


def exact(case, seed):
    c, op = case, case["op"]
    if op == "assign":
        return None  # labels only
    s = _inputs(case, seed)
    if op == "fit":
        return _fit64(s["T"], c["k"], c["iters"], 7)
    if op == "score":
        return dict(heat=_heat64(s["q"], s["k"], c["th"], c["tw"], s["bank"], s["counts"]), yx=None)
    if op == "pair":
        bank = _bank(c["th"], c["tw"], c["grid"])
        C = _fit64(s["T"], c["k"], c["iters"], 7)
        tl = _near64(s["T"], C).reshape(c["th"], c["tw"])
        ql = _near64(s["X"], C).reshape(c["H"], c["W"])
        heat = _heat64(ql, c["k"], c["th"], c["tw"], bank, _counts(tl, c["k"], bank))
        return dict(C=C, counts=None, heat=heat, ql=None, tl=None, yx=None)
    if op == "batch":
        sides = []
        for j, (T, k) in enumerate(zip(s["T"], s["ks"])):
            bank = _bank(T.shape[0], T.shape[1], c["grid"])
            C = _fit64(T, k, c["iters"], 7 + j)
            sides.append((bank, C, _counts(_near64(T, C).reshape(T.shape[:2]), k, bank)))
        heats = []
        for X in s["X"]:
            for (bank, C, counts), T, k in zip(sides, s["T"], s["ks"]):
                ql = _near64(X, C).reshape(X.shape[:2])
                heats.append(_heat64(ql, k, T.shape[0], T.shape[1], bank, counts))
        return dict(heat=heats, yx=None)
    # soft: the definition under autograd, one query at a time
    G, tau = c["grid"], c["tau"]
    T = s["T"].reshape(-1, c["D"]).double()
    C = s["C"].double().requires_grad_(True)
    wf = s["wf"].double().requires_grad_(True)
    bx, by = [i * c["tw"] // G for i in range(G + 1)], [i * c["th"] // G for i in range(G + 1)]
    cells = [(by[r], by[r + 1], bx[q], bx[q + 1]) for r in range(G) for q in range(G)]

    def soft(X, C):
        d = (X * X).sum(1)[:, None] - 2 * (X @ C.T) + (C * C).sum(1)
        return torch.softmax(-d / tau, 1)

    heats, grads = [], []
    for b in range(c["B"]):
        X = s["X"][b].reshape(-1, c["D"]).double().requires_grad_(True)
        pt = soft(T, C).T.reshape(-1, c["th"], c["tw"])
        p = soft(X, C).T.reshape(-1, c["H"], c["W"])
        S = torch.nn.functional.pad(p.cumsum(1).cumsum(2), (1, 0, 1, 0))
        H, W = c["H"] - c["th"] + 1, c["W"] - c["tw"] + 1
        heat = 0
        for f, (y0, y1, x0, x1) in enumerate(cells):
            at = lambda y, x: S[:, y:y + H, x:x + W]  # noqa: E731
            n = at(y1, x1) - at(y0, x1) - at(y1, x0) + at(y0, x0)
            l1 = (pt[:, y0:y1, x0:x1].sum((1, 2))[:, None, None] - n).abs().sum(0)
            heat = heat - wf[f] / ((y1 - y0) * (x1 - x0)) * l1
        heat.backward(s["dheat"][b].double())
        heats.append(heat.detach())
        grads.append(X.grad.reshape(c["H"], c["W"], c["D"]))
    return dict(heat=torch.stack(heats), dX=torch.stack(grads), dC=C.grad, dwf=wf.grad)
