"""The calls whose speed this library is judged by, each through its public entry points.

A case is a dict of plain values.  `prepare` makes what a program holds before
the call -- a context with its uploaded memory, the query embeddings, the
network's weights -- from the seed alone; `run` is one pass as a program makes
it; `work` counts the bytes and operations no implementation can avoid; `exact`
gives the floating-point outputs in 64 bits from plain torch and numpy.

Inputs follow the workloads of the benchmark: boxes uniform over the extent,
lognormal sizes, descriptors around unit class centroids (noise norm about
0.15) with 30% of the objects in dense look-alike classes, cameras on a
120-degree arc 2 m from each object, and queries planted on an object with
landmarks near it.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2606_15476_gb300 import farm as F

K_TOP = 10                    # TopK records a query returns
MU, W_BLEND, CLASS_MIS = 5.0, 0.5, 0.3
K_ANCHOR = 16
CHANNELS = ((1, 1.0, 1.0), (1, 0.5, 2.0), (0, 0.75, 1.0), (2, 1.0, 1.0))   # (space, weight, noise multiplier)
SPACE_DIMS = (1024, 2048)     # the text space and the second image space
HIDDEN, OUT_DIM = 512, 128    # the prefilter network
TAU_F, H_MAX, MAX_M = 0.8, 0.9, 8
PREC = {"fp32": F.PREC_FP32, "bf16": F.PREC_BF16, "fp8": F.PREC_FP8, "learned": F.PREC_LEARNED}


def listed():
    return [
        # the smallest call: a robot in a furnished room asks one question; latency and launches are all of it
        _query("room_one", n=200, dim=512, views=4, n_q=1, m_lo=2, m_hi=2, preds=9),
        # a query service: a dozen users' questions about a site arrive together in host memory, answers go back to it
        _query("site_dozen_host", n=20000, dim=1152, views=8, n_q=12, m_lo=0, m_hi=4, preds=9, host=True),
        # the benchmark: 4,096 standing queries over the 20,000-object site, re-scored as one graph
        _query("site_batch", n=20000, dim=1152, views=8, n_q=4096, m_lo=1, m_hi=4, graph=True),
        # a building portfolio: 67 memories of 100 to 20,000 objects, 44,000 queries in one batch
        {"name": "portfolio_batch", "kind": "multi", "scenes": 67, "n_lo": 100, "n_hi": 20000, "dim": 1152, "views": 8,
         "n_q": 44000, "m_lo": 0, "m_hi": 4, "preds": 5, "prec": "fp32", "graph": True},
        # the largest: a 100,000-object campus, 16,384 queries in BF16 with the FP32 rescore
        _query("campus_bf16", n=100000, dim=1152, views=8, n_q=16384, m_lo=1, m_hi=4, prec="bf16", graph=True),
        # the same campus through the learned prefilter, an odd number of queries
        _query("campus_learned", n=100000, dim=1152, views=8, n_q=6001, m_lo=1, m_hi=4, prec="learned", graph=True),
        # four retrieval channels over three embedding spaces (caption text, two image spaces)
        {"name": "channels_site", "kind": "channels", "n": 20000, "dim": 1152, "views": 8, "n_q": 1024, "m_lo": 1,
         "m_hi": 4, "preds": 5},
        # mapping: a frame batch's detections merged into the site's entities
        {"name": "associate_site", "kind": "associate", "n_ent": 20000, "n_det": 4096, "feat": 256},
        # a real-time loop with a fixed GPU memory budget: ranked lists of a few embeddings, nothing allocated
        {"name": "rank_realtime", "kind": "rank", "n": 20000, "dim": 1152, "rows": 48, "r": 95},
        # the similarity layer by itself: a tracker wants every cosine, for odd numbers of rows and objects
        {"name": "similarity_odd", "kind": "similarity", "n": 19997, "dim": 768, "rows": 501, "prec": "fp32"},
        # training: one epoch of the prefilter network over mined pairs (forward, backward, Adam)
        {"name": "prefilter_epoch", "kind": "train", "n": 20000, "dim": 1152, "rows": 2000, "pairs": 120000,
         "batch": 4096},
        # the memory changed: a mapper replaces a scene and asks again
        {"name": "refresh_and_ask", "kind": "refresh", "n": 20000, "dim": 1152, "views": 8, "n_q": 64, "m_lo": 1,
         "m_hi": 4, "preds": 9, "prec": "fp32", "graph": False, "host": False},
    ]


def _query(name, *, n, dim, views, n_q, m_lo, m_hi, preds=5, prec="fp32", graph=False, host=False):
    return {"name": name, "kind": "query", "n": n, "dim": dim, "views": views, "n_q": n_q, "m_lo": m_lo, "m_hi": m_hi,
            "preds": preds, "prec": prec, "graph": graph, "host": host}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the kinds in about the proportion of their use, sizes spread over the logarithm of their range."""
    kind = rng.choice(["query"] * 5 + ["multi", "channels", "associate", "rank", "similarity", "train", "refresh"])
    dim = rng.choice([256, 512, 768, 1000, 1152])
    if kind == "query":
        n = _log_int(rng, 40, 100000)
        m_hi = rng.randint(0, 4)
        prec = rng.choice(["fp32"] * 5 + ["bf16", "bf16", "learned", "fp8"])
        # no more rows x objects than the listed batches of that arithmetic
        most = 16384 * 100000 // (1 if prec in ("bf16", "learned") else 4)
        n_q = _log_int(rng, 1, max(1, min(16384, most // n)))
        c = _query("", n=n, dim=dim, views=rng.choice([1, 4, 8]), n_q=n_q, m_lo=rng.randint(0, m_hi), m_hi=m_hi,
                   preds=rng.choice([5, 9]), prec=prec, graph=rng.random() < 0.5, host=n_q <= 4096 and rng.random() < 0.3)
    elif kind == "multi":
        c = {"kind": kind, "scenes": rng.randint(2, 40), "n_lo": 100, "n_hi": _log_int(rng, 400, 20000), "dim": dim,
             "views": 8, "n_q": _log_int(rng, 60, 20000), "m_lo": 0, "m_hi": 4, "preds": 5,
             "prec": rng.choice(["fp32", "fp32", "bf16"]), "graph": rng.random() < 0.5}
    elif kind == "channels":
        c = {"kind": kind, "n": _log_int(rng, 600, 20000), "dim": dim, "views": 8, "n_q": _log_int(rng, 1, 1024), "m_lo": 1,
             "m_hi": 4, "preds": 5}
    elif kind == "associate":
        c = {"kind": kind, "n_ent": _log_int(rng, 300, 40000), "n_det": _log_int(rng, 16, 4096),
             "feat": rng.choice([64, 256, 500])}
    elif kind == "rank":
        n = _log_int(rng, 200, 30000)
        c = {"kind": kind, "n": n, "dim": dim, "rows": _log_int(rng, 1, 128), "r": rng.randint(1, 128)}
    elif kind == "similarity":
        c = {"kind": kind, "n": _log_int(rng, 100, 60000), "dim": dim, "rows": _log_int(rng, 1, 1500),
             "prec": rng.choice(["fp32", "fp32", "bf16"])}
    elif kind == "train":
        c = {"kind": kind, "n": _log_int(rng, 2000, 20000), "dim": dim, "rows": _log_int(rng, 100, 2000),
             "pairs": _log_int(rng, 4000, 120000), "batch": rng.choice([1024, 4096])}
    else:
        c = {"kind": kind, "n": _log_int(rng, 100, 20000), "dim": dim, "views": rng.choice([4, 8]), "n_q": rng.randint(1, 64),
             "m_lo": 1, "m_hi": 4, "preds": 9, "prec": "fp32", "graph": False, "host": False}
    c.pop("name", None)
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 13)


def _unit(x):
    return x / x.norm(dim=1, keepdim=True)


class _Scene:
    """One memory on the GPU: descriptors, classes, boxes [6, n], stored views [6, V, n]."""

    def __init__(self, g, rs, n, dim, views, extra_dims=()):
        side = 120.0 * math.sqrt(n / 20000.0)
        ext = torch.tensor([side, side, min(max(side / 12.0, 3.0), 10.0)], device="cuda")
        n_cls, n_dis = max(16, round(n / 50)), max(1, round(n / 1000))
        n_look = int(round(0.3 * n))
        cls = np.concatenate([np.arange(n_look) % n_dis, n_dis + rs.randint(0, n_cls - n_dis, n - n_look)])
        self.cls_np = cls[rs.permutation(n)].astype(np.int32)
        self.n, self.dim, self.n_dis, self.n_look, self.extent = n, dim, n_dis, n_look, ext
        self.cls = torch.from_numpy(self.cls_np).cuda()
        rows = self.cls.long()
        self.spaces = []                   # (descriptors, centroids, per-dimension noise) of each embedding space
        for d in (dim, *extra_dims):
            cen = _unit(torch.randn(n_cls, d, generator=g, device="cuda"))
            sg = 0.15 / math.sqrt(d)
            desc = _unit(cen[rows] + sg * torch.randn(n, d, generator=g, device="cuda"))
            self.spaces.append((desc.contiguous(), cen, sg))
        self.desc = self.spaces[0][0]
        centre = torch.rand(n, 3, generator=g, device="cuda") * ext
        size = torch.exp(-1.0 + 0.5 * torch.randn(n, 3, generator=g, device="cuda"))
        self.box = torch.cat([centre.T, size.T]).contiguous()
        th = 2 * math.pi * torch.rand(n, generator=g, device="cuda")
        step = math.radians(120.0) / max(views - 1, 1)
        v = torch.zeros(6, views, n, device="cuda")
        for k in range(views):
            dx, dy = torch.cos(th + step * k), torch.sin(th + step * k)
            v[0, k], v[1, k], v[2, k] = centre[:, 0] + 2.0 * dx, centre[:, 1] + 2.0 * dy, centre[:, 2]
            v[3, k], v[4, k] = -dx, -dy
        self.views = v


class _Queries:
    """Queries of one scene: planted targets (half of them look-alikes), landmarks near them, embeddings per channel."""

    def __init__(self, g, rs, sc, n_q, m_lo, m_hi, preds, channels=((0, 1.0, 1.0),)):
        look = np.flatnonzero(sc.cls_np < sc.n_dis)
        rest = np.flatnonzero(sc.cls_np >= sc.n_dis)
        pick = rs.uniform(size=n_q) < 0.5
        tgt = np.where(pick & (look.size > 0), look[rs.randint(0, max(look.size, 1), n_q)] if look.size else 0,
                       rest[rs.randint(0, rest.size, n_q)] if rest.size else 0)
        m = rs.randint(m_lo, m_hi + 1, n_q)
        self.c_off = np.concatenate([[0], np.cumsum(m)]).astype(np.int32)
        n_c = int(self.c_off[-1])
        self.c_pred = rs.randint(0, preds, n_c).astype(np.int32)
        self.tgt_cls = sc.cls_np[tgt].astype(np.int32)
        t = torch.from_numpy(tgt).cuda()
        # a landmark: the nearest to the target of a few hundred random objects
        owner = torch.from_numpy(np.repeat(np.arange(n_q), m)).cuda()
        centre = sc.box[:3].T.contiguous()
        lm = torch.zeros(n_c, dtype=torch.long, device="cuda")
        for c0 in range(0, n_c, 8192):
            own = t[owner[c0:c0 + 8192]]
            cand = torch.randint(0, sc.n, (own.numel(), 256), generator=g, device="cuda")
            d = (centre[cand] - centre[own][:, None]).square().sum(-1)
            d[cand == own[:, None]] = float("inf")
            lm[c0:c0 + 8192] = cand.gather(1, d.argmin(1, keepdim=True))[:, 0]
        self.tgt_emb, self.c_emb = [], []
        for sp, _, mult in channels:
            _, cen, sg = sc.spaces[sp]
            cl = sc.cls.long()
            noise = lambda k: mult * sg * torch.randn(k, cen.shape[1], generator=g, device="cuda")  # noqa: E731
            self.tgt_emb.append((cen[cl[t]] + noise(n_q)).contiguous())
            self.c_emb.append((cen[cl[lm]] + noise(n_c)).contiguous())
        self.n_q, self.n_c = n_q, n_c


def _inputs(case, seed):
    """Everything random of a case, on the GPU (metadata on the host)."""
    g, rs, kind = _gen(seed), np.random.RandomState((int(seed) * 2654435761 + 17) % (1 << 32)), case["kind"]
    if kind in ("query", "refresh"):
        sc = _Scene(g, rs, case["n"], case["dim"], case["views"])
        q = _Queries(g, rs, sc, case["n_q"], case["m_lo"], case["m_hi"], case["preds"])
        return dict(scenes=[sc], parts=[q], mlp=_network(g, case["dim"]) if case["prec"] == "learned" else None)
    if kind == "multi":
        k = case["scenes"]
        ns = np.exp(rs.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]), k)).astype(np.int64)
        per = [case["n_q"] // k + (i < case["n_q"] % k) for i in range(k)]
        scenes = [_Scene(g, rs, int(n), case["dim"], case["views"]) for n in ns]
        parts = [_Queries(g, rs, s, p, case["m_lo"], case["m_hi"], case["preds"]) for s, p in zip(scenes, per)]
        return dict(scenes=scenes, parts=parts, mlp=None)
    if kind == "channels":
        sc = _Scene(g, rs, case["n"], case["dim"], case["views"], SPACE_DIMS)
        return dict(scenes=[sc], parts=[_Queries(g, rs, sc, case["n_q"], case["m_lo"], case["m_hi"], case["preds"], CHANNELS)])
    if kind in ("rank", "similarity"):
        sc = _Scene(g, rs, case["n"], case["dim"], 1)
        _, cen, sg = sc.spaces[0]
        own = torch.randint(0, sc.n, (case["rows"],), generator=g, device="cuda")
        return dict(scenes=[sc], rows=(cen[sc.cls[own].long()] + sg * torch.randn(case["rows"], case["dim"], generator=g,
                                                                                 device="cuda")).contiguous())
    if kind == "train":
        sc = _Scene(g, rs, case["n"], case["dim"], 1)
        q = _Queries(g, rs, sc, case["rows"], 0, 0, 5)
        rows, p = q.tgt_emb[0], case["pairs"]
        pr = torch.randint(0, case["rows"], (p,), generator=g, device="cuda")
        po = torch.randint(0, sc.n, (p,), generator=g, device="cuda")
        # a quarter of the pairs join a row with one of its best objects
        best = (_unit(rows) @ sc.desc.T).topk(min(256, sc.n), dim=1).indices
        near = torch.rand(p, generator=g, device="cuda") < 0.25
        po = torch.where(near, best[pr, torch.randint(0, best.shape[1], (p,), generator=g, device="cuda")], po)
        y = torch.empty(p, device="cuda")
        un = _unit(rows)
        for c0 in range(0, p, 65536):
            y[c0:c0 + 65536] = (un[pr[c0:c0 + 65536]] * sc.desc[po[c0:c0 + 65536]]).sum(1)
        host = lambda x, t: x.cpu().numpy().astype(t)  # noqa: E731
        return dict(scenes=[sc], mlp=_network(g, case["dim"]), rows=host(rows, np.float32), pair_row=host(pr, np.int32),
                    pair_obj=host(po, np.int32), y=host(y, np.float32), w=host(torch.where(near, 4.0, 1.0), np.float32))
    return _association(g, rs, case)


def _network(g, dim):
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    ws = (r(HIDDEN, dim) / math.sqrt(dim), 0.05 * r(HIDDEN), r(OUT_DIM, HIDDEN) / math.sqrt(HIDDEN), 0.05 * r(OUT_DIM))
    return [w.cpu().numpy().astype(np.float32) for w in ws]


def _association(g, rs, case):
    """Entities as Gaussians with features; detections re-observe one, bridge two of a class, or are new."""
    n, b, f = case["n_ent"], case["n_det"], case["feat"]
    sc = _Scene(g, rs, n, f, 1)
    centre, size = sc.box[:3].T, sc.box[3:].T
    rand = lambda *s: torch.rand(*s, generator=g, device="cuda")    # noqa: E731
    randn = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731

    def cov(sz, yaw):
        v, c, s = sz.square() / 12.0, torch.cos(yaw), torch.sin(yaw)
        z = torch.zeros_like(c)
        return torch.stack([c * c * v[:, 0] + s * s * v[:, 1], c * s * (v[:, 0] - v[:, 1]), z,
                            s * s * v[:, 0] + c * c * v[:, 1], z, v[:, 2]]).contiguous()

    yaw = math.pi * rand(n)
    src = torch.randint(0, n, (b,), generator=g, device="cuda")
    kind = rand(b)
    new, bridge = kind < 0.1, (kind >= 0.1) & (kind < 0.2)
    mu = centre[src] + 0.05 * randn(b, 3)
    sz, yw, cl = size[src] * (1 + 0.05 * randn(b, 3)).abs(), yaw[src] + 0.1 * randn(b), sc.cls[src].long()
    for c0 in range(0, b, 1024):
        e = src[c0:c0 + 1024]
        d = torch.cdist(centre[e], centre)
        d[(sc.cls[None, :] != sc.cls[e][:, None]) | (torch.arange(n, device="cuda")[None, :] == e[:, None])] = float("inf")
        far, o = d.min(1)
        on = bridge[c0:c0 + 1024] & torch.isfinite(far)
        mu[c0:c0 + 1024][on] = 0.5 * (centre[e] + centre[o])[on]
        sz[c0:c0 + 1024][on] = ((centre[e] - centre[o]).abs() + 0.5 * (size[e] + size[o]))[on]
    mu[new] = (rand(b, 3) * sc.extent)[new]
    cl[new] = torch.randint(0, int(sc.cls_np.max()) + 1, (b,), generator=g, device="cuda")[new]
    cen, sg = sc.spaces[0][1:]
    ent = dict(mu=sc.box[:3].contiguous(), cov=cov(size, yaw), feat=sc.desc,
               w=torch.randint(1, 21, (n,), generator=g, device="cuda").float(), active=(rand(n) >= 0.05).int())
    det = dict(mu=mu.T.contiguous(), cov=cov(sz, yw), feat=_unit(cen[cl] + sg * randn(b, f)).contiguous())
    return dict(ent=ent, det=det)


# ---------------------------------------------------------------------------
# What a program keeps, and one pass
# ---------------------------------------------------------------------------

class _State:
    def __init__(self, **kw):
        self.ctx = None
        self.__dict__.update(kw)

    def __del__(self):
        if self.ctx is not None:
            F.farm_destroy(self.ctx)      # (synchronises the context's stream)
            self.ctx = None


def _upload(ctx, sid, sc):
    F.farm_memory_upload(ctx, sid, sc.desc, sc.cls, sc.box, sc.views)


def prepare(case, seed):
    x, kind = _inputs(case, seed), case["kind"]
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    ctx = F.farm_create(0, stream)
    s = _State(ctx=ctx, case=case, kind=kind, stream=stream)
    if kind == "associate":
        s.ent, s.det = x["ent"], x["det"]
        n, b, f = case["n_ent"], case["n_det"], case["feat"]
        i32 = lambda *sh: torch.zeros(*sh, dtype=torch.int32, device="cuda")      # noqa: E731
        f32 = lambda *sh: torch.zeros(*sh, dtype=torch.float32, device="cuda")    # noqa: E731
        s.out = dict(match_cnt=i32(b), match_idx=i32(b, MAX_M), match_h=f32(b, MAX_M), parent=i32(n + b), w=f32(n + b),
                     mu=f32(3, n + b), cov=f32(6, n + b), feat=f32(n + b, f))
        torch.cuda.synchronize()
        return s
    for sid, sc in enumerate(x["scenes"]):
        if kind != "refresh":
            _upload(ctx, sid, sc)
    if x.get("mlp") is not None:
        F.farm_mlp_set(ctx, *x["mlp"])
    if kind in ("rank", "similarity"):
        s.rows, s.n = x["rows"], case["n"]
        if kind == "rank":
            s.idx = torch.zeros(case["rows"], case["r"], dtype=torch.int32, device="cuda")
            s.cos = torch.zeros(case["rows"], case["r"], device="cuda")
        else:
            s.out = torch.zeros(case["rows"], case["n"], device="cuda")
    elif kind == "train":
        s.weights, s.x = x["mlp"], x
        x.pop("scenes")
    else:
        parts = x["parts"]
        offs = np.cumsum([0] + [p.n_c for p in parts])
        s.c_off = np.concatenate([[0]] + [p.c_off[1:].astype(np.int64) + o for p, o in zip(parts, offs)]).astype(np.int32)
        s.c_pred = np.concatenate([p.c_pred for p in parts])
        s.tgt_cls = np.concatenate([p.tgt_cls for p in parts])
        s.scene_of_q = np.concatenate([np.full(p.n_q, i, np.int32) for i, p in enumerate(parts)])
        n_q = s.n_q = int(s.tgt_cls.size)
        s.tgt = [torch.cat([p.tgt_emb[c] for p in parts]) for c in range(len(parts[0].tgt_emb))]
        s.lm = [torch.cat([p.c_emb[c] for p in parts]) for c in range(len(parts[0].c_emb))]
        s.host = bool(case.get("host"))
        k = s.k = min([K_TOP] + [sc.n for sc in x["scenes"]])
        if kind == "channels":
            for sp in range(len(SPACE_DIMS)):
                F.farm_memory_add_space(ctx, 0, sp + 1, x["scenes"][0].spaces[sp + 1][0])
            s.channels = [(sp, w) for sp, w, _ in CHANNELS]
            s.tgt = torch.cat([t.reshape(-1) for t in s.tgt])      # channel after channel, as the call takes them
            s.lm = torch.cat([t.reshape(-1) for t in s.lm])
        else:
            s.tgt, s.lm, s.prec, s.graph = s.tgt[0], s.lm[0], PREC[case["prec"]], bool(case["graph"])
        if kind == "refresh":
            s.scene = x["scenes"][0]
            _upload(ctx, 0, s.scene)      # the scene that the refresh replaces
        shapes = [("idx", (n_q, k), torch.int32), ("score", (n_q, k), torch.float32), ("pred", (n_q, k, 4), torch.float32),
                  ("anchor", (n_q, k, 4), torch.int32)]
        if s.host:
            s.pinned = [t.cpu().pin_memory() for t in (s.tgt, s.lm)] + [torch.zeros(sh, dtype=dt).pin_memory()
                                                                        for _, sh, dt in shapes]
            s.tgt, s.lm = (t.numpy() for t in s.pinned[:2])
            s.out = {nm: t.numpy() for (nm, _, _), t in zip(shapes, s.pinned[2:])}
        else:
            s.out = {nm: torch.zeros(sh, dtype=dt, device="cuda") for nm, sh, dt in shapes}
    torch.cuda.synchronize()
    return s


def _ask(s):
    h = F.farm_query_batch(s.ctx, s.scene_of_q, s.tgt, s.tgt_cls, s.c_off, s.c_pred, s.lm, s.prec, graph=s.graph)
    return F.farm_topk(s.ctx, h, s.k, s.n_q, s.out["idx"], s.out["score"], s.out["pred"], s.out["anchor"])


def run(s):
    if s.kind in ("query", "multi"):
        return _ask(s)
    if s.kind == "refresh":
        _upload(s.ctx, 0, s.scene)
        return _ask(s)
    if s.kind == "channels":
        h = F.farm_query_batch_rrf(s.ctx, 0, s.channels, s.tgt, s.tgt_cls, s.c_off, s.c_pred, s.lm)
        return F.farm_topk(s.ctx, h, s.k, s.n_q, s.out["idx"], s.out["score"], s.out["pred"], s.out["anchor"])
    if s.kind == "associate":
        return F.farm_associate(s.ctx, s.ent, s.det, TAU_F, H_MAX, MAX_M, s.out)
    if s.kind == "rank":
        F.farm_rank_rows_noalloc(s.ctx, 0, s.rows, s.case["r"], F.PREC_FP32, s.idx, s.cos)
        return {"idx": s.idx, "cos": s.cos}
    if s.kind == "similarity":
        return {"cos": F.farm_similarity(s.ctx, 0, s.rows, s.n, PREC[s.case["prec"]], s.out)}
    F.farm_mlp_set(s.ctx, *s.weights)
    x = s.x
    losses = F.farm_mlp_train(s.ctx, 0, x["rows"], x["pair_row"], x["pair_obj"], x["y"], x["w"], epochs=1,
                              batch=s.case["batch"], lr=1e-3, seed=1)
    w1, b1, w2, b2 = F.farm_mlp_get(s.ctx, s.case["dim"], HIDDEN, OUT_DIM)
    return {"W1": w1, "b1": b1, "W2": w2, "b2": b2, "losses": losses}


def work(case):
    """Each input read once in the width the arithmetic needs, each output written once; 2 operations per product."""
    kind, dim = case["kind"], case.get("dim", 0)
    if kind == "associate":
        n, b, f = case["n_ent"], case["n_det"], case["feat"]
        return {"bytes": 4 * (n + b) * (f + 9) + 8 * n + 4 * b * (1 + 2 * MAX_M) + 4 * (n + b) * (f + 11),
                "flops": 2 * n * b * f}
    if kind == "rank":
        return {"bytes": 4 * dim * (case["n"] + case["rows"]) + 8 * case["rows"] * case["r"],
                "flops": 2 * case["rows"] * case["n"] * dim}
    if kind == "similarity":
        per = 2 if case["prec"] == "bf16" else 4
        return {"bytes": per * dim * case["n"] + 4 * dim * case["rows"] + 4 * case["rows"] * case["n"],
                "flops": 2 * case["rows"] * case["n"] * dim}
    if kind == "train":
        p = HIDDEN * dim + HIDDEN + OUT_DIM * HIDDEN + OUT_DIM
        steps = -(-case["pairs"] // case["batch"])
        # two towers forward and backward per pair; per step the gathered BF16 rows and Adam's weights and moments
        return {"bytes": case["pairs"] * 2 * dim * 2 + steps * p * 4 * 7, "flops": case["pairs"] * 2 * 6 * (p - HIDDEN - OUT_DIM)}
    rows = case["n_q"] * (1 + 0.5 * (case["m_lo"] + case["m_hi"]))
    out = case["n_q"] * K_TOP * 40
    if kind == "channels":
        dims = [(dim, *SPACE_DIMS)[sp] for sp, _, _ in CHANNELS]
        return {"bytes": 4 * case["n"] * (dim + sum(SPACE_DIMS)) + 4 * rows * sum(dims) + out,
                "flops": 2 * rows * case["n"] * sum(dims)}
    if kind == "multi":
        lo, hi, k = case["n_lo"], case["n_hi"], case["scenes"]
        n_mean = (hi - lo) / math.log(hi / lo) if hi > lo else lo
        return {"bytes": 4 * k * n_mean * dim + 4 * rows * dim + out, "flops": 2 * rows * n_mean * dim}
    per = {"fp32": 4, "bf16": 2, "fp8": 1}.get(case["prec"])
    if per is None:     # learned: the compressed rows for every object, then a list of 512 in full
        lists = case["n_q"] * min(512, case["n"])
        return {"bytes": 2 * OUT_DIM * case["n"] + 4 * rows * dim + out,
                "flops": 2 * rows * (case["n"] * OUT_DIM + HIDDEN * (dim + OUT_DIM)) + 2 * lists * dim}
    fresh = case["n"] * (4 * dim + 4 + 24 + 24 * case["views"]) if kind == "refresh" else 0
    return {"bytes": per * dim * case["n"] + fresh + 4 * rows * dim + out, "flops": 2 * rows * case["n"] * dim}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------

def exact(case, seed):
    kind = case["kind"]
    x = _inputs(case, seed)
    if kind == "associate":
        return _exact_association(x["ent"], x["det"])
    if kind in ("rank", "similarity"):
        cos = _unit(x["rows"].double()) @ _unit(x["scenes"][0].desc.double()).T
        return {"cos": cos} if kind == "similarity" else {"idx": None, "cos": cos.topk(case["r"], dim=1).values}
    if kind == "train":
        return _exact_training(case, x)
    if case["n_q"] * (1 + case["m_hi"]) * case.get("n", case.get("n_hi", 0)) * case["dim"] > 6e12:
        return None       # (more than about 20 seconds of 64-bit products)
    k = min([K_TOP] + [s.n for s in x["scenes"]])
    chan = [(sp, w) for sp, w, _ in CHANNELS] if kind == "channels" else [(0, None)]
    got = [_exact_scene(sc, q, chan, k) for sc, q in zip(x["scenes"], x["parts"])]
    # (reduced arithmetic may miss a true candidate, whose loss shifts the breakdown of all that follow it)
    whole = case.get("prec", "fp32") == "fp32"
    return {"idx": None, "score": torch.cat([a for a, _ in got]), "pred": torch.cat([b for _, b in got]) if whole else None,
            "anchor": None}


def _ranks(cos):
    order = torch.argsort(cos, dim=1, descending=True, stable=True)
    r = torch.empty_like(order)
    r.scatter_(1, order, torch.arange(1, cos.shape[1] + 1, device=cos.device).expand_as(order))
    return order, r


def _exact_scene(sc, q, chan, k):
    desc = {sp: _unit(sc.spaces[sp][0].double()) for sp, _ in chan}
    many = chan[0][1] is not None

    def best(rows, count):       # (objects, similarity score) of the best `count` objects per row
        if not many:
            idx = _topk_stable(_unit(rows[0].double()) @ desc[0].T, count)
            return idx, 1.0 / (MU + torch.arange(1, count + 1, device="cuda").double()).expand(idx.shape)
        f = 0.0
        for (sp, w), r in zip(chan, rows):
            f = f + w / (MU + _ranks(_unit(r.double()) @ desc[sp].T)[1].double())
        return None, f

    scores, preds = [], []
    step = max(1, int(1.5e8 / max(sc.n, 4096)))
    step = min(step, 256)
    off = q.c_off.astype(np.int64)
    for q0 in range(0, q.n_q, step):
        q1 = min(q.n_q, q0 + step)
        nq, c0, c1 = q1 - q0, off[q0], off[q1]
        tc = torch.from_numpy(q.tgt_cls[q0:q1]).cuda()
        ti, ts = best([t[q0:q1] for t in q.tgt_emb], min(128, sc.n))
        if many:
            full = torch.where(sc.cls[None] == tc[:, None], 1.0, CLASS_MIS) * ts
            cand = full.topk(min(512, sc.n), dim=1).indices.sort(dim=1).values
            s_sem = full.gather(1, cand)
        else:
            cand = ti
            s_sem = torch.where(sc.cls[ti] == tc[:, None], 1.0, CLASS_MIS) * ts
        t = torch.full((nq, cand.shape[1], 4), -1.0, dtype=torch.float64, device="cuda")
        if c1 > c0:
            li, ls = best([e[c0:c1] for e in q.c_emb], min(K_ANCHOR, sc.n))
            if many:
                li = _topk_stable(ls, min(K_ANCHOR, sc.n))
            owner = np.repeat(np.arange(nq), np.diff(off[q0:q1 + 1]))
            slot = np.arange(c1 - c0) - (off[q0:q1] - c0)[owner]
            ow = torch.from_numpy(owner).cuda()
            for p in np.unique(q.c_pred[c0:c1]):
                at = torch.from_numpy(np.flatnonzero(q.c_pred[c0:c1] == p)).cuda()
                for a0 in range(0, at.numel(), 64):
                    a = at[a0:a0 + 64]
                    e = cand[ow[a]]                                       # [m, candidates]
                    r = _relation(sc, int(p), e[:, :, None], li[a][:, None, :])
                    r = torch.where(li[a][:, None, :] == e[:, :, None], 0.0, r)
                    t[ow[a], :, torch.from_numpy(slot).cuda()[a]] = r.max(-1).values
        m = torch.from_numpy(np.diff(off[q0:q1 + 1])).cuda()
        has = t >= 0
        gbar = torch.where(has, t, 1.0).prod(-1).pow(1.0 / m.clamp(min=1).double()[:, None])
        s = s_sem * ((1 - W_BLEND) + W_BLEND * gbar)
        by_index = torch.argsort(cand, dim=1)                              # lower object index first on ties
        order = torch.argsort(s.gather(1, by_index), dim=1, descending=True, stable=True)[:, :k]
        pos = by_index.gather(1, order)
        scores.append(s.gather(1, pos))
        preds.append(t.gather(1, pos[:, :, None].expand(-1, -1, 4)))
    return torch.cat(scores), torch.cat(preds)


def _topk_stable(v, count):
    """The `count` largest per row in descending order (exact ties are not met)."""
    return v.topk(count, dim=1).indices


def _relation(sc, p, e, a):
    """The predicates 0-8 (above, below, left of, right of, near, next to, on, in front of, behind) in 64 bits."""
    box = sc.box.double()
    ce, ca = [box[i][e] for i in range(3)], [box[i][a] for i in range(3)]
    dz = ce[2] - ca[2]
    if p in (0, 1):
        return torch.sigmoid((dz if p == 0 else -dz) / 0.25)
    if p in (4, 5):
        d2 = sum((u - v).square() for u, v in zip(ce, ca))
        return torch.exp(-d2 / (2.0 * (0.5 if p == 4 else 1.0) ** 2))
    if p == 6:
        # (the library's float parameters 0.10)
        tenth = float(np.float32(0.10))
        rho = 0.5 * torch.maximum(box[3][a], box[4][a])
        dxy = torch.sqrt((ce[0] - ca[0]).square() + (ce[1] - ca[1]).square())
        gap = (ce[2] - 0.5 * box[5][e]) - (ca[2] + 0.5 * box[5][a])
        return torch.sigmoid((rho - dxy) / tenth) * torch.exp(-gap.square() / (2.0 * tenth ** 2))
    acc, cnt = 0.0, 0.0
    for k in range(sc.views.shape[1]):
        v = sc.views[:, k].double()
        fwd = v[3:] / v[3:].norm(dim=0)
        right = torch.stack([fwd[1], -fwd[0]])
        right = right / right.norm(dim=0)
        o, f, r = [v[i][e] for i in range(3)], [fwd[i][e] for i in range(3)], [right[i][e] for i in range(2)]
        ze = sum((c - w) * d for c, w, d in zip(ce, o, f))
        za = sum((c - w) * d for c, w, d in zip(ca, o, f))
        ok = ((ze > float(np.float32(0.05))) & (za > float(np.float32(0.05)))).double()
        if p in (7, 8):
            x = (za - ze) / 0.25
        else:
            xe = sum((c - w) * d for c, w, d in zip(ce[:2], o, r))
            xa = sum((c - w) * d for c, w, d in zip(ca[:2], o, r))
            x = (xa / za - xe / ze) / float(np.float32(0.10))
        acc, cnt = acc + ok * torch.sigmoid(torch.nan_to_num(x if p in (2, 7) else -x)), cnt + ok
    return torch.where(cnt > 0, acc / cnt.clamp(min=1.0), 0.5)


def _exact_training(case, x):
    """Full-precision Adam over the same shuffled mini-batches."""
    pairs, batch = case["pairs"], case["batch"]
    perm, state, m64 = list(range(pairs)), 1, (1 << 64) - 1
    for i in range(pairs - 1, 0, -1):                        # Fisher-Yates by SplitMix64 from the seed
        state = (state + 0x9E3779B97F4A7C15) & m64
        z = state
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m64
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m64
        j = (z ^ (z >> 31)) % (i + 1)
        perm[i], perm[j] = perm[j], perm[i]
    rows = _unit(torch.from_numpy(x["rows"]).cuda().double())
    desc = _unit(x["scenes"][0].desc.double())
    ps = [torch.from_numpy(w).cuda().double().requires_grad_() for w in x["mlp"]]
    opt = torch.optim.Adam(ps, lr=1e-3, betas=(0.9, 0.999), eps=1e-8)
    perm = np.asarray(perm)
    to = lambda v: torch.from_numpy(v).cuda()  # noqa: E731
    losses = []
    for s0 in range(0, pairs, batch):
        at = perm[s0:s0 + batch]
        pr, po, y, w = to(x["pair_row"][at]).long(), to(x["pair_obj"][at]).long(), to(x["y"][at]).double(), to(x["w"][at]).double()

        def f(v):
            return _unit(torch.nn.functional.gelu(v @ ps[0].T + ps[1]) @ ps[2].T + ps[3])
        loss = (w * ((f(rows[pr]) * f(desc[po])).sum(1) - y).square()).sum() / w.sum()
        opt.zero_grad()
        loss.backward()
        opt.step()
        losses.append(float(loss.detach()))
    w1, b1, w2, b2 = (p.detach().cpu().numpy() for p in ps)
    return {"W1": w1, "b1": b1, "W2": w2, "b2": b2, "losses": np.array([sum(losses) / len(losses)])}


def _exact_association(ent, det):
    n, b = ent["mu"].shape[1], det["mu"].shape[1]
    ef, df = _unit(ent["feat"].double()), _unit(det["feat"].double())
    full = lambda c: torch.stack([c[0], c[1], c[2], c[1], c[3], c[4], c[2], c[4], c[5]], -1).reshape(-1, 3, 3)  # noqa: E731
    em, dm, ec, dc = ent["mu"].T.double(), det["mu"].T.double(), full(ent["cov"].double()), full(det["cov"].double())
    di, ei, hs = [], [], []
    for d0 in range(0, b, 512):
        ok = (df[d0:d0 + 512] @ ef.T >= float(np.float32(TAU_F))) & (ent["active"][None] != 0)
        d, e = ok.nonzero(as_tuple=True)
        d = d + d0
        s = 0.5 * (dc[d] + ec[e])
        dx = (dm[d] - em[e])[:, :, None]
        q = (dx.transpose(1, 2) @ torch.linalg.inv(s) @ dx).reshape(-1)
        lbc = 0.25 * (torch.logdet(dc[d]) + torch.logdet(ec[e])) - 0.5 * torch.logdet(s) - 0.125 * q
        h = torch.sqrt(torch.clamp(-torch.expm1(lbc), min=0.0))
        keep = h <= float(np.float32(H_MAX))
        di.append(d[keep]), ei.append(e[keep]), hs.append(h[keep])
    di, ei, hs = torch.cat(di).cpu().numpy(), torch.cat(ei).cpu().numpy(), torch.cat(hs).cpu().numpy()
    order = np.lexsort((ei, hs, di))
    di, ei, hs = di[order], ei[order], hs[order]
    pos = np.arange(di.size) - np.searchsorted(di, di)
    keep = pos < MAX_M
    match_h = np.full((b, MAX_M), -1.0)
    match_h[di[keep], pos[keep]] = hs[keep]
    u, v = n + di[keep], ei[keep]
    label = np.arange(n + b)
    while True:                                               # components: the smallest slot of each
        low = np.minimum(label[u], label[v])
        new = label.copy()
        np.minimum.at(new, u, low)
        np.minimum.at(new, v, low)
        new = np.minimum(new, new[new])
        if np.array_equal(new, label):
            break
        label = new
    ew = ent["w"].double().cpu().numpy()
    win = np.full(n + b, -1)
    o = np.lexsort((-np.arange(n), ew))                       # ascending weight; of equals the lower index last
    win[label[:n][o]] = o
    parent = np.where(win[label] >= 0, win[label], np.arange(n + b))
    t = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    par, w = t(parent), torch.cat([ent["w"].double(), torch.ones(b, dtype=torch.float64, device="cuda")])
    mu, cov, feat = torch.cat([em, dm]), torch.cat([ec, dc]), torch.cat([ent["feat"].double(), det["feat"].double()])
    add = lambda v: torch.zeros_like(v).index_add_(0, par, v)  # noqa: E731
    wg = add(w)
    own = (par == torch.arange(n + b, device="cuda")) & (wg > 0)
    den = torch.where(own, wg, 1.0)
    mu_g = add(w[:, None] * mu) / den[:, None]
    dmu = mu - mu_g[par]
    cov_g = add((w[:, None, None] * (cov + dmu[:, :, None] * dmu[:, None, :])).reshape(-1, 9)) / den[:, None]
    feat_g = add(w[:, None] * feat) / den[:, None]
    z = own.double()
    return {"match_cnt": None, "match_idx": None, "match_h": match_h, "parent": None, "w": wg * z, "mu": (mu_g * z[:, None]).T,
            "cov": (cov_g[:, [0, 1, 2, 4, 5, 8]] * z[:, None]).T, "feat": feat_g * z[:, None]}
