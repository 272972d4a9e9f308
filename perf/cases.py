"""What is measured of this framework: frames rendered, mixtures fitted and the single layers of
both (the cull, the evaluation with its gradients), through the package's public entry points.

A case is a dict of plain values; `kind` says which path it takes:

  render       one frame, cull and forward (`render.Frame.render`)
  conditioned  one frame whose inputs beyond position are constant (Section 3.2): the conditioned
               cull and the forward
  batch        several frames of uneven N and size in one launch (`render.render_batch`)
  fit          one step of a fit (`train.Trainer.step`): cull, forward, loss, backward, Adam
  eval         differentiable evaluation on given candidate lists (`train.evaluate`), forward and
               backward
  cull         the candidate lists alone (`ndg.build_cull`)

Inputs follow the recipes of `synth` (drawn on the GPU): precision factors with a diagonal
log-uniform in [2, 20], weights U[0, 1]^3, queries that are Morton-ordered points of the box
("box"), grids on random planes ("planes") or the pixels of one frame.
"""
import math

import torch

from paper_2405_20067_gb300 import ndg, render, train

CUTOFF = 1.0 / 255.0
PARENT = ["mean", "theta", "alpha_raw", "color_raw"]
CHILD = ["u_theta", "m_u", "c_alpha_raw", "c_color_raw"]
MODES = {"fp32": ndg.NDG_MODE_FP32, "tc": ndg.NDG_MODE_TC, "auto": ndg.NDG_MODE_AUTO}


def listed():
    return [
        # the smallest frame of a batched render (256 x 256, 10,000 Gaussians): latency and launches
        dict(name="render n6 256x256", kind="render", N=6, G=10_000, W=256, H=256, form="tc", tile=256),
        # an ordinary frame of odd size (ragged last row and column of tiles), the form picked per tile
        dict(name="render n8 701x397", kind="render", N=8, G=60_000, W=701, H=397, form="auto", tile=256),
        # a preview frame of the render benchmark's dimension
        dict(name="render n10 480x272", kind="render", N=10, G=100_000, W=480, H=272, form="tc", tile=256),
        # the render benchmark: one full-HD frame of 500,000 10-D Gaussians
        dict(name="render n10 1080p", kind="render", N=10, G=500_000, W=1920, H=1080, form="tc", tile=256),
        # the same mixture and frame with the inputs beyond position constant: short lists, the cull decides
        dict(name="conditioned n10 1080p", kind="conditioned", N=10, G=500_000, W=1920, H=1080, form="auto", tile=256),
        # frames of N = 6, 8, 10 in one persistent launch
        dict(name="batch of 6 frames", kind="batch", G=30_000, W=320, H=240, frames=6),
        # the fit benchmark: 100,000 parents with live children, 2^20 queries
        dict(name="fit n6 100k", kind="fit", N=6, G=100_000, Q=1 << 20, queries="box", children=True, k=16, form="tc", loss="l2"),
        # the 10-D fit: 50,000 parents with children, a minibatch of 2^18 surface queries, relative L2
        dict(name="fit n10 50k", kind="fit", N=10, G=50_000, Q=1 << 18, queries="planes", children=True, k=16, form="tc", loss="rel_l2"),
        # the smallest fit: 1,000 Gaussians, 16,384 queries, no cull, the default FP32 forms
        dict(name="fit n6 1k dense", kind="fit", N=6, G=1_000, Q=16_384, queries="box", children=False, k=0, form="fp32", loss="l2"),
        # evaluation and gradients in the default FP32 forms (the culling ablation's size)
        dict(name="eval n6 20k fp32", kind="eval", N=6, G=20_000, Q=1 << 18, queries="box", children=False, k=16, form="fp32", tile=256),
        # evaluation and gradients on the tensor cores, children, a ragged last tile, tiles of 200
        dict(name="eval n8 5k tc", kind="eval", N=8, G=5_000, Q=30_011, queries="box", children=True, k=16, form="tc", tile=200),
        # the fit benchmark's candidate lists alone
        dict(name="cull n6 100k", kind="cull", N=6, G=100_000, Q=1 << 20, queries="box", children=True, k=16, tile=256),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["render", "render", "fit", "fit", "eval", "eval", "conditioned", "batch", "cull"])
    t = rng.random()  # one exponent for both sides of a frame, as the batched render's recipe has it
    W, H = round(256 * (1920 / 256) ** t), round(256 * (1080 / 256) ** t)
    while True:
        if kind == "render":
            tile = rng.choice([256, 256, 128])
            c = dict(kind=kind, N=rng.choice([6, 8, 10]), G=_log(rng, 10_000, 500_000), W=W, H=H,
                     form=rng.choice(["tc", "auto"]), tile=tile)
        elif kind == "conditioned":
            c = dict(kind=kind, N=rng.choice([6, 8, 10]), G=_log(rng, 10_000, 500_000), W=W, H=H,
                     form=rng.choice(["tc", "auto", "fp32"]), tile=256)
        elif kind == "batch":
            c = dict(kind=kind, G=_log(rng, 10_000, 60_000), W=min(W, 640), H=min(H, 400), frames=rng.randint(3, 8))
        elif kind == "fit":
            N = rng.choice([6, 10])
            form = rng.choice(["tc", "tc", "fp32"])
            c = dict(kind=kind, N=N, G=_log(rng, 1_000, 100_000 if N == 6 else 50_000), Q=0,
                     queries="box" if N == 6 else "planes", children=rng.random() < 0.7, k=16, form=form,
                     loss=rng.choice(["l2", "rel_l2"]))
            c["Q"] = _log(rng, 1 << 14, (1 << 20 if N == 6 else 1 << 18) >> (2 if form == "fp32" else 0))
        elif kind == "eval":
            form = rng.choice(["tc", "tc", "fp32"])
            c = dict(kind=kind, N=rng.choice([3, 5, 6, 7, 8, 10, 12]), G=_log(rng, 1_000, 20_000),
                     Q=_log(rng, 4_000, 1 << 16), queries="box", children=rng.random() < 0.5,
                     k=rng.choice([8, 16]), form=form, tile=rng.choice([256, 256, 200, 128]))
        else:
            c = dict(kind=kind, N=rng.choice([6, 10]), G=_log(rng, 10_000, 100_000), Q=_log(rng, 1 << 16, 1 << 20),
                     queries="box", children=rng.random() < 0.5, k=16, tile=256)
        if work(c)["flops"] <= 0.5 * work(listed()[3])["flops"]:
            return c


# ---- inputs ----------------------------------------------------------------------------------


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _uniform(g, *shape, lo=-1.0, hi=1.0, dtype=torch.float32):
    return torch.rand(*shape, generator=g, device="cuda", dtype=dtype) * (hi - lo) + lo


def _tril(A):
    r, c = torch.tril_indices(A.shape[-1], A.shape[-1], device=A.device)
    return A[..., r, c]


def _parents(N, G, g):
    f8 = dict(device="cuda", dtype=torch.float64)
    M = torch.tril(0.5 * torch.randn(G, N, N, generator=g, **f8), -1)
    d = torch.exp(_uniform(g, G, N, lo=math.log(2.0), hi=math.log(20.0), dtype=torch.float64))
    M = M + torch.diag_embed(d)
    L = torch.linalg.solve_triangular(M, torch.eye(N, **f8).expand(G, N, N), upper=False)
    off = torch.tril(L, -1).clamp(-0.99, 0.99)
    theta = torch.log((1 + off) / (1 - off)) + torch.diag_embed(torch.log(torch.diagonal(L, dim1=-2, dim2=-1)))
    w = _uniform(g, G, 3, lo=0.0)
    alpha = w.amax(1).clamp_min(1e-6)
    c = (w / alpha[:, None]).clamp(1e-4, 1 - 1e-4)
    return dict(mean=_uniform(g, G, N), theta=_tril(theta).float(), alpha_raw=alpha.log(),
                color_raw=torch.log(c / (1 - c)))


def _children(N, G, g):
    """The state after a refinement: children spanning their parents at brightness t / 10."""
    n = lambda s, *sh: s * torch.randn(*sh, generator=g, device="cuda")  # noqa: E731
    return dict(u_theta=n(0.05, G, N * (N + 1) // 2), m_u=n(0.05, G, N),
                c_alpha_raw=_uniform(g, G, lo=9e-4, hi=1.1e-3).log(), c_color_raw=n(1.0, G, 3))


def _mixture(N, G, g, children=False):
    return ndg.Mixture.from_arrays(N, _parents(N, G, g), _children(N, G, g) if children else None)


def _morton(x):
    N = x.shape[1]
    bits = max(1, 60 // N)
    q = ((x.double() + 1) * 0.5 * (1 << bits)).long().clamp(0, (1 << bits) - 1)
    code = torch.zeros(x.shape[0], dtype=torch.int64, device=x.device)
    for b in range(bits):
        for d in range(N):
            code |= ((q[:, d] >> b) & 1) << (b * N + d)
    return x[torch.argsort(code, stable=True)].contiguous()


def _tiled(W, H):
    """(row, col) of every pixel, 16 x 16 tiles row-major, pixels row-major inside a tile."""
    r, c = torch.meshgrid(torch.arange(H, device="cuda"), torch.arange(W, device="cuda"), indexing="ij")
    key = (((r // 16) * ((W + 15) // 16) + c // 16) * 16 + r % 16) * 16 + c % 16
    order = torch.argsort(key.reshape(-1))
    return r.reshape(-1)[order], c.reshape(-1)[order]


def _frame(N, W, H, g, constant=False):
    r, c = _tiled(W, H)
    pos = torch.stack([(c + 0.5) / W * 2 - 1, ((r + 0.5) / H * 2 - 1) * (H / W), torch.zeros_like(r)], 1)
    rest = _uniform(g, 1, N - 3).expand(W * H, N - 3) if constant else _uniform(g, W * H, N - 3)
    return torch.cat([pos.float(), rest], 1).contiguous()


def _planes(N, Q, g):
    """Grids of 128 x 128 on random planes, cut at Q queries."""
    n = -(-Q // (128 * 128))
    r, c = _tiled(128, 128)
    basis = torch.linalg.qr(torch.randn(n, 3, 3, generator=g, device="cuda")).Q
    s, t = (c + 0.5) / 128 - 0.5, (r + 0.5) / 128 - 0.5
    pos = _uniform(g, n, 1, 3) + s[None, :, None] * basis[:, None, :, 0] + t[None, :, None] * basis[:, None, :, 1]
    return torch.cat([pos.reshape(-1, 3), _uniform(g, n * 128 * 128, N - 3)], 1)[:Q].contiguous()


def _queries(case, g):
    N, Q = case["N"], case["Q"]
    return _planes(N, Q, g) if case["queries"] == "planes" else _morton(_uniform(g, Q, N))


def _params(N, k, g, children):
    if k == 0:
        return ndg.CullParams(0, None, 0.0, 3.0, 1)
    p = torch.randn(k, N, generator=g, device="cuda")
    return ndg.CullParams(k, (p / p.norm(dim=1, keepdim=True)).contiguous(), CUTOFF, 3.0, 64,
                          child_k_min=3.0 if children else 0.0)


def _one_frame(N, G, W, H, seed, constant=False):
    g = _gen(seed)
    return _mixture(N, G, g), _frame(N, W, H, g, constant), _params(N, 16, g, False)


def _batch_sizes(case):
    """Frames of uneven size: N = 6, 8, 10 in turn, each a little larger than the one before."""
    return [((6, 8, 10)[i % 3], case["G"] + 1_000 * i, case["W"] + 13 * i, case["H"] + 7 * i)
            for i in range(case["frames"])]


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "batch":
        st["frames"] = [render.Frame(*_one_frame(*s, seed * 16 + i)) for i, s in enumerate(_batch_sizes(case))]
        for f in st["frames"]:
            f.evaluator(256)
        st["batch_ws"] = ndg.batch_workspace(len(st["frames"]))
        return st
    if kind in ("render", "conditioned"):
        mix, x, cp = _one_frame(case["N"], case["G"], case["W"], case["H"], seed, kind == "conditioned")
        if kind == "render":
            st["frame"] = render.Frame(mix, x, cp)
            st["frame"].evaluator(case["tile"])  # the frame's buffers, sized once
        else:
            xc = x[0, 3:].contiguous()
            ev = ndg.Evaluator(mix, x, case["tile"], cp, backward=False)
            ev.build(mix, xc=xc)
            st.update(mix=mix, ev=ev, xc=xc, y=torch.empty(x.shape[0], 3, device="cuda"))
        return st
    g = _gen(seed)
    N = case["N"]
    mix = _mixture(N, case["G"], g, case["children"])
    x = _queries(case, g)
    cp = _params(N, case["k"], g, case["children"])
    if kind == "fit":
        target = _uniform(g, x.shape[0], 3, lo=0.0)
        m = MODES[case["form"]]
        st["trainer"] = train.Trainer(mix, x, target, 256, cp, lr=1e-3, phase=0, mode=m, bwd_mode=m, loss=case["loss"])
        return st
    # the lists alone: a buffer that any lists of these sizes fit, so that it does not depend on the inputs
    E_cap = -(-x.shape[0] // case["tile"]) * mix.Ge if kind == "cull" else None
    ev = ndg.Evaluator(mix, x, case["tile"], cp, E_cap=E_cap, backward=kind == "eval")
    ev.build(mix)
    st.update(mix=mix, ev=ev)
    if kind == "eval":
        ev.mode = ev.bwd_mode = MODES[case["form"]]
        for p in mix.tensors():
            p.requires_grad_(True)
        st["dy"] = torch.randn(x.shape[0], 3, generator=g, device="cuda") / (3 * x.shape[0])
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "render":
        f = state["frame"]
        y = f.render((case["form"], case["tile"]))
        cull = f.evaluator(case["tile"]).cull
        return dict(y=y, offsets=cull.offsets, entries=cull.E_dev)
    if kind == "conditioned":
        mix, ev, y = state["mix"], state["ev"], state["y"]
        ndg.build_cull_conditioned(mix, ev.x, ev.tile, ev.cp, state["xc"], ev.cull, ev.ws)
        ndg.forward(mix, ev.x, ev.tile, ev.cull, y, ev.ws, mode=MODES[case["form"]] | ndg.NDG_RECORDS_READY)
        return dict(y=y, offsets=ev.cull.offsets, ids=ev.cull.ids)
    if kind == "batch":
        render.render_batch(state["frames"], state["batch_ws"])
        return [f.y for f in state["frames"]]
    if kind == "cull":
        mix, ev = state["mix"], state["ev"]
        ndg.build_cull(mix, ev.x, ev.tile, ev.cp, ev.cull, ev.ws)
        return dict(offsets=ev.cull.offsets, ids=ev.cull.ids, entries=ev.cull.E_dev)
    names = PARENT + (CHILD if case["children"] else [])
    if kind == "fit":
        tr = state["trainer"]
        loss = tr.step()
        out = dict(loss=loss.float())
        for n in names:
            out[n] = getattr(tr.mix, n).detach()
            out["m1 " + n] = getattr(tr.m1, n)  # the gradients' first moments
        return out
    mix, ev = state["mix"], state["ev"]
    for p in mix.tensors():
        p.grad = None
    y = train.evaluate(ev, mix)
    y.backward(state["dy"])
    out = {n: getattr(mix, n).grad for n in names}
    out["y"] = y.detach()
    return out


# ---- what a pass cannot do without ----------------------------------------------------------------

#: share of the Gaussians in a tile's list, as these recipes come out: by N for frames and planes
#: (their free inputs span the box), 0.3 for Morton-ordered points of the box
SHARE = {6: 0.7, 8: 0.83, 10: 0.95}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        ws = [work(dict(kind="render", N=n, G=G, W=W, H=H, form="tc", tile=256)) for n, G, W, H in _batch_sizes(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    N, G = case["N"], case["G"]
    P = N * (N + 1) // 2
    Q = case["Q"] if "Q" in case else case["W"] * case["H"]
    ge = G * (2 if case.get("children") else 1)
    params = 4 * ge * (P + N + 4)
    # a pair's evaluation on the centred form; its gradients; a projection of a Gaussian and of a query
    fwd, bwd, proj = N * N + 4 * N + 7, 2 * N * N + 7 * N + 13, N * N + 3 * N
    k = case.get("k", 16)
    share = (0.3 if case.get("queries") == "box" else SHARE[N]) if k else 1.0
    tiles = -(-Q // case.get("tile", 256))
    cull = 2 * k * (ge * proj + Q * N)
    if kind == "conditioned":
        return dict(bytes=params + 4 * Q * (N + 3), flops=cull)
    pairs = Q * ge * share
    if kind == "cull":
        return dict(bytes=params + 4 * Q * N + 4 * tiles * ge * share, flops=cull)
    if kind == "render":
        return dict(bytes=params + 4 * Q * (N + 3), flops=cull + pairs * fwd)
    if kind == "eval":
        return dict(bytes=2 * params + 4 * Q * (N + 6), flops=pairs * (fwd + bwd))
    return dict(bytes=6 * params + 4 * Q * (N + 6), flops=cull + pairs * (fwd + bwd))


# ---- the same in 64 bits ----------------------------------------------------------------------------


def _lower(th, N):
    r, c = torch.tril_indices(N, N, device=th.device)
    L = torch.zeros(th.shape[0], N, N, dtype=th.dtype, device=th.device)
    return L.index_put((torch.arange(th.shape[0], device=th.device)[:, None], r, c),
                       torch.where(r == c, torch.exp(th), 2 * torch.sigmoid(th) - 1))


def _activated(raw, N):
    """L, m, w of every evaluated Gaussian (Eq. 2, 6-8)."""
    L, m = _lower(raw["theta"], N), raw["mean"]
    w = torch.exp(raw["alpha_raw"])[:, None] * torch.sigmoid(raw["color_raw"])
    if "u_theta" in raw:
        Lc, mc = L @ _lower(raw["u_theta"], N), (L @ raw["m_u"][:, :, None])[:, :, 0] + m
        wc = torch.exp(raw["c_alpha_raw"])[:, None] * torch.sigmoid(raw["c_color_raw"])
        L, m, w = torch.cat([L, Lc]), torch.cat([m, mc]), torch.cat([w, wc])
    return L, m, w


def _chain(a, b):
    """sum_d a[..., d] b[..., d] as a chain of FP32 fused multiply-adds."""
    acc = torch.zeros(torch.broadcast_shapes(a.shape[:-1], b.shape[:-1]), device=a.device)
    for d in range(a.shape[-1]):
        acc = (a[..., d].double() * b[..., d].double() + acc.double()).float()
    return acc


def _kept(L, m, w, x, tile, cp, parents):
    """[T, Ge] candidates by the FP32 bucket contract of the cull (Section 3.2)."""
    T, Ge = -(-x.shape[0] // tile), L.shape[0]
    if cp.k == 0:
        return torch.ones(T, Ge, dtype=torch.bool, device=x.device)
    L, m, w = L.float(), m.float(), w.float()
    B, at = cp.buckets, torch.arange(x.shape[0], device=x.device) // tile
    wm = w.amax(1).double()
    kg = torch.where(wm > CUTOFF_F, torch.sqrt(2 * torch.log(wm / CUTOFF_F)), torch.full_like(wm, -1.0)).float()
    if cp.child_k_min > 0:
        kg[parents:] = kg[parents:].clamp_min(cp.child_k_min)
    keep = (kg > 0)[None, :].expand(T, Ge).clone()
    for r in cp.proj:
        q = _chain(x, r[None])
        lo_t = torch.full((T,), math.inf, device=x.device).scatter_reduce(0, at, q, "amin")
        hi_t = torch.full((T,), -math.inf, device=x.device).scatter_reduce(0, at, q, "amax")
        lo, hi = lo_t.min(), hi_t.max()
        inv = torch.where(hi - lo > 1e-3 * (1 + torch.maximum(lo.abs(), hi.abs())), torch.tensor(float(B), device=x.device) / (hi - lo), torch.zeros((), device=x.device))
        bucket = lambda v: torch.floor((v - lo) * inv).clamp(-2, B + 1)  # noqa: E731
        s2 = torch.zeros(Ge, device=x.device)
        for c in range(L.shape[1]):
            tc = _chain(L[:, c:, c], r[None, c:])
            s2 = (tc.double() * tc.double() + s2.double()).float()
        ks, mr = kg * torch.sqrt(s2), _chain(m, r[None])
        g0, g1 = bucket(mr - ks) - 1, bucket(mr + ks) + 1
        keep &= ((g1 >= 0) & (g0 <= B - 1))[None]
        t0, t1 = bucket(lo_t).clamp(0, B - 1), bucket(hi_t).clamp(0, B - 1)
        keep &= (g0[None] <= t1[:, None]) & (t0[:, None] <= g1[None])
    return keep


CUTOFF_F = float(torch.tensor(CUTOFF, dtype=torch.float32))


def _evaluate(raw, N, x, tile, cp, parents, dy=None):
    """y at every query and, for a given dl/dy (a function of y and the query range), the raw gradients."""
    leaf = {n: p.double().requires_grad_(dy is not None) for n, p in raw.items()}
    L, m, w = _activated(leaf, N)
    eye = torch.eye(N, dtype=torch.float64, device=x.device)
    M = torch.linalg.solve_triangular(L, eye.expand_as(L), upper=False)
    kept = _kept(L.detach(), m.detach(), w.detach(), x, tile, cp, parents)
    part = [p.detach().requires_grad_(dy is not None) for p in (M, m, w)]
    y = torch.zeros(x.shape[0], 3, dtype=torch.float64, device=x.device)
    for t in range(kept.shape[0]):
        q = slice(t * tile, min(x.shape[0], (t + 1) * tile))
        ids = kept[t].nonzero()[:, 0]
        Mt, mt, wt = (p[ids] for p in part)
        z = torch.einsum("cij,cqj->cqi", Mt, x[q].double()[None] - mt[:, None])
        yt = torch.einsum("cq,cr->qr", torch.exp(-0.5 * z.square().sum(-1)), wt)
        y[q] = yt.detach()
        if dy is not None:
            yt.backward(dy(yt.detach(), q))
    if dy is None:
        return y, None
    torch.autograd.backward([M, m, w], [p.grad for p in part])
    return y, {n: p.grad for n, p in leaf.items()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for i, s in enumerate(_batch_sizes(case)):
            mix, x, cp = _one_frame(*s, seed * 16 + i)
            big = s[1] * s[2] * s[3] > 4e9
            out.append(None if big else _evaluate({n: getattr(mix, n) for n in PARENT}, s[0], x, 256, cp, mix.G)[0])
        return out if any(y is not None for y in out) else None
    if kind in ("conditioned", "cull"):
        return None  # whole numbers; and lists whose exact rounding is the contract's own
    N, G = case["N"], case["G"]
    Q = case["Q"] if "Q" in case else case["W"] * case["H"]
    pairs = Q * G * (2 if case.get("children") else 1)
    if pairs > (2e10 if kind == "render" else 6e9):
        return None
    if kind == "render":
        mix, x, cp = _one_frame(N, G, case["W"], case["H"], seed)
        y, _ = _evaluate({n: getattr(mix, n) for n in PARENT}, N, x, case["tile"], cp, G)
        return dict(y=y, offsets=None, entries=None)
    g = _gen(seed)
    names = PARENT + (CHILD if case["children"] else [])
    mix = _mixture(N, G, g, case["children"])
    x = _queries(case, g)
    cp = _params(N, case["k"], g, case["children"])
    raw = {n: getattr(mix, n) for n in names}
    if kind == "eval":
        up = torch.randn(x.shape[0], 3, generator=g, device="cuda") / (3 * x.shape[0])
        y, grad = _evaluate(raw, N, x, case["tile"], cp, G, lambda _, q: up[q].double())
        return dict(grad, y=y)
    target = _uniform(g, x.shape[0], 3, lo=0.0).double()
    n = 3 * x.shape[0]
    den = lambda y: y.square() + 1e-2 if case["loss"] == "rel_l2" else 1.0  # noqa: E731
    y, grad = _evaluate(raw, N, x, 256, cp, G, lambda v, q: 2 * (v - target[q]) / den(v) / n)
    out = {"loss": ((y - target).square() / den(y)).sum().reshape(1) / n}
    for k in names:
        out[k] = None  # a first step of Adam is the gradient's sign
        out["m1 " + k] = 0.1 * grad[k]
    return out
