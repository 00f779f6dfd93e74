"""The layer-potential work that a program has this library do, as cases that can be timed and compared.

A case is one pass through the public calls of ``paper_1801_04070_gb300``:

  eval   a density evaluated on a built geometry              Geometry.eval
  step   new targets on a geometry: set, build, evaluate      Geometry.set_targets, build, eval
  apply  one matvec of the exterior Neumann operator          Geometry.apply
  solve  an exterior Neumann solve                            Geometry.gmres
  batch  several geometries x several densities               Batch.eval
  order  features and predicted errors of every centre        Geometry.features, MLP.predict
  train  one epoch of the order-selection network             MLP.train, MLP.weights

Geometries are nx x ny grids (spacing 3) of starfish r = 1 + 0.25 cos(k theta) with random rotation, scale
and arm count, `panels` Gauss-Legendre panels of 16 density nodes and `nu` quadrature nodes each; densities
are random Fourier series per curve; targets are nodes on the curves ("base": the density nodes, "up": the
quadrature nodes) and `off` points uniform in the bounding box.
"""
import math

import numpy as np
import torch

from paper_1801_04070_gb300 import MLP, Batch, Geometry, params_default

NB = 16                     # density nodes per panel
PREC = {"fp64": 0, "mixed": 1, "mixed_fmm": 2}


def _grid(name, op, nx, ny, panels, kernel, q, p, off=0, on="base", prec="fp64", eps=0.0, nu=64, n_max=32, **more):
    return dict(name=name, op=op, nx=nx, ny=ny, panels=panels, kernel=kernel, q=q, p=p, off=off, on=on, prec=prec,
                eps=eps, nu=nu, n_max=n_max, **more)


def listed():
    return [
        # one small curve, its potential at its own nodes: what an interactive user or an outer iteration calls
        # over and over; a few hundred microseconds of launches
        _grid("curve-eval-S", "eval", 1, 1, 64, "S", 5, 10),
        # a few curves with new targets each time (plotting, a moving probe): the build counts as much as the
        # evaluation; odd panel and target counts
        _grid("curves-step-D", "step", 3, 1, 37, "D", 5, 10, off=4001),
        # the benchmark problem: 256 curves, 1.05 M quadrature nodes, 2.1 M targets on and off the curves
        _grid("grid-step-S", "step", 16, 16, 64, "S", 8, 15, off=1 << 20, on="up"),
        # the double layer (indirect Dirichlet problems) of a medium ragged array, on and off the curves
        _grid("grid-eval-D", "eval", 7, 5, 61, "D", 8, 15, off=60007, on="up"),
        # orders from a requested accuracy of 1e-10 in plain FP64 (p_qbx 7, p_fmm 30)
        _grid("grid-eval-S-1e-10", "eval", 13, 11, 64, "S", 7, 30, off=250000, on="up", eps=1e-10),
        # the mixed precision tiers: FP32 pairs with FP64 translations on the full array at 1e-6 ...
        _grid("grid-mixed-S-1e-6", "eval", 16, 16, 64, "S", 4, 19, off=1 << 20, on="up", prec="mixed", eps=1e-6),
        # ... and FP32 direct sums with paired translations on a ragged array at 1e-4
        _grid("grid-mixedfmm-D-1e-4", "eval", 12, 7, 50, "D", 2, 13, off=100003, on="up", prec="mixed_fmm", eps=1e-4),
        # one application of the exterior Neumann operator -mu/2 + S' mu, for a caller with its own solver
        _grid("operator-SP", "apply", 6, 5, 64, "SP", 8, 15),
        # a whole exterior Neumann solve to 1e-10 on four curves
        _grid("solve-neumann", "solve", 2, 2, 64, "SP", 8, 15),
        # independent geometries of uneven size with several densities each (parameter studies)
        _grid("batch-S", "batch", 0, 0, 0, "S", 8, 15, geoms=12, dens=8, largest=60000),
        # learned order selection: features of every centre and the network's predictions
        _grid("order-selection", "order", 8, 8, 64, "S", 4, 8),
        # training that network: an epoch of shuffled mini-batches on labelled centres
        dict(name="order-training", op="train", n=100000, batch=1024),
    ]


def draw(rng):
    op = rng.choice(["eval", "eval", "eval", "eval", "step", "step", "apply", "solve", "batch", "order", "train"])

    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if op == "train":
        return dict(op=op, n=log(5000, 100000), batch=rng.choice([512, 1000, 1024, 2048]))
    most = {"eval": 10000, "step": 16000, "apply": 4000, "solve": 400, "order": 4000}.get(op, 0)   # panels in all
    panels = rng.randint(16, 64)
    curves = max(1, log(16, max(17, most)) // panels) if most else 0
    nx = max(1, int(round(math.sqrt(curves) * rng.uniform(0.7, 1.4)))) if most else 0
    ny = max(1, curves // nx) if most else 0
    c = _grid(None, op, nx, ny, panels if most else 0, rng.choice(["S", "D"]), rng.choice([4, 5, 8]), rng.randint(8, 15),
              nu=rng.choice([32, 48, 64, 64]), n_max=rng.choice([24, 32, 32, 48]))
    del c["name"]
    if op in ("eval", "step"):
        c.update(off=log(300, 60 * nx * ny * panels), on=rng.choice(["base", "up"]))
        prec, eps = rng.choice([("fp64", 0.0), ("fp64", 1e-10), ("mixed", 1e-4), ("mixed", 1e-6), ("mixed", 1e-8),
                                ("mixed_fmm", 1e-4), ("mixed_fmm", 1e-6), ("mixed_fmm", 1e-8), ("mixed_fmm", 1e-10)])
        if eps:
            q, p = {1e-4: (2, 13), 1e-6: (4, 19), 1e-8: (5, 26), 1e-10: (7, 30)}[eps]
            c.update(prec=prec, eps=eps, q=q, p=p)
    elif op in ("apply", "solve"):
        c.update(kernel="SP", q=8, p=15)
        if op == "apply":
            c.update(q=rng.choice([5, 8]), kernel=rng.choice(["SP", "S", "D"]))
    elif op == "batch":
        c.update(geoms=rng.randint(3, 12), dens=rng.randint(2, 8), largest=log(10000, 60000), q=rng.choice([5, 8]), nu=64, n_max=32)
    elif op == "order":
        c.update(q=4, p=8, kernel="S")
    return c


# ------------------------------------------------------------------ inputs
def _curves(rng, nx, ny, panels, nu):
    """The discretised curves (what a program hands to Geometry) and their curve parameter per density node."""
    n = nx * ny
    arms = rng.integers(3, 9, n)[:, None, None]
    scale = rng.uniform(0.5, 1.0, n)[:, None, None]
    rot = rng.uniform(0.0, 2.0 * np.pi, n)[:, None, None]
    cx = 3.0 * (np.arange(n) % nx)[:, None, None]
    cy = 3.0 * (np.arange(n) // nx)[:, None, None]
    dth = 2.0 * np.pi / panels

    def nodes(ref):
        th = dth * np.arange(panels)[None, :, None] + (ref[None, None, :] + 1.0) * (0.5 * dth)
        r, dr = 1.0 + 0.25 * np.cos(arms * th), -0.25 * arms * np.sin(arms * th)
        c, s = np.cos(th + rot), np.sin(th + rot)
        x, y = cx + scale * r * c, cy + scale * r * s
        dx, dy = scale * (dr * c - r * s), scale * (dr * s + r * c)
        speed = np.hypot(dx, dy)
        return np.broadcast_to(th, x.shape), np.stack([x, y], -1).reshape(-1, 2), np.stack([dy / speed, -dx / speed], -1).reshape(-1, 2), speed
    ref_b, _ = np.polynomial.legendre.leggauss(NB)
    ref_u, w_u = np.polynomial.legendre.leggauss(nu)
    th, bxy, bn, _ = nodes(ref_b)
    _, uxy, un, speed = nodes(ref_u)
    w = w_u[None, None, :] * speed * (0.5 * dth)
    near = np.argmin(np.abs(ref_u[:, None] - ref_b[None, :]), axis=1)
    return dict(npanels=n * panels, nb=NB, nu=nu, ref_b=ref_b, ref_u=ref_u, base_xy=bxy, base_n=bn, up_xy=uxy, up_n=un,
                up_w=w.reshape(-1), panel_len=w.sum(-1).reshape(-1), theta=th.reshape(n, -1),
                up_base=(NB * np.arange(n * panels)[:, None] + near[None, :]).reshape(-1).astype(np.int32))


def _density(rng, g, count=1):
    """Random Fourier series of 10 modes per curve, N(0, 1) coefficients."""
    th = g["theta"]
    out = np.empty((count,) + th.shape)
    for j in range(count):
        a, b = rng.normal(0.0, 1.0, (2, th.shape[0], 10))
        out[j] = a[:, :1]
        for k in range(1, 10):
            out[j] += a[:, k:k + 1] * np.cos(k * th) + b[:, k:k + 1] * np.sin(k * th)
    return out.reshape(count, -1)


def _targets(rng, g, off, on):
    lo, hi = g["up_xy"].min(0), g["up_xy"].max(0)
    xy = [rng.uniform(lo, hi, (off, 2)), g["base_xy"] if on == "base" else g["up_xy"]]
    node = [np.full(off, -1, np.int32), np.arange(len(g["base_xy"]), dtype=np.int32) if on == "base" else g["up_base"]]
    return np.concatenate(xy), np.concatenate(node)


def _params(case):
    return params_default(p_qbx=case["q"], p_fmm=case["p"], n_max=case["n_max"], precision=PREC[case["prec"]],
                          **({"eps": case["eps"]} if case["eps"] else {}))


def _batch_sizes(case, rng):
    """(nx, ny, panels) per geometry: 2,000 to `largest` quadrature nodes, log-uniform."""
    sizes = []
    for _ in range(case["geoms"]):
        ns = float(np.exp(rng.uniform(np.log(2000), np.log(case["largest"]))))
        curves = max(1, int(ns / 4096))
        nx = int(np.sqrt(curves))
        sizes.append((nx, curves // nx, 64 if curves > 1 else max(8, min(64, int(ns / 64)))))
    return sizes


def _inputs(case, seed):
    """Everything made from the seed, as host arrays."""
    rng = np.random.default_rng(seed)
    if case["op"] == "train":
        X = rng.normal(0.0, 1.0, (case["n"], 32)).astype(np.float32)
        M = rng.normal(0.0, 0.3, (32, 2))
        Y = (np.tanh(X @ M) * 2.0 - 6.0 + rng.normal(0.0, 0.3, (case["n"], 2))).astype(np.float32)
        return dict(X=X, Y=Y)
    if case["op"] == "batch":
        items = []
        for nx, ny, panels in _batch_sizes(case, np.random.default_rng(case["geoms"])):
            g = _curves(rng, nx, ny, panels, case["nu"])
            items.append((g, _density(rng, g, case["dens"]), *_targets(rng, g, len(g["base_xy"]), "base")))
        return dict(items=items)
    g = _curves(rng, case["nx"], case["ny"], case["panels"], case["nu"])
    d = dict(g=g, density=_density(rng, g)[0])
    d["xy"], d["node"] = _targets(rng, g, case["off"], case["on"])
    if case["op"] == "solve":    # boundary data: normal derivative of Re 1/(z - z0), z0 inside the first curve
        x, n = (g[k][:, 0] + 1j * g[k][:, 1] for k in ("base_xy", "base_n"))
        z0 = x[:g["theta"].shape[1]].mean() + 0.05 * complex(*rng.uniform(-1.0, 1.0, 2))
        d["rhs"] = np.ascontiguousarray((n * (-1.0 / (x - z0) ** 2)).real)
    return d


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def prepare(case, seed):
    op, d = case["op"], _inputs(case, seed)
    if op == "train":
        owner = Geometry(_curves(np.random.default_rng(seed), 1, 1, 16, 64))
        m = MLP(owner, seed=seed & 0xffff)
        return dict(op=op, owner=owner, mlp=m, w0=m.weights(), batch=case["batch"], **d)
    if op == "batch":
        geos, dens, outs = [], [], []
        for g, mu, xy, node in d["items"]:
            geo = Geometry(g, _params(case))
            geo.set_targets(xy, node)
            geos.append(geo.build())
            dens.append(_cuda(mu))
            outs.append(torch.zeros(len(mu), len(node), dtype=torch.float64, device="cuda"))
        return dict(op=op, kernel=case["kernel"], geos=geos, batch=Batch(geos), dens=dens, outs=outs)
    geo = Geometry(d["g"], _params(case))
    s = dict(op=op, kernel=case["kernel"], geo=geo, mu=_cuda(d["density"]), xy=_cuda(d["xy"]), node=_cuda(d["node"]))
    if op != "step":
        geo.set_targets(s["xy"], s["node"])
        geo.build()
    if op == "order":
        s["mlp"] = MLP(geo, seed=7)
    elif op == "solve":
        s["rhs"] = _cuda(d["rhs"])
    s["out"] = torch.zeros(len(d["node"]) if op in ("eval", "step") else len(d["density"]), dtype=torch.float64, device="cuda")
    return s


def run(s):
    op = s["op"]
    if op == "eval":
        return s["geo"].eval(s["kernel"], s["mu"], s["out"])
    if op == "step":
        s["geo"].set_targets(s["xy"], s["node"])
        s["geo"].build()
        return s["geo"].eval(s["kernel"], s["mu"], s["out"])
    if op == "apply":
        return s["geo"].apply(s["kernel"], s["mu"], s["out"], identity=-0.5)
    if op == "solve":
        mu, iters, _ = s["geo"].gmres(s["rhs"], tol=1e-10, maxit=200, restart=30, mu=s["out"])
        return mu, iters
    if op == "batch":
        return s["batch"].eval(s["kernel"], s["dens"], s["outs"])
    if op == "order":
        f = s["geo"].features()
        return f, s["mlp"].predict(f)
    s["mlp"].weights(set=s["w0"])
    s["mlp"].train(s["X"], s["Y"], epochs=1, batch=s["batch"], lr=1e-3, seed=0)
    return s["mlp"].weights()


# ------------------------------------------------------------------ what a pass cannot do without
def _eval_work(case, nsrc, nbase, off, on, density):
    """Interaction counts per centre, target and box as measured on the 16 x 16 array (272 direct sources and 7
    List 3 far boxes per centre, 60 direct sources per point target, 12 particles and 9 List 2 boxes per box)."""
    q, p, nc = case["q"], case["p"], 2 * nbase
    pts = int(0.85 * off)
    flops = nc * min(nsrc, 8.5 * case["n_max"]) * (14 * q + 20) + pts * min(nsrc, 60) * 17
    flops += (nsrc + nc + pts) / 12 * 9 * 8 * (p + 1) ** 2 + 7 * nc * 8 * (p + 1) * (q + 1)
    return flops * density, nsrc * 40 + nbase * 24 + (off + on) * 20 + density * (nbase * 8 + (off + on) * 8)


def work(case):
    if case["op"] == "train":
        # forward, backward for inputs and weights: three products of 5,184 weights per sample
        return {"bytes": case["n"] * 34 * 4, "flops": case["n"] * 3 * 2 * 5184}
    if case["op"] == "batch":
        f = b = 0
        for nx, ny, panels in _batch_sizes(case, np.random.default_rng(case["geoms"])):
            nb = nx * ny * panels * NB
            df, db = _eval_work(case, nx * ny * panels * case["nu"], nb, nb, nb, case["dens"])
            f, b = f + df, b + db
        return {"bytes": int(b), "flops": int(f)}
    n = case["nx"] * case["ny"] * case["panels"]
    if case["op"] == "order":   # the network per centre, and the distances to its direct sources
        return {"bytes": n * (case["nu"] * 16 + NB * 40 + 2 * NB * 34 * 4), "flops": n * 2 * NB * (2 * 5184 + 272 * 5)}
    on = n * (NB if case["on"] == "base" else case["nu"])
    f, b = _eval_work(case, n * case["nu"], n * NB, case["off"], on, 1)
    if case["op"] == "solve":
        f *= 15                 # matvecs of a solve
    return {"bytes": int(b), "flops": int(f)}


# ------------------------------------------------------------------ the same values in 64 bits
def _cplx(a):
    a = torch.as_tensor(a, dtype=torch.float64, device="cuda")
    return torch.complex(a[..., 0].contiguous(), a[..., 1].contiguous())


def _upsample(g, mu):
    rb, ru = g["ref_b"], g["ref_u"]
    L = np.array([[np.prod([(x - rb[k]) / (rb[j] - rb[k]) for k in range(NB) if k != j]) for j in range(NB)] for x in ru])
    return mu.reshape(-1, NB) @ torch.as_tensor(L.T, device="cuda"), L


def _centres(g):
    t, n = _cplx(g["base_xy"]), _cplx(g["base_n"])
    r = torch.as_tensor(0.5 * g["panel_len"], device="cuda").repeat_interleave(NB)
    return torch.stack([t - r * n, t + r * n], 1).reshape(-1), r.repeat_interleave(2)


def _blocks(n, width):
    step = max(1, int(4e7 / max(1, width)))
    return [(i, min(n, i + step)) for i in range(0, n, step)]


def _direct(g, kernel, q, mu, xy, node):
    """QBX of order q without acceleration: each centre's expansion summed over every source, each target
    evaluated from its centre (two-sided mean on the curve), other targets by direct summation."""
    qs = _upsample(g, mu)[0].reshape(-1) * torch.as_tensor(g["up_w"], device="cuda")
    y, c, r = _cplx(g["up_xy"]), *_centres(g)
    st = qs * _cplx(g["up_n"]) if kernel == "D" else qs.to(torch.complex128)
    # expansions scaled by the radius: beta_m r^m
    beta = torch.zeros(len(c), q + 1, dtype=torch.complex128, device="cuda")
    for i, j in _blocks(len(c), len(y)):
        w = y[None, :] - c[i:j, None]
        if kernel == "D":
            t = 1.0 / w
            u = t * r[i:j, None]
            for m in range(q + 1):
                beta[i:j, m] = t @ st
                t *= u
        else:
            beta[i:j, 0] = (w.abs().log() @ qs).to(torch.complex128)
            u = r[i:j, None] / w
            t = u.clone()
            for m in range(1, q + 1):
                beta[i:j, m] = -(t @ st) / m
                t *= u

    def at(ci, x, normal=None):
        z = (x - c[ci]) / r[ci]
        v = torch.zeros_like(z)
        if normal is None:
            for m in range(q, -1, -1):
                v = v * z + beta[ci, m]
        else:
            for m in range(q, 0, -1):
                v = v * z + m * beta[ci, m]
            v = v * normal / r[ci]
        return v.real
    x, node = _cplx(xy), torch.as_tensor(node, device="cuda").long()
    out = torch.zeros(len(x), dtype=torch.float64, device="cuda")
    on = node >= 0
    nd = node[on]
    nrm = _cplx(g["base_n"])[nd] if kernel == "SP" else None
    out[on] = 0.5 * (at(2 * nd, x[on], nrm) + at(2 * nd + 1, x[on], nrm))
    off = torch.nonzero(~on)[:, 0]
    for i, j in _blocks(len(off), max(len(c), len(y))):
        k = off[i:j]
        d = (x[k, None] - c[None, :]).abs() / r[None, :]
        best, ci = d.min(1)
        w = y[None, :] - x[k, None]
        far = (1.0 / w @ st).real if kernel == "D" else w.abs().log() @ qs
        out[k] = torch.where(best <= 1.2, at(ci, x[k]), far)
    return out / (-2.0 * math.pi)


def _neumann_matrix(g, q):
    """-1/2 + S' at the density nodes as a dense matrix."""
    y, c, r = _cplx(g["up_xy"]), *_centres(g)
    x, n = _cplx(g["base_xy"]), _cplx(g["base_n"])
    w = torch.as_tensor(g["up_w"], device="cuda")
    L = torch.as_tensor(_upsample(g, torch.zeros(NB, dtype=torch.float64, device="cuda"))[1], device="cuda")
    A = torch.zeros(len(x), len(x), dtype=torch.float64, device="cuda")
    for i, j in _blocks(len(x), len(y)):
        K = torch.zeros(j - i, len(y), dtype=torch.float64, device="cuda")
        for side in (0, 1):
            ci = 2 * torch.arange(i, j, device="cuda") + side
            inv = 1.0 / (y[None, :] - c[ci, None])
            u = (x[i:j] - c[ci])[:, None] * inv
            v = torch.ones_like(u)
            for _ in range(q - 1):
                v = v * u + 1.0
            K += 0.5 / (2.0 * math.pi) * (n[i:j, None] * inv * v).real
        K *= w[None, :]
        A[i:j] = (K.reshape(j - i, -1, g["nu"]) @ L).reshape(j - i, -1)
    A.diagonal().sub_(0.5)
    return A


def exact(case, seed):
    op = case["op"]
    if op in ("train", "order"):
        return None       # shuffled FP32 training; features depend on the tree, predictions are BF16 by design
    if op != "batch":
        n = case["nx"] * case["ny"] * case["panels"]
        if n * n * case["nu"] * (2 * NB + 2 * case["off"] / n) > 6e10 or (op == "solve" and n * NB > 8200):
            return None   # the direct sums would take too long
    d = _inputs(case, seed)
    if op == "batch":
        return [torch.stack([_direct(g, case["kernel"], case["q"], _cuda(m), xy, node) for m in mu])
                if len(g["up_w"]) <= 10000 else None for g, mu, xy, node in d["items"]]
    g, mu = d["g"], _cuda(d["density"])
    if op == "apply":
        return _direct(g, case["kernel"], case["q"], mu, g["base_xy"], np.arange(len(mu))) - 0.5 * mu
    if op == "solve":
        return torch.linalg.solve(_neumann_matrix(g, case["q"]), _cuda(d["rhs"])), None
    return _direct(g, case["kernel"], case["q"], mu, d["xy"], d["node"])
