"""The calls whose speed is measured: what users of this framework have it do, through its
public entry points (``pm.Mesh``, ``pm.Batch``, ``autograd.quality``), from the smallest mesh
to the largest workload of the benchmark.

A case is a dict of plain values.  ``kind`` says which path it takes:

  adapt    one mesh: create, set the metric, adapt (Algorithm 1, smoothing), read the mesh back
  batch    the batch recipe: many grids of log-uniform sizes, each with its own constant
           anisotropic metric, in one batch handle
  readapt  one time step of the time-dependent psi benchmark: the mesh adapted to psi at t = 0
           is adapted to psi one step of 50 later
  opt      optimisation-based smoothing rounds on an adapted mesh
  grad     the quality functional and its gradient (forward and backward) on an adapted mesh

Inputs are made on the GPU: jittered grids, the psi-Hessian metric (sizes clamped, the scale
bisected for an element count), uniform and constant anisotropic metrics.  The jitter and the
priorities' seed come from ``seed``, so inputs of another seed are another mesh of the same size.
"""
import math

import numpy as np
import torch

from paper_1505_04694_gb300 import inputs, pm
from paper_1505_04694_gb300.autograd import quality

PERIOD = 50  # time steps per period of psi(x, y, t)


def listed():
    return [
        # the smallest call: a 41 x 41 grid under a uniform metric (latency: launches, round trips)
        dict(name="adapt_uniform_41", kind="adapt", n=41, metric="uniform", elements=5773.5,
             memory="device", select=0),
        # the paper's own benchmark size: about 200 x 200, a requirement of 550k elements
        dict(name="adapt_psi_201", kind="adapt", n=201, metric="psi", elements=5.5e5,
             memory="device", select=0),
        # the 2M anisotropic workload: mostly refinement, large rounds
        dict(name="adapt_psi_257", kind="adapt", n=257, metric="psi", elements=2.0e6,
             memory="device", select=0),
        # the largest single mesh: about 20M triangles
        dict(name="adapt_psi_1025", kind="adapt", n=1025, metric="psi", elements=1.36e7,
             memory="device", select=0),
        # a fine grid coarsened to a constant anisotropic metric, from and to host arrays
        dict(name="coarsen_host_317", kind="adapt", n=317, metric="aniso", elements=8.0e3,
             memory="host", select=0),
        # independent sets from a colouring of the vertex graph (the paper's own scheme)
        dict(name="adapt_colour_129", kind="adapt", n=129, metric="psi", elements=5.0e4,
             memory="device", select=1),
        # a few small meshes in one handle
        dict(name="batch_16_small", kind="batch", count=16, tmin=200.0, tmax=3.0e3, recipe=9),
        # the headline workload: 512 meshes of 1k to 200k triangles
        dict(name="batch_512", kind="batch", count=512, tmin=1.0e3, tmax=2.0e5, recipe=5),
        # one time step: a mesh that nearly fits its new metric
        dict(name="readapt_psi_201", kind="readapt", n=201, elements=5.5e5),
        # the optimisation-based smoother, 20 rounds
        dict(name="opt_smooth_129", kind="opt", n=129, elements=2.0e5, rounds=20),
        # forward and backward of the quality functional: a mesh inside an optimisation loop
        dict(name="grad_41", kind="grad", n=41, metric="uniform", elements=5773.5),
        # and on the adapted 2M mesh
        dict(name="grad_257", kind="grad", n=257, metric="psi", elements=2.0e6),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["adapt", "adapt", "adapt", "batch", "batch", "readapt", "opt", "grad"])
    if kind == "batch":
        count = int(round(_log_uniform(rng, 2, 256)))
        tmin = _log_uniform(rng, 200, 4000)
        return dict(kind=kind, count=count, tmin=tmin, tmax=tmin * rng.uniform(4, 50),
                    recipe=rng.randrange(6, 1000))
    # the benchmark's own workloads refine 7 to 15 times and coarsen up to 25 times
    top = {"adapt": 900, "readapt": 400, "opt": 300, "grad": 400}[kind]
    n = int(round(_log_uniform(rng, 17, top)))
    elements = min(2.0 * (n - 1) ** 2 * _log_uniform(rng, 0.5, 14), 1.0e7)
    if kind == "readapt":
        return dict(kind=kind, n=n, elements=elements)
    if kind == "opt":
        return dict(kind=kind, n=n, elements=elements, rounds=rng.randint(1, 20))
    metric = rng.choice(["uniform", "psi", "psi"])
    if kind == "grad":
        return dict(kind=kind, n=n, metric=metric, elements=elements)
    if rng.random() < 0.3:
        metric = "aniso"
        elements = 2.0 * (n - 1) ** 2 * _log_uniform(rng, 0.04, 4)
    return dict(kind=kind, n=n, metric=metric, elements=elements,
                memory=rng.choice(["device", "device", "host"]),
                select=rng.choice([0, 0, 0, 0, 1]))


# ---- inputs ------------------------------------------------------------------


def _rand(gen, *shape):
    return torch.rand(*shape, generator=gen, dtype=torch.float64, device="cuda")


def _grid(n, gen):
    """n x n vertices on the unit square, interior jittered by 10% of the spacing, both
    triangles of every square along its rising diagonal."""
    i = torch.arange(n, dtype=torch.float64, device="cuda") / (n - 1)
    y, x = torch.meshgrid(i, i, indexing="ij")
    xy = torch.stack([x, y], dim=2)
    if n > 2:
        xy[1:-1, 1:-1] += (2.0 * _rand(gen, n - 2, n - 2, 2) - 1.0) * (0.1 / (n - 1))
    v = torch.arange(n * n, dtype=torch.int32, device="cuda").reshape(n, n)
    v00, v10, v01, v11 = (t.reshape(-1) for t in (v[:-1, :-1], v[:-1, 1:], v[1:, :-1], v[1:, 1:]))
    tri = torch.stack([v00, v10, v11, v00, v11, v01], dim=1).reshape(-1, 3)
    return xy.reshape(-1, 2).contiguous(), tri.contiguous()


def _constant_metric(nv, theta, aspect, h):
    m = inputs.constant_aniso_metric(1, theta, aspect, h)
    return torch.tensor(m, device="cuda").expand(nv, 3).contiguous()


def _bounds(elements):
    """Size bounds of the psi metric: those of the 2M workload, scaled for larger counts so
    that the field stays reachable (an adapted mesh then holds about 1.47 times the estimate)."""
    f = 1.0 if elements <= 2.0e6 else math.sqrt(2.0e6 / (1.47 * elements))
    return 1e-3 * f, 0.3 * f


def _psi_metric(xy, tri, elements, phase=0.0):
    """|Hessian of psi| with its eigenvalues scaled and clamped; the scale is bisected until
    the element-count estimate over the mesh is `elements`."""
    hmin, hmax = _bounds(elements)
    x, y = xy[:, 0], xy[:, 1]
    s = 5.0 * y + phase
    d = torch.sin(s) - 2.0 * x
    den = 1.0 + 100.0 * d * d
    g1, g2, c5 = -10.0 / den, 2000.0 * d / (den * den), torch.cos(s)
    hxx = -250.0 * torch.sin(50.0 * x + phase) + 4.0 * g2
    hxy = -10.0 * c5 * g2
    hyy = 25.0 * c5 * c5 * g2 - 25.0 * torch.sin(s) * g1
    half, dif = 0.5 * (hxx + hyy), 0.5 * (hxx - hyy)
    rad = torch.sqrt(dif * dif + hxy * hxy)
    theta = 0.5 * torch.atan2(2.0 * hxy, hxx - hyy)
    l1, l2, ct, st = (half + rad).abs(), (half - rad).abs(), torch.cos(theta), torch.sin(theta)
    t = tri.long()
    a, b, c = xy[t[:, 0]], xy[t[:, 1]], xy[t[:, 2]]
    area = 0.5 * ((b[:, 0] - a[:, 0]) * (c[:, 1] - a[:, 1])
                  - (b[:, 1] - a[:, 1]) * (c[:, 0] - a[:, 0])).abs()
    # each vertex's share of the area, so that one pass over the vertices gives the estimate
    share = torch.zeros(xy.shape[0], dtype=torch.float64, device="cuda")
    for k in range(3):
        share.index_add_(0, t[:, k], area / 3.0)
    lo, hi = 1.0 / (hmax * hmax), 1.0 / (hmin * hmin)

    def eig(scale):
        return (scale * l1).clamp(lo, hi), (scale * l2).clamp(lo, hi)

    u, w = 1e-8, 1e8
    for _ in range(48):
        mid = math.sqrt(u * w)
        e1, e2 = eig(mid)
        n = 4.0 / math.sqrt(3.0) * float((share * torch.sqrt(e1 * e2)).sum())
        u, w = (mid, w) if n < elements else (u, mid)
    e1, e2 = eig(math.sqrt(u * w))
    return torch.stack([e1 * ct * ct + e2 * st * st, (e1 - e2) * ct * st,
                        e1 * st * st + e2 * ct * ct], dim=1).contiguous()


def _generator(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    return gen


def _mesh(case, seed):
    """Grid and metric of a one-mesh case on the GPU."""
    xy, tri = _grid(case["n"], _generator(seed))
    e = case["elements"]
    metric = case.get("metric", "psi")
    if metric == "psi":
        m = _psi_metric(xy, tri, e)
    else:  # the unit square holds (4 / sqrt 3) / (h * h * aspect) unit triangles
        aspect = 8.0 if metric == "aniso" else 1.0
        h = math.sqrt(4.0 / math.sqrt(3.0) / (e * aspect))
        m = _constant_metric(xy.shape[0], 0.6 if metric == "aniso" else 0.0, aspect, h)
    return xy, tri, m


def _adapted(case, seed):
    """Vertices, triangles and metric after adapting the case's mesh."""
    xy, tri, m = _mesh(case, seed)
    torch.cuda.synchronize()
    with pm.Mesh.from_device(xy, tri) as g:
        g.set_metric_dev(m)
        g.adapt(pm.Params(seed=seed & 0xFFFF))
        nv, ne = g.sizes()
        out = _buffers(nv, ne)
        g.get_mesh_dev(*out)
    return out


def _recipe(case):
    """(grid size, rotation, aspect ratio, size) of every mesh of a batch."""
    out = []
    for i in range(case["count"]):
        u = inputs.uniform01((case["recipe"] << 32) + i, 4)
        t = math.exp(math.log(case["tmin"]) + u[0] * math.log(case["tmax"] / case["tmin"]))
        out.append((int(round(math.sqrt(t / 2.0))) + 1, math.pi * float(u[1]),
                    math.exp(float(u[2]) * math.log(100.0)),
                    math.exp(math.log(0.002) + float(u[3]) * math.log(25.0))))
    return out


def _buffers(nv, ne, host=False):
    kw = dict(pin_memory=True) if host else dict(device="cuda")
    return (torch.zeros((nv, 2), dtype=torch.float64, **kw),
            torch.zeros((ne, 3), dtype=torch.int32, **kw),
            torch.zeros((nv, 3), dtype=torch.float64, **kw))


def _room(nv, ne, elements):
    """Rows of the output buffers: more than any adaptation to `elements` unit triangles
    leaves (checked before they are written)."""
    e = int(1.25 * ne + 2.5 * elements) + 8192
    return max(nv, int(0.55 * e) + 4096), e


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "batch":
        gen = _generator(seed)
        xy, tri, m, est = [], [], [], 0.0
        for n, theta, aspect, h in _recipe(case):
            v, t = _grid(n, gen)
            xy.append(v)
            tri.append(t)
            m.append(_constant_metric(v.shape[0], theta, aspect, h))
            est += 4.0 / math.sqrt(3.0) / (h * h * aspect)
        st["nv"] = np.array([len(v) for v in xy], np.int32)
        st["ne"] = np.array([len(t) for t in tri], np.int32)
        st["mesh"] = (torch.cat(xy), torch.cat(tri), torch.cat(m))
        st["params"] = [pm.Params(seed=(seed * 1000003 + i) & 0xFFFFFFFF)
                        for i in range(case["count"])]
        nv, ne = int(st["nv"].sum()), int(st["ne"].sum())
        v, e = _room(nv, ne, est)
        st["out"] = _buffers(v + 2048 * case["count"], e + 4096 * case["count"])
    elif kind == "grad":
        # the mesh of one adaptation, turned and stretched, its metric scaled vertex by vertex:
        # the same connectivity for every seed, as the gradients' shapes follow from it
        xy, tri, m = _adapted(case, 1)
        gen = _generator(seed)
        a, s = 2.0 * math.pi * float(_rand(gen, 1)), 0.9 + 0.2 * float(_rand(gen, 1))
        turn = torch.tensor([[math.cos(a), -math.sin(a)], [s * math.sin(a), s * math.cos(a)]],
                            dtype=torch.float64, device="cuda")
        xy = (xy @ turn).contiguous()
        m = (m * (0.8 + 0.4 * _rand(gen, xy.shape[0], 1))).contiguous()
        st["args"] = (xy.requires_grad_(), m.requires_grad_(), tri)
    else:
        if kind == "adapt":
            xy, tri, m = _mesh(case, seed)
        else:
            xy, tri, m = _adapted(case, seed)
            if kind == "readapt":
                m = _psi_metric(xy, tri, case["elements"], 2.0 * math.pi / PERIOD)
        host = case.get("memory") == "host"
        nv, ne = case["n"] ** 2, 2 * (case["n"] - 1) ** 2
        extra = 0.0 if kind == "adapt" else case["elements"]
        st["out"] = _buffers(*_room(nv, ne, case["elements"] + extra), host=host)
        if host:
            st["mesh"] = tuple(t.cpu().pin_memory().numpy() for t in (xy, tri, m))
            st["out_np"] = tuple(t.numpy() for t in st["out"])
        else:
            st["mesh"] = (xy, tri, m)
        st["params"] = pm.Params(seed=seed & 0xFFFF, select=case.get("select", 0),
                                 opt_smooth_rounds=case.get("rounds", 0))
    torch.cuda.synchronize()
    return st


# ---- one pass ------------------------------------------------------------------

_COUNTS = ("rounds", "collapses", "splits", "flips", "moves", "converged")


def _read(g, st, stats, sizes):
    """The adapted mesh into the caller's buffers, once they are known to hold it."""
    nv, ne = sizes
    xy, tri, m = st["out"]
    if int(np.sum(nv)) > xy.shape[0] or int(np.sum(ne)) > tri.shape[0]:
        raise ValueError("the output buffers are too small")
    g.get_mesh_dev(xy, tri, m)
    return {"xy": xy, "tri": tri, "m": m, "nv": np.array(nv), "ne": np.array(ne),
            "stats": np.array([[s[k] for k in _COUNTS] for s in stats], np.int64)}


def run(st):
    kind = st["case"]["kind"]
    if kind == "grad":
        xy, m, tri = st["args"]
        q = quality(xy, m, tri)
        gxy, gm = torch.autograd.grad(q, (xy, m))
        return {"q": q.detach(), "dxy": gxy, "dm": gm}
    xy, tri, m = st["mesh"]
    if kind == "batch":
        with pm.Batch.from_device(xy, st["nv"], tri, st["ne"]) as g:
            g.set_metric_dev(m)
            stats = g.adapt(st["params"])
            return _read(g, st, stats, g.sizes())
    if st["case"].get("memory") == "host":
        with pm.Mesh.from_host(xy, tri) as g:
            g.set_metric(m)
            s = g.adapt(st["params"])
            oxy, otri, _ = g.get_mesh(out=st["out_np"])  # refuses buffers that are too small
        nv, ne = oxy.shape[0], otri.shape[0]
        oxy, otri, om = st["out_np"]
        return {"xy": oxy, "tri": otri, "m": om, "nv": nv, "ne": ne,
                "stats": np.array([[s[k] for k in _COUNTS]], np.int64)}
    with pm.Mesh.from_device(xy, tri) as g:
        g.set_metric_dev(m)
        s = g.opt_smooth(st["params"]) if kind == "opt" else g.adapt(st["params"])
        return _read(g, st, [s], g.sizes())


# ---- what a pass cannot do without ---------------------------------------------


def work(case):
    """Bytes: the mesh and the metric read, the adapted mesh and metric (or the gradient)
    written, each once.  Operations: the quality of every element of the result (77) and the
    lengths of its edges (17 each, three to two elements); a gradient takes 250 an element."""
    vertex, triangle = 5 * 8, 3 * 4
    kind = case["kind"]
    if kind == "batch":
        nv = sum(n * n for n, _, _, _ in _recipe(case))
        ne = sum(2 * (n - 1) ** 2 for n, _, _, _ in _recipe(case))
        out = sum(max(2.0, 4.0 / math.sqrt(3.0) / (h * h * a)) for _, _, a, h in _recipe(case))
    else:
        nv, ne, out = case["n"] ** 2, 2 * (case["n"] - 1) ** 2, case["elements"]
        if kind != "adapt":  # the input is an adapted mesh
            nv, ne = 0.5 * out, out
    if kind == "grad":
        return {"bytes": 2 * nv * vertex + ne * triangle, "flops": 250.0 * ne}
    flops = out * (77 + 1.5 * 17)
    if kind == "opt":
        flops *= case["rounds"]
    return {"bytes": nv * vertex + ne * triangle + out * (0.5 * vertex + triangle), "flops": flops}


def exact(case, seed):
    """The quality functional and its gradient in 64 bits by torch's own differentiation.  An
    adapted mesh has no closed form: None."""
    if case["kind"] != "grad":
        return None
    st = prepare(case, seed)
    xy, m, tri = st["args"]
    t = tri.long()
    p, k = xy[t], m[t].sum(dim=1) / 3.0
    e = torch.stack([p[:, 1] - p[:, 0], p[:, 2] - p[:, 1], p[:, 0] - p[:, 2]], dim=1)
    dx, dy = e[..., 0], e[..., 1]
    length = torch.sqrt(k[:, None, 0] * dx * dx + 2.0 * k[:, None, 1] * dx * dy
                        + k[:, None, 2] * dy * dy).sum(dim=1)
    area = 0.5 * (dx[:, 0] * -dy[:, 2] - dy[:, 0] * -dx[:, 2])
    area = area * torch.sqrt(k[:, 0] * k[:, 2] - k[:, 1] * k[:, 1])
    s = torch.minimum(length / 3.0, 3.0 / length)
    q = (12.0 * math.sqrt(3.0) * area / (length * length) * (s * (2.0 - s)) ** 3).sum()
    gxy, gm = torch.autograd.grad(q, (xy, m))
    return {"q": q.detach(), "dxy": gxy, "dm": gm}
