"""Performance cases: what a program does with this library, through its public entry points.

A case is a dict of plain values with a "kind":

  walk         node values of one model (host buffers, or device buffers on a stream)
  target       node values to a target standard error (pilot walks, then a top-up)
  batch        node values of several raster models in one launch
  interp       walks at every stride-th node of an interface, interpolation for the others
  interpolate  interpolation of given knot values
  mt           apparent resistivity and phase at measurement sites
  rbffd        sub-domain solve from the values on its boundary

prepare() makes inputs from a seed (the walks' stream seed, the places of the
nodes, the random models and boundary values), run() is one pass, work() the
bytes and operations a pass cannot do without, exact() the outputs in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1603_09311_gb300 import inputs as I
from paper_1603_09311_gb300 import sdd

# ------------------------------------------------------------------- cases


def listed():
    return [
        # the smallest call: one interface node while a grid is being refined,
        # device buffers on the caller's stream
        {"name": "one_node", "kind": "walk", "model": "quarterspace", "nodes": 1, "paths": 1000,
         "paths_hi": 1000, "dt": 1e-3, "precision": "fp32", "device": True},
        # a quick look at one line of nodes of a uniform earth
        {"name": "halfspace_line", "kind": "walk", "model": "halfspace", "nodes": 16, "paths": 10000,
         "paths_hi": 10000, "dt": 1e-3, "precision": "fp32", "device": False},
        # a whole vertical contact at the time step of a final result
        {"name": "quarterspace_line", "kind": "walk", "model": "quarterspace", "nodes": 64, "paths": 100000,
         "paths_hi": 100000, "dt": 1e-4, "precision": "fp32", "device": False},
        # 16 evaluations (8 frequencies x 2 block rates) on a block's perimeter,
        # uneven path counts
        {"name": "block_perimeter", "kind": "walk", "model": "block", "nodes": 256, "paths": 10000,
         "paths_hi": 100000, "dt": 1e-4, "precision": "fp32", "device": False},
        # a triangle's edges at the coarse end of a time-step sweep
        {"name": "triangle_edges", "kind": "walk", "model": "triangle", "nodes": 128, "paths": 100000,
         "paths_hi": 100000, "dt": 1e-3, "precision": "fp32", "device": False},
        # double-precision walks: the check of a single-precision result
        {"name": "fp64_check", "kind": "walk", "model": "quarterspace", "nodes": 7, "paths": 2001,
         "paths_hi": 2001, "dt": 1e-3, "precision": "fp64", "device": False},
        # TM mode on the whole analytic-test grid
        {"name": "tm_grid", "kind": "walk", "model": "tm_analytic", "nodes": 2401, "paths": 4000,
         "paths_hi": 4000, "dt": 1e-4, "precision": "fp32", "device": False},
        # one served request: a random raster model to a standard error of 1e-3
        {"name": "raster_target", "kind": "target", "nodes": 57, "pilot": 4096, "n_max": 1000000,
         "target_se": 1e-3, "dt": 1e-3},
        # a batch of random raster models
        {"name": "raster_batch", "kind": "batch", "models": 12, "nodes": 64, "paths": 4096, "dt": 1e-3},
        # an interface of 1025 nodes with walks at every fourth
        {"name": "interp_interface", "kind": "interp", "nodes": 1025, "stride": 4, "paths": 10000,
         "spline": True, "dt": 1e-3},
        # apparent resistivity at five sites, 16 evaluations, 4e5 walks per point
        {"name": "mt_sites", "kind": "mt", "sites": 5, "paths": 400000, "dt": 1e-4},
        # a sub-domain on 181 x 181 nodes from its boundary values
        {"name": "rbffd_subdomain", "kind": "rbffd", "nx": 181, "nz": 181, "stencil": 9, "eps": 5.0,
         "tol": 1e-10},
    ]


# Euler steps of the largest drawn walk (about those of the listed quarter-space line)
_MAX_STEPS = 1.2e10


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["walk"] * 5 + ["target", "batch", "interp", "interpolate", "mt", "rbffd"])
    dt = rng.choice([1e-3, 3e-4, 1e-4])
    if kind == "walk":
        fp64 = rng.random() < 0.15
        model = rng.choice(["halfspace", "quarterspace", "block", "triangle", "tm_analytic"])
        nodes = _logint(rng, 1, 512)
        paths = _logint(rng, 300, 2e5)
        if fp64:
            dt, nodes = 1e-3, min(nodes, 16)
        cap = 3e6 if fp64 else _MAX_STEPS
        paths = max(1, min(paths, int(cap * dt / (0.35 * nodes))))
        hi = paths if rng.random() < 0.5 else max(1, paths // rng.randint(2, 10))
        return {"kind": kind, "model": model, "nodes": nodes, "paths": min(paths, hi), "paths_hi": max(paths, hi),
                "dt": dt, "precision": "fp64" if fp64 else "fp32", "device": rng.random() < 0.5}
    if kind == "target":
        return {"kind": kind, "nodes": _logint(rng, 16, 120), "pilot": rng.choice([1024, 4096, 5000]),
                "n_max": 400000, "target_se": rng.choice([1e-3, 2e-3, 3e-3]), "dt": 1e-3}
    if kind == "batch":
        m = rng.randint(2, 16)
        return {"kind": kind, "models": m, "nodes": _logint(rng, 8, 200), "paths": _logint(rng, 500, 8000),
                "dt": 1e-3}
    if kind == "interp":
        return {"kind": kind, "nodes": _logint(rng, 17, 2000), "stride": rng.randint(2, 9),
                "paths": _logint(rng, 1000, 20000), "spline": rng.random() < 0.7, "dt": 1e-3}
    if kind == "interpolate":
        return {"kind": kind, "knots": _logint(rng, 5, 1500), "targets": _logint(rng, 50, 6000),
                "comps": rng.choice([2, 6, 32, 64]), "spline": rng.random() < 0.7, "se": rng.random() < 0.7}
    if kind == "mt":
        return {"kind": kind, "sites": _logint(rng, 1, 40), "paths": _logint(rng, 2000, 50000),
                "dt": rng.choice([1e-3, 3e-4])}
    nx, nz = _logint(rng, 12, 200), _logint(rng, 12, 200)
    return {"kind": "rbffd", "nx": nx, "nz": nz, "stencil": rng.choice([9, 9, 13]), "eps": 5.0,
            "tol": rng.choice([1e-10, 1e-9])}


# ------------------------------------------------------------------- inputs

_MODELS = {"halfspace": I.halfspace, "quarterspace": I.quarterspace, "block": I.block_batched,
           "triangle": I.triangle, "tm_analytic": I.tm_analytic}


def _walk_inputs(case, seed):
    """Model, nodes, path counts and stream seed of a walk case: the nodes of
    the model's interface, moved by up to 0.01 along it."""
    rng = np.random.default_rng(seed)
    n, name = case["nodes"], case["model"]
    off = rng.uniform(0.0, 0.01)
    if name == "halfspace":
        nodes = I.nodes_line((-0.5 + off, 0.25), (0.5 + off, 0.25), n)
    elif name == "quarterspace":
        nodes = I.nodes_line((0.0, off if n > 1 else 0.3 + off), (0.0, 0.9 + off), n)
    elif name == "tm_analytic":
        m = math.isqrt(n)
        if m * m == n and m > 1:  # a grid of interior points
            g = np.linspace(-1.0, 1.0, m + 2)[1:-1] * (1.0 - off)
            X, Z = np.meshgrid(g, g)
            nodes = np.stack([X.ravel(), Z.ravel()], axis=1)
        else:
            nodes = I.nodes_line((-0.9, -0.3 + off), (0.9, 0.4), n)
    else:
        verts = I.rect_vertices(I.BLOCK) if name == "block" else I.TRIANGLE
        nodes = I.nodes_on_polygon([(x + off, z) for x, z in verts], n)
    lo, hi = case["paths"], case["paths_hi"]
    paths = np.exp(rng.uniform(math.log(lo), math.log(hi), n)).astype(np.int64) if hi > lo \
        else np.full(n, lo, dtype=np.int64)
    return _MODELS[name](), np.ascontiguousarray(nodes), paths, int(seed) + 17


def _raster_request(rng, n):
    """A random raster model and n nodes on its shapes' perimeters."""
    r = I.random_request(rng, 0)
    nodes = r["nodes"]
    at = np.linspace(0, len(nodes) - 1, n) if n <= len(nodes) else np.arange(n) % len(nodes)
    return r["model"], np.ascontiguousarray(nodes[np.round(at).astype(int)])


def _raster_requests(case, seed, count):
    rng = np.random.default_rng(seed)
    return [_raster_request(rng, case["nodes"]) for _ in range(count)]


def _interface(case, seed):
    """A block's outline, shifted by the seed, as an open polyline."""
    off = np.random.default_rng(seed).uniform(0.0, 0.01)
    return I.nodes_on_polygon([(x + off, z) for x, z in I.rect_vertices(I.BLOCK)], case["nodes"])


def _sites(case, seed):
    off = np.random.default_rng(seed).uniform(0.0, 0.01)
    return np.stack([np.linspace(0.0, 0.8, case["sites"]) + off, np.zeros(case["sites"])], axis=1)


_MT_H = 0.02


def _kappa_ref(model):
    """The host rock's rate in each evaluation."""
    return np.asarray(model["kappa"], dtype=np.float64)[:, 1].copy()


def _column(kappa, z):
    k = np.sqrt(1j * kappa)
    return np.where(z >= 0.0, np.exp(-k * np.maximum(z, 0.0)), 1.0 - k * z)


def _subdomain(case, seed):
    """The quarter-space sub-domain [0, 0.9]^2 on an nx x nz grid: boundary
    values a smooth field plus the noise of walk estimates."""
    rng = np.random.default_rng(seed)
    nodes, edge = I.rect_grid(0.0, 0.9, 0.0, 0.9, case["nx"], case["nz"])
    x, z = nodes[:, 0], nodes[:, 1]
    t = np.clip(x / 0.9, 0.0, 1.0)
    u = (1.0 - t) * _column(6.0, z) + t * _column(20.0, z)
    n = len(nodes)
    u = u + 1e-3 * (rng.standard_normal(n) + 1j * rng.standard_normal(n))
    return nodes, edge, np.where(edge == 1, u, 0.0), np.full(n, 20.0)


def _knots(case, seed):
    rng = np.random.default_rng(seed)
    nk, nt, V = case["knots"], case["targets"], case["comps"]
    s = np.cumsum(rng.uniform(0.5, 1.5, nk)) / nk
    ph = rng.uniform(0.0, 6.0, V)
    v = np.sin(4.0 * s[:, None] + ph) + 1e-3 * rng.standard_normal((nk, V))
    se = np.abs(1e-3 * (1.0 + 0.3 * rng.standard_normal((nk, V)))) if case["se"] else None
    t = np.sort(rng.uniform(s[0], s[-1], nt))
    return s, v, se, np.clip(t, s[0], s[-1])


def prepare(case, seed):
    k = case["kind"]
    st = {"case": case}
    if k == "walk":
        model, nodes, paths, stream_seed = _walk_inputs(case, seed)
        st.update(ctx=sdd.sdd_create(model), nodes=nodes, paths=paths, seed=stream_seed,
                  config=sdd.make_config(precision=case["precision"]))
        if case["device"]:
            E = st["ctx"].E
            st["d_nodes"] = torch.from_numpy(nodes).cuda()
            st["d_mean"] = torch.zeros((len(nodes), E, 2), dtype=torch.float64, device="cuda")
            st["d_se"] = torch.zeros_like(st["d_mean"])
            st["d_counters"] = torch.zeros(3, dtype=torch.int64, device="cuda")
    elif k == "target":
        model, nodes = _raster_requests(case, seed, 1)[0]
        st.update(ctx=sdd.sdd_create(model), nodes=nodes, seed=int(seed) + 17)
    elif k == "batch":
        reqs = _raster_requests(case, seed, case["models"])
        st.update(seed=int(seed) + 17,
                  entries=[{"ctx": sdd.sdd_create(m), "nodes": p, "n_paths": np.full(len(p), case["paths"])}
                           for m, p in reqs])
    elif k == "interp":
        st.update(ctx=sdd.sdd_create(I.block_batched()), nodes=_interface(case, seed), seed=int(seed) + 17)
    elif k == "interpolate":
        st.update(knots=_knots(case, seed))
    elif k == "mt":
        model = I.block_batched()
        st.update(ctx=sdd.sdd_create(model), sites=_sites(case, seed), kref=_kappa_ref(model), seed=int(seed) + 17)
    else:
        st.update(sub=_subdomain(case, seed))
    return st


# --------------------------------------------------------------------- runs

def run(st):
    case = st["case"]
    k = case["kind"]
    if k == "walk" and case["device"]:
        sdd.sdd_interface_values_device(
            st["ctx"], st["d_nodes"].data_ptr(), len(st["nodes"]), st["paths"], case["dt"], st["seed"],
            st["d_mean"].data_ptr(), st["d_se"].data_ptr(), d_counters_ptr=st["d_counters"].data_ptr(),
            stream=torch.cuda.current_stream().cuda_stream, config=st["config"])
        return {"mean": st["d_mean"], "se": st["d_se"], "counters": st["d_counters"]}
    if k == "walk":
        mean, se, s = sdd.sdd_interface_values(st["ctx"], st["nodes"], st["paths"], case["dt"], st["seed"],
                                               config=st["config"])
        return {"mean": mean, "se": se, "steps": s["steps"], "walks": s["walks"]}
    if k == "target":
        mean, se, used, s = sdd.sdd_interface_values_target(
            st["ctx"], st["nodes"], case["pilot"], case["n_max"], case["target_se"], case["dt"], st["seed"])
        return {"mean": mean, "se": se, "used": used, "steps": s["steps"], "walks": s["walks"]}
    if k == "batch":
        res, s = sdd.sdd_batch_values(st["entries"], case["dt"], st["seed"])
        return {"mean": [m for m, _ in res], "se": [e for _, e in res], "steps": s["steps"], "walks": s["walks"]}
    if k == "interp":
        mean, se, s = sdd.sdd_interface_values_interp(
            st["ctx"], st["nodes"], case["stride"], case["paths"], 1 if case["spline"] else 0, case["dt"],
            st["seed"])
        return {"mean": mean, "se": se, "steps": s["steps"], "walks": s["walks"]}
    if k == "interpolate":
        s, v, se, t = st["knots"]
        val, err = sdd.sdd_interpolate(s, v, se, t, 1 if case["spline"] else 0)
        return {"values": val} if err is None else {"values": val, "se": err}
    if k == "mt":
        r = sdd.sdd_apparent_resistivity(st["ctx"], st["sites"], _MT_H, case["paths"], st["kref"], case["dt"],
                                         st["seed"])
        return {f: r[f] for f in ("rho", "phase", "rho_se", "phase_se", "u0", "uz")}
    nodes, edge, values, kappa = st["sub"]
    u, _ = sdd.sdd_rbffd_solve(nodes, edge, values, kappa, n_stencil=case["stencil"], eps=case["eps"],
                               tol=case["tol"], max_iter=20000)
    return {"u": u}


# --------------------------------------------------------------------- work

# Operations of one Euler step: half a Philox call, two uniforms, Box-Muller,
# the move, the wall tests and the occupation update (43), and the interface
# tests of a TM step (47).  Operations of one sample: phase, its sine and
# cosine, boundary value, sums.
_STEP, _STEP_TM, _SAMPLE = 43.0, 47.0, 40.0


def _mean_exit(nodes, domain, D=1.0):
    """Mean exit time of a Brownian motion of diffusion D from a rectangle
    (generator D Lap / 2): its double sine series."""
    a, b = domain[1] - domain[0], domain[3] - domain[2]
    k = np.arange(1, 40, 2)
    sx = np.sin(np.pi * np.outer(nodes[:, 0] - domain[0], k) / a)
    sz = np.sin(np.pi * np.outer(nodes[:, 1] - domain[2], k) / b)
    lam = 0.5 * D * np.pi ** 2 * ((k[:, None] / a) ** 2 + (k[None, :] / b) ** 2)
    c = 16.0 / (np.pi ** 2 * k[:, None] * k[None, :]) / lam
    return np.maximum(np.einsum("ni,ij,nj->n", sx, c, sz), 0.0)


def _walk_work(nodes, paths, dt, E, domain=I.DOMAIN, tm=False):
    paths = np.broadcast_to(np.asarray(paths, dtype=np.float64), (len(nodes),))
    tau = _mean_exit(nodes, domain, 10.0 if tm else 1.0)
    if tm:  # strips of diffusion 1 (x < 0) and 10
        tau = np.where(nodes[:, 0] < 0.0, 5.0 * tau, tau)
    steps = float((paths * (tau / dt + 1.0)).sum())
    return {"bytes": 16.0 * len(nodes) + 32.0 * len(nodes) * E + 8.0 * len(nodes),
            "flops": steps * (_STEP_TM if tm else _STEP) + float(paths.sum()) * E * _SAMPLE}


def work(case):
    k = case["kind"]
    if k == "walk":
        model, nodes, _, _ = _walk_inputs(case, 0)
        lo, hi = case["paths"], case["paths_hi"]
        paths = lo if hi == lo else (hi - lo) / math.log(hi / lo)
        return _walk_work(nodes, paths, case["dt"], len(model["kappa"]), model["domain"], "diffusion" in model)
    if k in ("target", "batch"):
        # nodes all over the earth: mean exit time about 0.25; variances about
        # 0.1 a component at the target's path count
        count = case.get("models", 1)
        paths = case["paths"] if k == "batch" else max(case["pilot"], min(case["n_max"], 0.1 / case["target_se"] ** 2))
        nodes = np.tile([[0.0, 0.6]], (case["nodes"] * count, 1))
        w = _walk_work(nodes, paths, case["dt"], 1)
        w["bytes"] += count * I.RASTER_NX * I.RASTER_NZ
        return w
    if k == "interp":
        nodes = _interface(case, 0)
        knots = nodes[::case["stride"]]
        w = _walk_work(knots, case["paths"], case["dt"], 16)
        w["bytes"] += 16.0 * len(nodes) * 33
        w["flops"] += len(nodes) * 32 * (60.0 if case["spline"] else 8.0)
        return w
    if k == "interpolate":
        nk, nt, V = case["knots"], case["targets"], case["comps"]
        m = 2 if case["se"] else 1
        per = 12.0 if not case["spline"] else 12.0 + 60.0 * (m - 1)
        return {"bytes": 8.0 * (nk + nt + m * V * (nk + nt)), "flops": (nk * 10.0 + nt * per) * V}
    if k == "mt":
        s = _sites(case, 0)
        pts = np.concatenate([s + [0.0, d] for d in (-_MT_H, 0.0, _MT_H)])
        w = _walk_work(pts, case["paths"], case["dt"], 16)
        w["bytes"] += case["sites"] * 16 * 8 * 8.0
        return w
    n, ns = case["nx"] * case["nz"], case["stencil"]
    iters = 3.8 * max(case["nx"], case["nz"])  # BiCGStab iterations grow with the grid's side
    per_row = 2 * (4.0 * ns + 4.0) + 110.0
    return {"bytes": n * (16.0 + 1.0 + 16.0 + 8.0 + 16.0),
            "flops": n * (ns ** 3 * 2.0 / 3.0 + ns * ns * 12.0 + iters * per_row)}


# ---------------------------------------------------- the same, in 64 bits

_M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11) on int64 tensors."""
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for r in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & _M32) ^ c1 ^ k0, p1 & _M32, ((p0 >> 32) & _M32) ^ c3 ^ k1, p0 & _M32
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


def _materials(models, dev):
    """material(x, z, model index) of a list of models that are all rasters or
    one analytic model."""
    m0 = models[0]
    xmin, xmax, zmin, zmax = m0["domain"]
    if m0.get("raster") is not None:
        R = torch.from_numpy(np.stack([np.asarray(m["raster"]) for m in models])).to(dev)
        nz, nx = R.shape[1:]

        def mat(x, z, mi):
            ix = torch.floor((x - xmin) * (nx / (xmax - xmin))).clamp(0, nx - 1).long()
            iz = torch.floor((z - zmin) * (nz / (zmax - zmin))).clamp(0, nz - 1).long()
            return R[mi, iz, ix].long()
        return mat
    air, earth = m0["bg"]

    def mat(x, z, mi):
        m = torch.where(z >= 0.0, earth, air)
        for kind, sm, v in m0["shapes"]:
            if kind == 0:
                inside = (x >= v[0]) & (x < v[1]) & (z >= v[2]) & (z < v[3])
            else:
                p = [(v[0], v[1]), (v[2], v[3]), (v[4], v[5])]
                s = 1.0 if (p[1][0] - p[0][0]) * (p[2][1] - p[0][1]) >= (p[1][1] - p[0][1]) * (p[2][0] - p[0][0]) else -1.0
                inside = torch.ones_like(x, dtype=torch.bool)
                for q in range(3):
                    (ax, az), (bx, bz) = p[q], p[(q + 1) % 3]
                    inside &= s * ((bx - ax) * (z - az) - (bz - az) * (x - ax)) >= 0
            m = torch.where(inside, sm, m)
        return m
    return mat


def _exact_walks(models, nodes, ids, model_of, paths, dt, seed, fp64):
    """Per node and evaluation (mean re, im), (se re, im) of the walks of TE
    models with the library's random streams, every number in 64 bits."""
    dev = torch.device("cuda")
    xmin, xmax, zmin, zmax = models[0]["domain"]
    mat = _materials(models, dev)
    K = max(np.asarray(m["kappa"]).shape[-1] for m in models)
    E = np.atleast_2d(models[0]["kappa"]).shape[0]
    paths = np.asarray(paths, dtype=np.int64)
    N = int(paths.sum())
    reps = torch.from_numpy(paths).to(dev)
    node = torch.repeat_interleave(torch.arange(len(nodes), device=dev), reps)
    first = torch.cumsum(reps, 0) - reps
    path = torch.arange(N, device=dev) - first[node]
    nid = torch.from_numpy(np.asarray(ids, dtype=np.int64)).to(dev)[node]
    mod = torch.from_numpy(np.asarray(model_of, dtype=np.int64)).to(dev)[node]
    P = torch.from_numpy(np.ascontiguousarray(nodes)).to(dev)
    out = {"x": torch.zeros(N, dtype=torch.float64, device=dev), "z": torch.zeros(N, dtype=torch.float64, device=dev),
           "occ": torch.zeros((N, K), dtype=torch.float64, device=dev), "w": torch.zeros(N, dtype=torch.long, device=dev)}
    x, z, idx = P[node, 0], P[node, 1], torch.arange(N, device=dev)
    occ = torch.zeros((N, K), dtype=torch.float64, device=dev)
    alive = torch.ones(N, dtype=torch.bool, device=dev)
    max_steps = (math.ceil(20.0 / dt) + 7) // 8 * 8
    tau2 = 2.0 * math.pi
    for n in range(0, max_steps, 2):
        W = _philox(torch.full_like(path, n >> 1), path, nid, torch.zeros_like(path), seed)
        for h in range(2):
            a, b = W[2 * h], W[2 * h + 1]
            if fp64:
                u0, u1 = (a.double() + 0.5) / 2.0 ** 32, (b.double() + 0.5) / 2.0 ** 32
            else:
                u0, u1 = ((a & 0x7FFFFF).double() + 0.5) / 2.0 ** 23, ((b & 0x7FFFFF).double() + 0.5) / 2.0 ** 23
            r = torch.sqrt(-2.0 * torch.log(u0) * dt)
            xn, zn = x + r * torch.cos(tau2 * u1), z + r * torch.sin(tau2 * u1)
            d = torch.stack([x - xmin, xmax - x, z - zmin, zmax - z])
            e = torch.stack([xn - xmin, xmax - xn, zn - zmin, zmax - zn])
            over = (e <= 0.0).any(0)
            th = torch.where(e <= 0.0, d / (d - e), 3.0)
            th_o, w_o = th.min(0)
            q = 2.0 * d * e / dt
            qm, w_b = q.min(0)
            if fp64:
                u = torch.ones_like(x)
                near = torch.nonzero((qm <= 40.0) & alive).squeeze(1)
                if len(near):
                    v = _philox(torch.full_like(near, n + h), path[near], nid[near], torch.ones_like(near), seed)[0]
                    u[near] = (v.double() + 0.5) / 2.0 ** 32
            else:
                u = (((a >> 23) << 9 | (b >> 23)).double() + 0.5) / 2.0 ** 18
            lu = -torch.log(u)
            hit = over | (qm <= lu)
            end = alive & hit
            at = torch.nonzero(end).squeeze(1)
            if len(at):
                ov = over[at]
                t = torch.where(ov, th_o[at], qm[at] / lu[at])
                w = torch.where(ov, w_o[at], w_b[at])
                ex, ez = x[at] + t * (xn[at] - x[at]), z[at] + t * (zn[at] - z[at])
                ex = torch.where(w == 0, xmin, torch.where(w == 1, xmax, ex))
                ez = torch.where(w == 2, zmin, torch.where(w == 3, zmax, ez))
                o = occ[at]
                o.scatter_add_(1, mat(x[at], z[at], mod[at])[:, None], t[:, None])
                g = idx[at]
                out["x"][g], out["z"][g], out["occ"][g], out["w"][g] = ex, ez, o, w
            alive = alive & ~hit
            occ.scatter_add_(1, mat(xn, zn, mod)[:, None], alive.double()[:, None])
            x, z = torch.where(alive, xn, x), torch.where(alive, zn, z)
        if n % 32 == 30:
            keep = torch.nonzero(alive).squeeze(1)
            if len(keep) == 0:
                break
            if len(keep) < 0.9 * len(alive):
                x, z, idx, path, nid, mod, occ, alive = (v[keep] for v in (x, z, idx, path, nid, mod, occ, alive))
    node_mod = torch.from_numpy(np.asarray(model_of, dtype=np.int64)).to(dev)[node]
    kap = np.zeros((len(models), E, K))
    for i, m in enumerate(models):
        km = np.atleast_2d(np.asarray(m["kappa"], dtype=np.float64))
        kap[i, :, :km.shape[1]] = km
    kap = torch.from_numpy(kap).to(dev)
    gl, gr = models[0]["g"][1:3]
    tx = (out["x"] - xmin) / (xmax - xmin)
    mean = np.zeros((len(nodes), E, 2))
    se = np.zeros((len(nodes), E, 2))

    def col(kappa, zz):
        k = torch.sqrt(1j * kappa.to(torch.complex128))
        return torch.where(zz >= 0.0, torch.exp(-k * zz.clamp(min=0.0)), 1.0 - k * zz)

    cnt = reps.double()
    for e in range(E):
        ke = kap[node_mod, e]
        phase = 0.5 * dt * (ke * out["occ"]).sum(1)
        left, right = col(ke[:, gl], out["z"]), col(ke[:, gr], out["z"])
        blend = left + tx * (right - left)
        g = torch.where(out["w"] == 0, left, torch.where(out["w"] == 1, right, blend))
        s = g * torch.exp(-1j * phase)
        for c, v in enumerate((s.real, s.imag)):
            m = torch.zeros(len(nodes), dtype=torch.float64, device=dev).index_add_(0, node, v) / cnt
            var = torch.zeros(len(nodes), dtype=torch.float64, device=dev).index_add_(0, node, (v - m[node]) ** 2)
            mean[:, e, c] = m.cpu().numpy()
            se[:, e, c] = torch.sqrt(var / (cnt - 1.0) / cnt).cpu().numpy()
    return mean[..., 0] + 1j * mean[..., 1], se


def _exact_spline(s, v, se, t):
    """Natural cubic spline through (s, v) at t, and its standard errors."""
    n = len(s)
    h = np.diff(s)
    A, B = np.eye(n), np.zeros((n, n))
    for i in range(1, n - 1):
        A[i, i - 1:i + 2] = h[i - 1], 2.0 * (h[i - 1] + h[i]), h[i]
        B[i, i - 1:i + 2] = 6.0 / h[i - 1], -6.0 / h[i - 1] - 6.0 / h[i], 6.0 / h[i]
    G = np.linalg.solve(A, B)
    i = np.clip(np.searchsorted(s, t, side="right") - 1, 0, n - 2)
    a, b = (s[i + 1] - t) / h[i], (t - s[i]) / h[i]
    C = ((a ** 3 - a) * h[i] ** 2 / 6.0)[:, None] * G[i] + ((b ** 3 - b) * h[i] ** 2 / 6.0)[:, None] * G[i + 1]
    C[np.arange(len(t)), i] += a
    C[np.arange(len(t)), i + 1] += b
    return C @ v, None if se is None else np.sqrt((C ** 2) @ (se ** 2))


def _exact_linear(s, v, se, t):
    i = np.clip(np.searchsorted(s, t, side="right") - 1, 0, len(s) - 2)
    h = s[i + 1] - s[i]
    a, b = ((s[i + 1] - t) / h)[:, None], ((t - s[i]) / h)[:, None]
    val = a * v[i] + b * v[i + 1]
    return val, None if se is None else np.sqrt((a * se[i]) ** 2 + (b * se[i + 1]) ** 2)


def _exact_subdomain(case, seed):
    """RBF-FD weights by dense solves, the system by a dense solve."""
    nodes, edge, values, kappa = _subdomain(case, seed)
    n, ns, eps = len(nodes), case["stencil"], case["eps"]
    d = nodes[:, None, :] - nodes[None, :, :]
    d2 = d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]
    st = np.stack([np.lexsort((np.arange(n), d2[i]))[:ns] for i in range(n)])
    p = nodes[st]
    r2 = ((p[:, :, None, :] - p[:, None, :, :]) ** 2).sum(-1)
    q2 = ((p - nodes[:, None, :]) ** 2).sum(-1)
    rhs = (2.0 * eps ** 2 + eps ** 4 * q2) / np.sqrt(1.0 + eps ** 2 * q2) ** 3
    w = np.linalg.solve(np.sqrt(1.0 + eps ** 2 * r2), rhs[..., None])[..., 0]
    A = np.zeros((n, n), dtype=np.complex128)
    A[np.arange(n)[:, None], st] = w
    A[np.arange(n), np.arange(n)] -= 1j * kappa
    u = np.where(edge == 1, values, 0.0).astype(np.complex128)
    f = edge == 0
    u[f] = np.linalg.solve(A[np.ix_(f, f)], -A[np.ix_(f, ~f)] @ u[~f])
    return u


def exact(case, seed):
    k = case["kind"]
    if k == "walk":
        # walks at a coarse time step: a small one takes minutes
        if "tm" in case["model"] or case["dt"] < 9e-4 or case["nodes"] * case["paths_hi"] > 2e6:
            return None
        model, nodes, paths, s = _walk_inputs(case, seed)
        if paths.min() < 2:
            return None
        mean, se = _exact_walks([model], nodes, np.arange(len(nodes)), np.zeros(len(nodes)), paths, case["dt"], s,
                                case["precision"] == "fp64")
        if case["device"]:
            return {"mean": np.stack([mean.real, mean.imag], axis=-1), "se": se, "counters": None}
        return {"mean": mean, "se": se, "steps": None, "walks": None}
    if k == "batch":
        if case["models"] * case["nodes"] * case["paths"] > 4e6:
            return None
        reqs = _raster_requests(case, seed, case["models"])
        nodes = np.concatenate([p for _, p in reqs])
        n = case["nodes"]
        mean, se = _exact_walks([m for m, _ in reqs], nodes, np.tile(np.arange(n), len(reqs)),
                                np.repeat(np.arange(len(reqs)), n), np.full(len(nodes), case["paths"]), case["dt"],
                                int(seed) + 17, False)
        cut = [slice(i * n, (i + 1) * n) for i in range(len(reqs))]
        return {"mean": [mean[c] for c in cut], "se": [se[c] for c in cut], "steps": None, "walks": None}
    if k == "interp":
        nodes = _interface(case, seed)
        at = list(range(0, len(nodes), case["stride"]))
        at += [len(nodes) - 1] if at[-1] != len(nodes) - 1 else []
        if len(at) * case["paths"] > 4e6:
            return None
        mean, se = _exact_walks([I.block_batched()], nodes[at], np.array(at), np.zeros(len(at)),
                                np.full(len(at), case["paths"]), case["dt"], int(seed) + 17, False)
        s = np.concatenate([[0.0], np.cumsum(np.hypot(*np.diff(nodes, axis=0).T))])
        f = _exact_spline if case["spline"] and len(at) > 2 else _exact_linear
        kv = np.stack([mean.real, mean.imag], axis=-1).reshape(len(at), -1)
        val, err = f(s[at], kv, se.reshape(len(at), -1), s)
        val[at], err[at] = kv, se.reshape(len(at), -1)
        val = val.reshape(len(nodes), -1, 2)
        return {"mean": val[..., 0] + 1j * val[..., 1], "se": err.reshape(len(nodes), -1, 2), "steps": None,
                "walks": None}
    if k == "interpolate":
        s, v, se, t = _knots(case, seed)
        val, err = (_exact_spline if case["spline"] else _exact_linear)(s, v, se, t)
        return {"values": val} if err is None else {"values": val, "se": err}
    if k == "rbffd" and case["nx"] * case["nz"] <= 2000:
        return {"u": _exact_subdomain(case, seed)}
    return None
