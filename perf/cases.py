"""Performance cases: the calls a user of this package makes, over the sizes they are made at.

Every case goes through the package's public entry points (``ftle.compute``, ``ftle.compute_pair``,
``ftle.ftle_compute_host``, ``ftle.ftle_gradient_eig``, ``ftle.BatchPlan``,
``ftle.ftle_csr_from_elements`` and ``autograd.ftle_field``).  ``exact`` restates the same results
in 64-bit torch without any of the package's code.

A case is a flat dict; ``kind`` says which call it stands for:

* ``compute``  the FTLE field of one mesh on the GPU (advection, gradient, refinement);
* ``pair``     forward and backward field of one mesh;
* ``host``     the same field from page-locked host buffers, copies included;
* ``core``     the FTLE core alone, on a flowmap that comes from elsewhere;
* ``batch``    many uneven double-gyre problems, captured once and replayed;
* ``grad``     a weighted mean of the field and its derivative in the flow's parameters;
* ``csr``      neighbour lists from element connectivity.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2408_02758_gb300 import ftle
from paper_2408_02758_gb300.autograd import ftle_field
from paper_2408_02758_gb300.inputs import FlowSpec

DEV = "cuda"
DT = 0.01  # step of every workload of this package

# neighbour offsets in ascending node order
_OFFS = {
    "axis2": [(0, -1), (-1, 0), (1, 0), (0, 1)],
    "tri": [(-1, -1), (0, -1), (-1, 0), (1, 0), (0, 1), (1, 1)],
    "kuhn": [(-1, -1, -1), (0, -1, -1), (-1, 0, -1), (0, 0, -1), (-1, -1, 0), (0, -1, 0), (-1, 0, 0),
             (1, 0, 0), (0, 1, 0), (1, 1, 0), (0, 0, 1), (1, 0, 1), (0, 1, 1), (1, 1, 1)],
}
_STENCIL_ID = {"axis2": ftle.STENCIL_AXIS, "tri": ftle.STENCIL_TRI, "kuhn": ftle.STENCIL_KUHN}
_JITTER = {"axis2": 0.0, "tri": 0.3, "kuhn": 0.25}


# --------------------------------------------------------------------------------- the cases


def listed():
    return [
        # the smallest call: a coarse preview field, where latency and launches are everything
        {"name": "dg_tri_64x32", "kind": "compute", "nx": 64, "ny": 32, "nz": 1, "stencil": "tri", "layout": "csr",
         "T": 15.0, "precision": "fp32c"},
        # the double-precision workload: a structured 4-neighbour grid
        {"name": "dg_axis_256x128_fp64", "kind": "compute", "nx": 256, "ny": 128, "nz": 1, "stencil": "axis2",
         "layout": "csr", "T": 10.0, "precision": "fp64"},
        # plain float, an ordinary 2D mesh
        {"name": "dg_tri_512x256_fp32", "kind": "compute", "nx": 512, "ny": 256, "nz": 1, "stencil": "tri",
         "layout": "csr", "T": 10.0, "precision": "fp32"},
        # the full-resolution 2D field
        {"name": "dg_tri_2048x1024", "kind": "compute", "nx": 2048, "ny": 1024, "nz": 1, "stencil": "tri",
         "layout": "csr", "T": 15.0, "precision": "fp32c"},
        # an odd-sized tetrahedral mesh integrated backward in time
        {"name": "abc_kuhn_61x47x53_back", "kind": "compute", "nx": 61, "ny": 47, "nz": 53, "stencil": "kuhn",
         "layout": "csr", "T": -5.0, "precision": "fp32c"},
        # the largest: the 3D workload of the benchmark, with the paper's fixed-width neighbour list
        {"name": "abc_kuhn_256", "kind": "compute", "nx": 256, "ny": 256, "nz": 256, "stencil": "kuhn",
         "layout": "ell", "T": 5.0, "precision": "fp32c"},
        # attracting and repelling structures of one mesh
        {"name": "pair_tri_512x256", "kind": "pair", "nx": 512, "ny": 256, "nz": 1, "stencil": "tri",
         "layout": "csr", "T": 10.0, "precision": "fp32c"},
        # a caller with host arrays, copies in and out
        {"name": "host_abc_96", "kind": "host", "nx": 96, "ny": 96, "nz": 96, "stencil": "kuhn", "layout": "csr",
         "T": 5.0, "precision": "fp32c"},
        # the paper's own core: flowmap and neighbour lists given, gradient to FTLE
        {"name": "core_kuhn_160_fp32", "kind": "core", "nx": 160, "ny": 160, "nz": 160, "stencil": "kuhn",
         "layout": "csr", "T": 2.0, "precision": "fp32"},
        # a parameter study: uneven instances replayed from one plan
        {"name": "batch_24", "kind": "batch", "n_inst": 24, "max_exp": 4, "mix": 3, "precision": "fp32c"},
        # one step of fitting the flow's parameters
        {"name": "grad_tri_512x256", "kind": "grad", "nx": 512, "ny": 256, "nz": 1, "stencil": "tri",
         "layout": "csr", "T": 5.0, "precision": "fp32c", "ckpt_every": 50},
        # a tetrahedral mesh that arrives as elements
        {"name": "csr_kuhn_96", "kind": "csr", "nx": 96, "ny": 96, "nz": 96, "stencil": "kuhn"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["compute2", "compute2", "compute3", "compute3", "fp64", "fp32", "pair", "host", "core", "core",
                       "batch", "grad", "csr"])
    two = {"nx": _log_int(rng, 64, 2048), "nz": 1, "stencil": "tri", "layout": rng.choice(["csr", "ell", "stencil"])}
    two["ny"] = max(32, two["nx"] // 2 + rng.randrange(-3, 4))
    e = _log_int(rng, 20, 224)
    three = {"nx": e, "ny": max(16, e + rng.randrange(-9, 10)), "nz": max(16, e + rng.randrange(-9, 10)),
             "stencil": "kuhn", "layout": rng.choice(["csr", "ell", "stencil"])}
    sign = rng.choice([1.0, 1.0, -1.0])
    if kind == "compute2":
        return {"kind": "compute", **two, "T": sign * rng.randrange(300, 1501) / 100, "precision": "fp32c"}
    if kind == "compute3":
        return {"kind": "compute", **three, "T": sign * rng.randrange(100, 501) / 100, "precision": "fp32c"}
    if kind == "fp64":
        nx = _log_int(rng, 32, 512)
        return {"kind": "compute", "nx": nx, "ny": max(16, nx // 2 + rng.randrange(-3, 4)), "nz": 1,
                "stencil": "axis2", "layout": "csr", "T": sign * rng.randrange(200, 1001) / 100, "precision": "fp64"}
    if kind == "fp32":
        return {"kind": "compute", **two, "T": sign * rng.randrange(200, 1001) / 100, "precision": "fp32"}
    if kind == "pair":
        two["nx"], two["ny"] = max(64, two["nx"] // 2), max(32, two["ny"] // 2)
        return {"kind": "pair", **two, "layout": "csr", "T": rng.randrange(300, 1001) / 100, "precision": "fp32c"}
    if kind == "host":
        base = rng.choice([two, three])
        return {"kind": "host", **base, "layout": "csr", "T": rng.randrange(200, 501) / 100, "precision": "fp32c"}
    if kind == "core":
        base = rng.choice([two, three])
        return {"kind": "core", **base, "T": rng.randrange(100, 301) / 100, "precision": "fp32"}
    if kind == "batch":
        return {"kind": "batch", "n_inst": _log_int(rng, 4, 24), "max_exp": rng.randrange(2, 5),
                "mix": rng.randrange(1000), "precision": "fp32c"}
    if kind == "grad":
        nx = _log_int(rng, 64, 768)
        return {"kind": "grad", "nx": nx, "ny": max(32, nx // 2 + rng.randrange(-3, 4)), "nz": 1, "stencil": "tri",
                "layout": "csr", "T": rng.randrange(200, 501) / 100, "precision": "fp32c",
                "ckpt_every": rng.choice([25, 50, 64, 100])}
    e = _log_int(rng, 16, 112)
    return {"kind": "csr", "nx": e, "ny": max(8, e + rng.randrange(-5, 6)), "nz": max(8, e + rng.randrange(-5, 6)),
            "stencil": "kuhn"}


# ----------------------------------------------------------------------------------- inputs


def _shape(case):
    return (case["nx"], case["ny"]) if case["nz"] == 1 else (case["nx"], case["ny"], case["nz"])


def _is_abc(case):
    return case.get("nz", 1) > 1


def _flow(case, seed):
    """The flow's parameters near the workloads' own, drawn from the seed."""
    r = random.Random(seed * 7919 + 17)
    if _is_abc(case):
        return [math.sqrt(3.0) * r.uniform(0.95, 1.0), math.sqrt(2.0) * r.uniform(0.95, 1.0), r.uniform(0.95, 1.0)]
    return [0.1, r.uniform(0.2, 0.3), 2 * math.pi / 10 * r.uniform(0.9, 1.1)]


def _spec(case, p):
    return FlowSpec.abc(*p) if _is_abc(case) else FlowSpec.double_gyre(*p)


def _coords(shape, jitter, seed, dtype):
    """Lattice nodes on [0, 2] x [0, 1] or [0, 2 pi]^3, jittered by U(-jitter, jitter) spacings per
    coordinate (nodes on a face keep their normal coordinate), rounded once to `dtype`."""
    hi = (2.0, 1.0) if len(shape) == 2 else (2 * math.pi,) * 3
    n = math.prod(shape)
    g = torch.Generator(device=DEV).manual_seed(seed)
    i = torch.arange(n, device=DEV)
    out = torch.empty((len(shape), n), dtype=dtype, device=DEV)
    for d, m in enumerate(shape):
        k = i % m
        i = i // m
        x = k.double()
        if jitter:
            u = (2 * torch.rand(n, generator=g, device=DEV, dtype=torch.float64) - 1) * jitter
            x = torch.where((k > 0) & (k < m - 1), x + u, x)
        out[d] = (x * (hi[d] / (m - 1))).to(dtype)
    return out


def _neighbours(shape, stencil):
    """(index, inside) per stencil offset, in ascending node order."""
    n = math.prod(shape)
    i = torch.arange(n, device=DEV, dtype=torch.int32)
    rest, pos = i, []
    for m in shape:
        pos.append(rest % m)
        rest = torch.div(rest, m, rounding_mode="floor")
    for off in _OFFS[stencil]:
        ok = torch.ones(n, dtype=torch.bool, device=DEV)
        step, stride = 0, 1
        for d, m in enumerate(shape):
            if off[d] < 0:
                ok &= pos[d] > 0
            elif off[d] > 0:
                ok &= pos[d] < m - 1
            step += off[d] * stride
            stride *= m
        yield torch.where(ok, i + step, i), ok


def _csr(shape, stencil):
    idx, ok = zip(*_neighbours(shape, stencil))
    ok = torch.stack(ok, 1)
    row_ptr = torch.zeros(ok.shape[0] + 1, dtype=torch.int32, device=DEV)
    row_ptr[1:] = ok.sum(1, dtype=torch.int32).cumsum(0, dtype=torch.int32)
    return row_ptr, torch.stack(idx, 1)[ok]


def _mesh(case, seed):
    shape, st = _shape(case), case["stencil"]
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    dm = ftle.DeviceMesh(_coords(shape, _JITTER[st], seed, dtype), *_csr(shape, st))
    if case["layout"] == "ell":
        dm.attach_ell(len(_OFFS[st]))
    elif case["layout"] == "stencil":
        dm.attach_stencil(_STENCIL_ID[st], shape)
    return dm


def _given_flowmap(case, seed):
    """A flowmap that a caller brings along: 40 steps of RK4 in double, rounded to float."""
    x = _coords(_shape(case), _JITTER[case["stencil"]], seed, torch.float32).double()
    return _rk4(x, _flow(case, seed), case["T"], abs(case["T"]) / 40).float()


def _batch_sizes(case):
    """Sizes and horizons of a batch's instances: 64 2^k x 32 2^k nodes, T in {5, 7.5, 10}."""
    r = random.Random(case["mix"])
    out = []
    for _ in range(case["n_inst"]):
        nx = 64 * 2 ** r.randrange(case["max_exp"] + 1)
        out.append(((nx, nx // 2), r.choice([5.0, 7.5, 10.0])))
    return out


def _batch_flows(case, seed):
    r = random.Random(seed * 31 + 5)
    return [[0.1, r.uniform(0.1, 0.3), r.uniform(math.pi / 10, math.pi / 4)] for _ in range(case["n_inst"])]


def _elements(case, seed):
    """Kuhn tetrahedra of a lattice whose nodes are renumbered at random within runs of 512, with
    each element's vertices in an order of its own: local but not sorted, as meshers number them."""
    nx, ny, nz = _shape(case)
    k, j, i = torch.meshgrid(torch.arange(nz - 1, device=DEV), torch.arange(ny - 1, device=DEV),
                             torch.arange(nx - 1, device=DEV), indexing="ij")
    c = (i + nx * (j + ny * k)).reshape(-1, 1)
    e = [1, nx, nx * ny]
    tets = [[0, e[a], e[a] + e[b], sum(e)] for a, b in [(0, 1), (0, 2), (1, 0), (1, 2), (2, 0), (2, 1)]]
    el = (c[:, :, None] + torch.tensor(tets, device=DEV)[None]).reshape(-1, 4)
    n = math.prod(_shape(case))
    g = torch.Generator(device=DEV).manual_seed(seed)
    key = torch.arange(n, device=DEV) // 512 + torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    el = torch.argsort(key)[el]
    turn = torch.randint(0, 4, (el.shape[0], 1), generator=g, device=DEV)
    el = torch.gather(el, 1, (torch.arange(4, device=DEV)[None] + turn) % 4)
    return el.to(torch.int32).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "csr":
        s["elems"], s["n"] = _elements(case, seed), math.prod(_shape(case))
        return s
    if kind == "batch":
        sizes, flows = _batch_sizes(case), _batch_flows(case, seed)
        meshes = [ftle.DeviceMesh(_coords(sh, 0.0, seed, torch.float32), *_csr(sh, "axis2")) for sh, _ in sizes]
        outs = [torch.empty(m.n_nodes, dtype=torch.float32, device=DEV) for m in meshes]
        ws = ftle.workspace_empty(ftle.ftle_batch_workspace_bytes(meshes, "fp32c"))
        s["outs"] = outs
        s["plan"] = ftle.BatchPlan(meshes, [FlowSpec.double_gyre(*p) for p in flows], [t for _, t in sizes], DT,
                                   "fp32c", outs, ws)
        return s
    p = _flow(case, seed)
    s["flow"] = _spec(case, p)
    if kind == "host":
        shape = _shape(case)
        lists = _csr(shape, case["stencil"])
        s["coords"] = _coords(shape, _JITTER[case["stencil"]], seed, torch.float32).cpu().pin_memory()
        s["row_ptr"], s["col_idx"] = (t.cpu().pin_memory() for t in lists)
        n, nnz = s["coords"].shape[1], s["col_idx"].numel()
        s["out"] = torch.empty(n, dtype=torch.float32).pin_memory()
        s["ws"] = ftle.workspace_empty(ftle.ftle_host_workspace_bytes(len(shape), n, nnz, "fp32c"))
        return s
    s["mesh"] = m = _mesh(case, seed)
    if kind == "core":
        s["phi"] = _given_flowmap(case, seed)
        s["out"] = ftle.ftle_out_empty(m.n_nodes, "fp32")
        s["ws"] = ftle.workspace_empty(ftle.ftle_workspace_bytes(m.n_nodes))
    if kind == "grad":
        s["params"] = torch.tensor(p, dtype=torch.float32, requires_grad=True)
        s["weights"] = _weights(m.coords)
    return s


def _weights(coords):
    """Mean over the nodes with x in [0.5, 1.5]."""
    region = ((coords[0] >= 0.5) & (coords[0] <= 1.5)).float()
    return region / region.sum()


# ------------------------------------------------------------------------------------ a pass


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "compute":
        if case["precision"] == "fp64":
            r = ftle.compute(state["mesh"], state["flow"], case["T"], DT, "fp64", want_lambda=True, return_all=True)
            return {"ftle": r["ftle"], "lam": r["lam"], "phi": r["phi"]}
        return ftle.compute(state["mesh"], state["flow"], case["T"], DT, case["precision"])
    if kind == "pair":
        return ftle.compute_pair(state["mesh"], state["flow"], case["T"], DT, "fp32c")
    if kind == "host":
        ftle.ftle_compute_host(state["coords"], state["row_ptr"], state["col_idx"], state["flow"], 0.0, case["T"], DT,
                               "fp32c", state["out"], state["ws"])
        return state["out"]
    if kind == "core":
        ftle.ftle_gradient_eig(state["mesh"], state["phi"], "fp32", case["T"], state["out"], None, state["ws"])
        return state["out"]
    if kind == "batch":
        state["plan"].launch()
        return state["outs"]
    if kind == "grad":
        field = ftle_field(state["params"], state["mesh"], case["T"], DT, "fp32c", case["ckpt_every"])
        loss = (field * state["weights"]).sum()
        (g,) = torch.autograd.grad(loss, state["params"])
        return {"field": field.detach(), "grad": g}
    row_ptr, col_idx = ftle.ftle_csr_from_elements(state["n"], state["elems"], 72)
    return {"row_ptr": row_ptr, "col_idx": col_idx}


def _n_edges(case):
    """Directed neighbour entries of the lattice."""
    shape = _shape(case)
    return sum(math.prod(m - abs(o) for m, o in zip(shape, off)) for off in _OFFS[case["stencil"]])


def work(case):
    """Bytes: each input read once, each output written once.  Flops: RK4 with one evaluation of the
    velocity's sines and cosines per step and their small-angle turns for the other stages (~150 per
    node and step in 2D and 3D alike), the moments of each neighbour, the closed-form finish."""
    kind = case["kind"]
    if kind == "batch":
        sizes = _batch_sizes(case)
        n = sum(math.prod(sh) for sh, _ in sizes)
        return {"bytes": n * (8 + 4 + 16 + 4),
                "flops": sum(math.prod(sh) * (150 * t / DT + 100) for sh, t in sizes)}
    n, nnz = math.prod(_shape(case)), _n_edges(case)
    dim = len(_shape(case))
    if kind == "csr":
        cells = math.prod(m - 1 for m in _shape(case))
        return {"bytes": 6 * cells * 16 + 4 * (n + 1) + 4 * nnz, "flops": 0}
    w = 8 if case["precision"] == "fp64" else 4
    b = n * dim * w + 4 * (0 if case["layout"] == "stencil" else nnz) + n * w
    if case["layout"] == "csr":
        b += 4 * n
    core = n * 120 + nnz * (30 if dim == 2 else 45)
    steps = abs(case["T"]) / DT
    if kind == "core":
        return {"bytes": b + n * dim * w, "flops": core}
    if kind == "pair":
        return {"bytes": b + n * w, "flops": 2 * (150 * n * steps + core)}
    if kind == "grad":  # forward, one more forward per segment, the reverse sweep
        return {"bytes": 2 * b, "flops": (150 + 150 + 250) * n * steps + 3 * core}
    if case["precision"] == "fp64":
        b += n * w * (1 + dim)
    return {"bytes": b, "flops": 150 * n * steps + core}


# ----------------------------------------------------------------------------- in 64 bits


def _velocity(x, p, t):
    """Double gyre (2 rows) or ABC (3 rows) at time t; p may hold tensors per node."""
    if len(x) == 3:
        A, B, C = p
        s, c = [torch.sin(v) for v in x], [torch.cos(v) for v in x]
        return [A * s[2] + C * c[1], B * s[0] + A * c[2], C * s[1] + B * c[0]]
    A, eps, om = p
    a = eps * (torch.sin(om * t) if torch.is_tensor(om) else math.sin(om * t))
    b = 1 - 2 * a
    f = (a * x[0] + b) * x[0]
    pf, py = math.pi * f, math.pi * x[1]
    return [-math.pi * A * torch.sin(pf) * torch.cos(py),
            math.pi * A * torch.cos(pf) * torch.sin(py) * (2 * a * x[0] + b)]


def _rk4(x, p, T, dt, steps=None):
    """Classic RK4 from t = 0; `steps`: per-node step counts, else the same for all."""
    n = int(round(abs(T) / dt))
    h = math.copysign(dt, T)
    x = list(x)
    for k in range(n):
        t = k * h
        k1 = _velocity(x, p, t)
        k2 = _velocity([a + h / 2 * b for a, b in zip(x, k1)], p, t + h / 2)
        k3 = _velocity([a + h / 2 * b for a, b in zip(x, k2)], p, t + h / 2)
        k4 = _velocity([a + h * b for a, b in zip(x, k3)], p, t + h)
        new = [a + h / 6 * (q1 + 2 * (q2 + q3) + q4) for a, q1, q2, q3, q4 in zip(x, k1, k2, k3, k4)]
        x = new if steps is None else [torch.where(steps > k, b, a) for a, b in zip(x, new)]
    return torch.stack(x)


def _top_eigenvalue(E, dim):
    """Largest eigenvalue of symmetric matrices given by their upper triangle, by cyclic Jacobi."""
    if dim == 2:
        hd = 0.5 * (E[0, 0] - E[1, 1])
        return 0.5 * (E[0, 0] + E[1, 1]) + torch.sqrt(hd * hd + E[0, 1] ** 2)
    a = {k: v.clone() for k, v in E.items()}

    def key(i, j):
        return (min(i, j), max(i, j))

    for _ in range(6):
        for i, j in ((0, 1), (0, 2), (1, 2)):
            k = 3 - i - j
            apq = a[i, j]
            th = (a[j, j] - a[i, i]) / (2 * torch.where(apq == 0, torch.ones_like(apq), apq))
            t = torch.sign(th) / (th.abs() + torch.sqrt(th * th + 1))
            t = torch.where(th == 0, torch.ones_like(t), t)
            t = torch.where(apq == 0, torch.zeros_like(t), t)
            c = 1 / torch.sqrt(t * t + 1)
            s = t * c
            a[i, i], a[j, j] = a[i, i] - t * apq, a[j, j] + t * apq
            a[i, j] = torch.zeros_like(apq)
            aik, ajk = a[key(i, k)], a[key(j, k)]
            a[key(i, k)], a[key(j, k)] = c * aik - s * ajk, s * aik + c * ajk
    return torch.maximum(torch.maximum(a[0, 0], a[1, 1]), a[2, 2])


def _gradient(x, phi, shape, stencil):
    """F = (sum dphi dx^T)(sum dx dx^T)^-1 per node, and M^-1."""
    d = len(shape)
    M = {(r, c): 0.0 for r in range(d) for c in range(r, d)}
    B = [[0.0] * d for _ in range(d)]
    for j, ok in _neighbours(shape, stencil):
        j = j.long()
        dx = [x[r][j] - x[r] for r in range(d)]
        dp = [phi[r][j] - phi[r] for r in range(d)]
        for r in range(d):
            for c in range(d):
                B[r][c] = B[r][c] + dp[r] * dx[c]
                if c >= r:
                    M[r, c] = M[r, c] + dx[r] * dx[c]
    if d == 2:
        det = M[0, 0] * M[1, 1] - M[0, 1] ** 2
        inv = {(0, 0): M[1, 1] / det, (0, 1): -M[0, 1] / det, (1, 1): M[0, 0] / det}
    else:
        co = {(0, 0): M[1, 1] * M[2, 2] - M[1, 2] ** 2, (0, 1): M[0, 2] * M[1, 2] - M[0, 1] * M[2, 2],
              (0, 2): M[0, 1] * M[1, 2] - M[0, 2] * M[1, 1], (1, 1): M[0, 0] * M[2, 2] - M[0, 2] ** 2,
              (1, 2): M[0, 1] * M[0, 2] - M[0, 0] * M[1, 2], (2, 2): M[0, 0] * M[1, 1] - M[0, 1] ** 2}
        det = M[0, 0] * co[0, 0] + M[0, 1] * co[0, 1] + M[0, 2] * co[0, 2]
        inv = {k: v / det for k, v in co.items()}
    F = [[sum(B[r][k] * inv[min(k, c), max(k, c)] for k in range(d)) for c in range(d)] for r in range(d)]
    return F, inv


def _mu(F):
    """lambda_max(F^T F) - 1."""
    d = len(F)
    E = {(r, c): sum(F[k][r] * F[k][c] for k in range(d)) - (1.0 if r == c else 0.0)
         for r in range(d) for c in range(r, d)}
    return _top_eigenvalue(E, d)


def _field(x, phi, shape, stencil, T):
    return torch.log1p(_mu(_gradient(x, phi, shape, stencil)[0])) / (2 * abs(T))


def _dg_tangents(x, p, T):
    """Flowmap and its derivatives in (A, eps, omega): RK4 of the variational equations."""
    A, eps, om = p
    pi = math.pi

    def f(z, t):
        X, Y, D = z
        s, c = math.sin(om * t), math.cos(om * t)
        a = eps * s
        F, fx = (a * X + 1 - 2 * a) * X, 2 * a * X + 1 - 2 * a
        sf, cf, sy, cy = torch.sin(pi * F), torch.cos(pi * F), torch.sin(pi * Y), torch.cos(pi * Y)
        g, gx = X * X - 2 * X, 2 * X - 2
        u, v = -pi * A * sf * cy, pi * A * cf * sy * fx
        ux, uy = -pi * pi * A * cf * cy * fx, pi * pi * A * sf * sy
        vx, vy = pi * A * sy * (2 * a * cf - pi * fx * fx * sf), pi * pi * A * cf * cy * fx
        ua, va = -pi * pi * A * cf * cy * g, pi * A * sy * (gx * cf - pi * fx * g * sf)  # d/da
        src = [(u / A, v / A), (s * ua, s * va), (eps * t * c * ua, eps * t * c * va)]
        return u, v, [(ux * dx + uy * dy + q, vx * dx + vy * dy + r) for (dx, dy), (q, r) in zip(D, src)]

    def add(z, w, k):
        return z[0] + w * k[0], z[1] + w * k[1], [(a + w * c, b + w * d) for (a, b), (c, d) in zip(z[2], k[2])]

    n, h = int(round(abs(T) / DT)), math.copysign(DT, T)
    o = torch.zeros_like(x[0])
    z = (x[0], x[1], [(o, o)] * 3)
    for i in range(n):
        t = i * h
        k1 = f(z, t)
        k2 = f(add(z, h / 2, k1), t + h / 2)
        k3 = f(add(z, h / 2, k2), t + h / 2)
        k4 = f(add(z, h, k3), t + h)
        for w, k in ((h / 6, k1), (h / 3, k2), (h / 3, k3), (h / 6, k4)):
            z = add(z, w, k)
    return z


def _exact_grad(case, seed):
    shape, st, T = _shape(case), case["stencil"], case["T"]
    x32 = _coords(shape, _JITTER[st], seed, torch.float32)
    x = x32.double()
    p = [float(v) for v in torch.tensor(_flow(case, seed), dtype=torch.float32)]
    X, Y, D = _dg_tangents(x, p, T)
    F, inv = _gradient(x, torch.stack([X, Y]), shape, st)
    mu = _mu(F)
    lam = mu + 1
    c01 = F[0][0] * F[0][1] + F[1][0] * F[1][1]
    c00, c11 = F[0][0] ** 2 + F[1][0] ** 2, F[0][1] ** 2 + F[1][1] ** 2
    v = torch.stack([c01, lam - c00])
    w = torch.stack([lam - c11, c01])
    v = torch.where((w * w).sum(0) > (v * v).sum(0), w, v)
    v = v / (v * v).sum(0).sqrt()
    Fv = [F[0][0] * v[0] + F[0][1] * v[1], F[1][0] * v[0] + F[1][1] * v[1]]
    weights = _weights(x32).double()
    g = []
    for d in D:
        G, _ = _gradient(x, torch.stack(d), shape, st)
        dl = 2 * sum(Fv[r] * (G[r][0] * v[0] + G[r][1] * v[1]) for r in range(2))
        g.append((weights * dl / (2 * abs(T) * lam)).sum())
    return {"field": torch.log1p(mu) / (2 * abs(T)), "grad": torch.stack(g).cpu()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "csr":
        return None  # whole numbers
    if kind == "grad":
        return _exact_grad(case, seed)
    if kind == "batch":
        sizes, flows = _batch_sizes(case), _batch_flows(case, seed)
        xs = [_coords(sh, 0.0, seed, torch.float32).double() for sh, _ in sizes]
        per = [x.shape[1] for x in xs]

        def spread(vals):
            return torch.cat([torch.full((m,), v, dtype=torch.float64, device=DEV) for m, v in zip(per, vals)])

        steps = spread([round(t / DT) for _, t in sizes])
        phi = _rk4(torch.cat(xs, 1), [spread([f[q] for f in flows]) for q in range(3)], max(t for _, t in sizes), DT,
                   steps)
        return [_field(x, f, sh, "axis2", t) for x, f, (sh, t) in zip(xs, phi.split(per, 1), sizes)]
    shape, st, T = _shape(case), case["stencil"], case["T"]
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    x = _coords(shape, _JITTER[st], seed, dtype).double()
    p = _flow(case, seed)
    if kind == "core":
        return _field(x, _given_flowmap(case, seed).double(), shape, st, T)
    if kind == "pair":
        return [_field(x, _rk4(x, p, s, DT), shape, st, s) for s in (T, -T)]
    phi = _rk4(x, p, T, DT)
    if case["precision"] == "fp64":
        mu = _mu(_gradient(x, phi, shape, st)[0])
        return {"ftle": torch.log1p(mu) / (2 * abs(T)), "lam": 1 + mu, "phi": phi}
    f = _field(x, phi, shape, st, T)
    return f.cpu() if kind == "host" else f
