"""Performance cases: the calls a program makes on a BDDC handle, over the sizes and options in use.

A program sets a handle up once per conductivity field and then calls it many times: M^-1 applies and
products with A inside its own Krylov method, whole PCG solves, load vectors, and the adjoint gradient.
Setup is preparation here; every case times one call on device data through the Python binding (`BDDC`) or
the autograd function (`adjoint.solve`).

A case is a dict: `kind` (apply, matvec, rhs, elem_grad, solve or adjoint), the grid (`dim`, `ne` elements
per direction), the partition (`part`: "box" with `nsub` subdomains per direction, or "voronoi" with `cells`
seeds), the conductivities (`sigma`: "one", "lognormal" = exp(N(0, 1)), or "layers" = 0.1 between Voronoi
cells), the operator `precision`, the number of columns `nrhs` and the `local` solver.
"""
import math

import numpy as np
import torch

import synth
from paper_2410_14786_gb300 import BDDC, adjoint


def _case(kind, dim, ne, nsub, precision, nrhs=1, sigma="lognormal", local="dense", part="box", cells=0):
    return {"kind": kind, "dim": dim, "ne": ne, "part": part, "nsub": nsub, "cells": cells, "sigma": sigma,
            "precision": precision, "nrhs": nrhs, "local": local}


def listed():
    def named(name, *a, **k):
        return dict(_case(*a, **k), name=name)

    return [
        # the smallest workload (2D Laplace, 16 subdomains): one apply is a chain of launches
        named("apply-2d64-fp64", "apply", 2, 64, 4, "fp64", sigma="one"),
        # the 3D heterogeneous workload, one column, the default precision: an outer Krylov method's preconditioner
        named("apply-3d96-fp64", "apply", 3, 96, 12, "fp64"),
        # the mixed form that the solver is fastest with
        named("apply-3d80-bf16", "apply", 3, 80, 10, "bf16"),
        # a block of load cases in float64: 8 columns at once
        named("apply-3d64-fp64-8rhs", "apply", 3, 64, 8, "fp64", nrhs=8),
        # a block of load cases in the mixed form, on the tensor cores
        named("apply-3d64-bf16-8rhs", "apply", 3, 64, 8, "bf16", nrhs=8),
        # cell-like subdomains of uneven sizes, many load cases, float32 operators
        named("apply-voronoi40-fp32-32rhs", "apply", 3, 40, 0, "fp32", nrhs=32, sigma="layers", part="voronoi",
              cells=60),
        # large 2D subdomains (10^4 dofs each), interior solves by sparse factors
        named("apply-2d800-sparse-fp64", "apply", 2, 800, 8, "fp64", sigma="one", local="sparse"),
        # the global product for a block of columns, as in a user's own block Krylov method or residual check
        named("matvec-3d72-8rhs", "matvec", 3, 72, 9, "fp64", nrhs=8),
        # the load vector of nodal values, on a grid whose extents divide into nothing round
        named("rhs-3d77", "rhs", 3, 77, 11, "fp64"),
        # the element term of the adjoint gradient
        named("elem-grad-3d72", "elem_grad", 3, 72, 9, "fp64"),
        # a whole solve to 1e-8 in the mixed form: the headline workload
        named("solve-3d96-bf16", "solve", 3, 96, 12, "bf16"),
        # the backward pass of a misfit through the solve: adjoint solve and gradient, in the default precision
        named("adjoint-3d48-fp64", "adjoint", 3, 48, 6, "fp64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply"] * 6 + ["matvec", "matvec", "rhs", "elem_grad", "solve", "adjoint"])
    shape = rng.choice(["3d", "3d", "3d", "2d", "voronoi", "sparse"] if kind == "apply" else ["3d", "3d", "2d"])
    precision = rng.choice(["fp64", "fp64", "fp32", "bf16", "tf32"]) if kind in ("apply", "solve", "adjoint") else "fp64"
    nrhs = rng.choice([1, 1, 1, _log_int(rng, 2, 32)])
    if shape == "3d":
        size = rng.randint(4, 10)                                  # elements per subdomain and direction
        nsub = _log_int(rng, 2, max(2, (72 if nrhs == 1 else 56) // size))
        return _case(kind, 3, size * nsub, nsub, precision, nrhs)
    if shape == "2d":
        size = _log_int(rng, 8, 30)
        nsub = _log_int(rng, 2, max(2, 300 // size))
        return _case(kind, 2, size * nsub, nsub, precision, nrhs, sigma=rng.choice(["one", "lognormal"]))
    if shape == "voronoi":
        ne = rng.randint(16, 40)
        return _case(kind, 3, ne, 0, precision, nrhs, sigma="layers", part="voronoi",
                     cells=max(4, int(ne ** 3 / rng.uniform(500, 1500))))
    size = _log_int(rng, 32, 110)
    nsub = rng.randint(3, 7)
    return _case(kind, 2, size * nsub, nsub, rng.choice(["fp64", "fp32"]), nrhs, sigma="one", local="sparse")


# -- inputs (from the seed alone) ------------------------------------------------------------------------------

def _partition(case):
    if case["part"] == "voronoi":
        sub, n_sub, cell = synth.voronoi_partition(case["ne"], case["cells"], 4000 + case["ne"])
        return sub, n_sub, cell
    return synth.box_partition(case["dim"], case["ne"], case["nsub"]), case["nsub"] ** case["dim"], None


def _sigma(case, seed, cell):
    n = case["ne"] ** case["dim"]
    if case["sigma"] == "layers":
        return synth.layer_sigma(case["ne"], cell)
    if case["sigma"] == "one":
        return np.ones(n)
    return np.exp(np.random.default_rng(seed).standard_normal(n))


def _shape(case):
    n = (case["ne"] + 1) ** case["dim"]
    return (n,) if case["nrhs"] == 1 else (n, case["nrhs"])


def _normal(case, seed, stream):
    g = torch.Generator(device="cuda").manual_seed(1000003 * (seed + 1) + stream)
    return torch.randn(_shape(case), dtype=torch.float64, device="cuda", generator=g)


def _field(case, seed, stream):
    """A discrete solution's look: a few smooth modes, a tenth of roughness, 0 on the boundary."""
    g = torch.Generator(device="cuda").manual_seed(1000003 * (seed + 1) + stream)
    t = torch.linspace(0, 1, case["ne"] + 1, dtype=torch.float64, device="cuda")
    out = torch.zeros((case["ne"] + 1,) * case["dim"], dtype=torch.float64, device="cuda")
    for k in (1, 2, 3):
        a = torch.rand(case["dim"], dtype=torch.float64, device="cuda", generator=g)
        m = torch.sin(math.pi * k * t)
        term = m
        for _ in range(case["dim"] - 1):
            term = term.unsqueeze(-1) * m
        out += (a.sum() / k) * term
    flat = out.reshape(-1) if case["nrhs"] == 1 else out.reshape(-1, 1).expand(_shape(case))
    flat = flat * (1 + 0.1 * _normal(case, seed, stream + 1))
    inner = _free(case)
    return flat * (inner if case["nrhs"] == 1 else inner.unsqueeze(1))


def _free(case):
    m = torch.zeros((case["ne"] + 1,) * case["dim"], dtype=torch.float64, device="cuda")
    m[(slice(1, -1),) * case["dim"]] = 1.0
    return m.reshape(-1)


def _load(case, seed):
    """The load vector of f = 1 + U[-1, 1] / 2 (lumped over the element mass), 0 on the boundary."""
    f = 1.0 + 0.25 * torch.clamp(_normal(case, seed, 7), -2, 2)
    w = _free(case) * (1.0 / case["ne"]) ** case["dim"]
    return f * (w if case["nrhs"] == 1 else w.unsqueeze(1))


def prepare(case, seed):
    sub, n_sub, cell = _partition(case)
    sigma = _sigma(case, seed, cell)
    if case["kind"] == "adjoint":
        s = torch.tensor(sigma, requires_grad=True)
        b = _load(case, seed).requires_grad_()
        u = adjoint.solve(s, b, case["dim"], case["ne"], sub, n_sub, precision=case["precision"],
                          local_solver=case["local"])
        misfit = 0.5 * ((u - 0.05 * _field(case, seed, 3)) ** 2).sum()
        return {"kind": "adjoint", "misfit": misfit, "sigma": s, "b": b}
    h = BDDC(case["dim"], case["ne"], sigma, sub, n_sub, precision=case["precision"], nrhs_max=case["nrhs"],
             local_solver=case["local"])
    state = {"kind": case["kind"], "handle": h}
    if case["kind"] == "elem_grad":
        state["x"], state["lam"] = _field(case, seed, 1), _field(case, seed, 3)
    elif case["kind"] == "solve":
        state["x"] = _load(case, seed)
    else:
        state["x"] = _normal(case, seed, 1)
    if case["kind"] != "elem_grad":
        state["out"] = h.empty(case["nrhs"])   # a solver keeps its vectors
    return state


def run(state):
    kind = state["kind"]
    if kind == "adjoint":
        g, lam = torch.autograd.grad(state["misfit"], (state["sigma"], state["b"]), retain_graph=True)
        return {"sigma": g, "b": lam}
    h, x = state["handle"], state["x"]
    if kind == "apply":
        return h.apply(x, out=state["out"])
    if kind == "matvec":
        return h.matvec(x, out=state["out"])
    if kind == "rhs":
        return h.rhs(x, out=state["out"])
    if kind == "elem_grad":
        return h.elem_grad(x, state["lam"])
    u, res = h.pcg_solve(x, x=state["out"], rtol=1e-8)
    return {"x": u, "iters": res.iters}


# -- what a pass cannot do without -----------------------------------------------------------------------------

def _local_sizes(case):
    """[(interior, interface, how many subdomains)]: exact for boxes, cubes of the mean volume for Voronoi cells."""
    d = case["dim"]
    if case["part"] == "voronoi":
        s = (case["ne"] ** 3 / case["cells"]) ** (1 / 3)
        return [((s - 1) ** 3, (s + 1) ** 3 - (s - 1) ** 3, case["cells"])]
    size, n = case["ne"] // case["nsub"], case["nsub"]
    # along one axis: a subdomain's nodes off the outer boundary, and its nodes shared with no other one
    axis = [(size + 1 - (i == 0) - (i == n - 1), 1) for i in range(n)]
    kinds = {}
    for a, c in axis:
        kinds[a] = kinds.get(a, 0) + c
    out = {(1, 1): 1}
    for _ in range(d):
        new = {}
        for (nodes, inner), c in out.items():
            for a, k in kinds.items():
                key = (nodes * a, inner * (size - 1))
                new[key] = new.get(key, 0) + c * k
        out = new
    return [(inner, nodes - inner, c) for (nodes, inner), c in out.items()]


def _apply_work(case):
    """The symmetric local operators' triangles (interior twice: a global coarse problem lies between its two
    uses), the vectors in and out; for sparse interior factors the nonzeros of nested dissection's factors."""
    e = {"fp64": 8, "fp32": 4, "tf32": 4, "bf16": 2}[case["precision"]]
    nb = case["nrhs"]
    entries = flops = 0.0
    for n_i, n_g, c in _local_sizes(case):
        inner = n_i * (n_i + 1) / 2
        full_inner = n_i * n_i
        if case["local"] == "sparse":
            inner = 31 / 4 * n_i * max(1.0, math.log2(max(n_i, 2) ** 0.5))   # George's 2D nested dissection
            full_inner = 2 * inner
        entries += c * (2 * inner + n_g * (n_g + 1) / 2)
        flops += c * 2 * nb * (2 * full_inner + n_g * n_g)
    n = (case["ne"] + 1) ** case["dim"]
    return {"bytes": entries * e + 16 * n * nb, "flops": flops}


def work(case):
    n, n_el, nb = (case["ne"] + 1) ** case["dim"], case["ne"] ** case["dim"], case["nrhs"]
    points = 21 if case["dim"] == 3 else 9
    matvec = {"bytes": 8 * n_el + 16 * n * nb, "flops": 2 * points * n * nb}
    if case["kind"] == "apply":
        return _apply_work(case)
    if case["kind"] == "matvec":
        return matvec
    if case["kind"] == "rhs":
        return {"bytes": 16 * n * nb, "flops": 9 * n * nb}
    if case["kind"] == "elem_grad":
        return {"bytes": 16 * n * nb + 8 * n_el, "flops": 2 * 4 ** case["dim"] * n_el * nb}
    a = _apply_work(case)
    its = 12 if case["dim"] == 2 else 30   # PCG iterations to 1e-8 on these workloads
    w = {k: its * (a[k] + matvec[k]) for k in a}
    if case["kind"] == "adjoint":
        w = {"bytes": w["bytes"] + 16 * n * nb + 8 * n_el, "flops": w["flops"]}
    return w


# -- the same in plain torch, 64 bits --------------------------------------------------------------------------

def _corners(dim):
    return [tuple((a >> k) & 1 for k in range(dim)) for a in range(1 << dim)]


def _stiffness(dim, h):
    """The Q1 element matrix: tensor products of the 1D stiffness and mass matrices."""
    k1 = np.array([[1.0, -1.0], [-1.0, 1.0]]) / h
    m1 = np.array([[2.0, 1.0], [1.0, 2.0]]) * h / 6
    c = _corners(dim)
    out = np.zeros((1 << dim, 1 << dim))
    for a in range(1 << dim):
        for b in range(1 << dim):
            for d in range(dim):
                v = 1.0
                for k in range(dim):
                    v *= (k1 if k == d else m1)[c[a][k], c[b][k]]
                out[a, b] += v
    return out


def _grid(case, v):
    """Nodal values [n] or [n, nrhs] as a grid, x last but for the columns."""
    return v.reshape((case["ne"] + 1,) * case["dim"] + (-1,))


def _window(case, corner):
    return tuple(slice(corner[case["dim"] - 1 - ax], corner[case["dim"] - 1 - ax] + case["ne"])
                 for ax in range(case["dim"]))


def _stiff_apply(case, sig, x):
    """A x on the grid, with the boundary rows and columns taken out."""
    K = _stiffness(case["dim"], 1.0 / case["ne"])
    c = _corners(case["dim"])
    free = _grid(case, _free(case))
    x = x * free
    y = torch.zeros_like(x)
    for a in range(len(c)):
        t = torch.zeros_like(x[_window(case, c[0])])
        for b in range(len(c)):
            if abs(K[a, b]) > 1e-14 * abs(K[0, 0]):
                t += K[a, b] * x[_window(case, c[b])]
        y[_window(case, c[a])] += sig * t
    return y * free


def _exact_solve(case, sig, b):
    """Conjugate gradients with the diagonal, far below the tolerance of the solves that are timed."""
    b = b * _grid(case, _free(case))
    diag = torch.zeros_like(b[..., :1])
    K = _stiffness(case["dim"], 1.0 / case["ne"])
    for a, c in enumerate(_corners(case["dim"])):
        diag[_window(case, c)] += K[a, a] * sig
    over = tuple(range(case["dim"]))
    x = torch.zeros_like(b)
    r = b.clone()
    z = r / diag
    p, rz = z.clone(), (r * z).sum(over)
    stop = 1e-13 * torch.sqrt((b * b).sum(over))
    for it in range(20000):
        q = _stiff_apply(case, sig, p)
        a = rz / (p * q).sum(over)
        a = torch.where(torch.isfinite(a), a, torch.zeros_like(a))
        x += a * p
        r -= a * q
        if it % 25 == 24 and bool((torch.sqrt((r * r).sum(over)) <= stop).all()):
            break
        z = r / diag
        new = (r * z).sum(over)
        p = z + torch.where(rz > 0, new / rz, torch.zeros_like(rz)) * p
        rz = new
    return x


def _element_nodes(case):
    n1, ne, d = case["ne"] + 1, case["ne"], case["dim"]
    e = np.arange(ne ** d)
    pos = [e % ne, (e // ne) % ne] + ([e // (ne * ne)] if d == 3 else [])
    return np.stack([sum((pos[k] + c[k]) * n1 ** k for k in range(d)) for c in _corners(d)], axis=1)


def _globs(case, nodes_of, kappa, n_sub):
    """The coarse dofs: connected pieces (along grid lines) of the nodes shared by the same subdomains."""
    n, d, n1 = (case["ne"] + 1) ** case["dim"], case["dim"], case["ne"] + 1
    pairs = np.concatenate([np.stack([v, np.full(v.size, s)], axis=1) for s, v in enumerate(nodes_of)])
    pairs = pairs[np.lexsort((pairs[:, 1], pairs[:, 0]))]
    first = np.searchsorted(pairs[:, 0], np.arange(n))
    shared = np.full((n, 1 << d), -1)
    shared[pairs[:, 0], np.arange(len(pairs)) - first[pairs[:, 0]]] = pairs[:, 1]
    face = np.flatnonzero(kappa >= 2)
    sets = np.full(n, -1)
    sets[face] = np.unique(shared[face], axis=0, return_inverse=True)[1].reshape(-1)
    label = np.where(kappa >= 2, np.arange(n), n).reshape((n1,) * d)
    sets = sets.reshape((n1,) * d)
    while True:
        new = label.copy()
        for ax in range(d):
            lo = tuple(slice(0, -1) if k == ax else slice(None) for k in range(d))
            hi = tuple(slice(1, None) if k == ax else slice(None) for k in range(d))
            same = (sets[lo] >= 0) & (sets[lo] == sets[hi])
            new[hi] = np.where(same, np.minimum(new[hi], new[lo]), new[hi])
            new[lo] = np.where(same, np.minimum(new[lo], new[hi]), new[lo])
        if np.array_equal(new, label):
            break
        label = new
    label = label.reshape(-1)
    glob = np.full(n, -1)
    glob[face] = np.unique(label[face], return_inverse=True)[1].reshape(-1)
    return glob


def _exact_apply(case, sigma, sub, n_sub, r):
    """M^-1 r = v1 + v2 + v3 by its definition: the constrained local problems as dense saddle-point systems, a
    dense coarse matrix, the interior problems of r - A (v1 + v2); None where that would take too long."""
    d, n = case["dim"], (case["ne"] + 1) ** case["dim"]
    en = _element_nodes(case)
    free = _free(case).cpu().numpy() > 0
    order = np.argsort(sub, kind="stable")
    elems = np.split(order, np.cumsum(np.bincount(sub, minlength=n_sub))[:-1])
    nodes_of = [v[free[v]] for v in (np.unique(en[e]) for e in elems)]
    if sum(float(v.size) ** 3 for v in nodes_of) > 1.5e12:
        return None
    kappa = np.bincount(np.concatenate(nodes_of), minlength=n)
    glob = _globs(case, nodes_of, kappa, n_sub)
    n_c = int(glob.max()) + 1
    if n_c > 16000:
        return None
    size = np.bincount(glob[glob >= 0], minlength=n_c)
    K = torch.tensor(_stiffness(d, 1.0 / case["ne"]), device="cuda")
    sig = torch.tensor(sigma, device="cuda")
    rc = torch.zeros((n_c, r.shape[1]), dtype=torch.float64, device="cuda")
    Ac = torch.zeros((n_c, n_c), dtype=torch.float64, device="cuda")
    v = torch.zeros_like(r)
    weight = torch.tensor(1.0 / np.maximum(kappa, 1), device="cuda").unsqueeze(1)
    # subdomains of equal sizes go through the dense solves together
    groups = {}
    for s, nodes in enumerate(nodes_of):
        cs = np.unique(glob[nodes][glob[nodes] >= 0])
        groups.setdefault((nodes.size, cs.size, elems[s].size), []).append((s, cs))
    kept = []
    for (m, nc, ne_), members in groups.items():
        per = max(1, int(2e9 // ((m + nc) ** 2 * 8)))
        for at in range(0, len(members), per):
            some = members[at:at + per]
            B = len(some)
            loc = np.stack([nodes_of[s] for s, _ in some])                          # [B, m] nodes
            le = np.stack([np.searchsorted(nodes_of[s], en[elems[s]]) for s, _ in some])
            hit = np.stack([free[en[elems[s]]] for s, _ in some])
            le = torch.tensor(np.where(hit, le, m), device="cuda")                   # row m: boundary nodes
            es = sig[torch.tensor(np.stack([elems[s] for s, _ in some]), device="cuda")]
            A = torch.zeros((B, (m + 1) * (m + 1)), dtype=torch.float64, device="cuda")
            for a in range(1 << d):
                for b in range(1 << d):
                    A.scatter_add_(1, le[:, :, a] * (m + 1) + le[:, :, b], K[a, b] * es)
            A = A.reshape(B, m + 1, m + 1)[:, :m, :m].contiguous()
            C = np.zeros((B, nc, m))
            for q, (s, cs) in enumerate(some):
                g = glob[nodes_of[s]]
                on = np.flatnonzero(g >= 0)
                C[q, np.searchsorted(cs, g[on]), on] = 1.0 / size[g[on]]
            C = torch.tensor(C, device="cuda")
            t = torch.tensor(loc, device="cuda")
            S = torch.zeros((B, m + nc, m + nc), dtype=torch.float64, device="cuda")
            S[:, :m, :m], S[:, :m, m:], S[:, m:, :m] = A, C.transpose(1, 2), C
            rhs = torch.zeros((B, m + nc, r.shape[1] + nc), dtype=torch.float64, device="cuda")
            wr = weight[t] * r[t]
            rhs[:, :m, :r.shape[1]] = wr
            rhs[:, m:, r.shape[1]:] = torch.eye(nc, dtype=torch.float64, device="cuda")
            sol = torch.linalg.solve(S, rhs)
            z, phi = sol[:, :m, :r.shape[1]], sol[:, :m, r.shape[1]:]
            ct = torch.tensor(np.stack([cs for _, cs in some]).reshape(B, nc), device="cuda")
            rc.index_add_(0, ct.reshape(-1), (phi.transpose(1, 2) @ wr).reshape(B * nc, -1))
            Aci = phi.transpose(1, 2) @ A @ phi
            Ac.view(-1).index_add_(0, (ct.unsqueeze(2) * n_c + ct.unsqueeze(1)).reshape(-1), Aci.reshape(-1))
            v.index_add_(0, t.reshape(-1), (weight[t] * z).reshape(B * m, -1))
            kept.append((t, ct, phi))
            inner = torch.tensor(kappa[loc] == 1, device="cuda")
            if bool(inner.any()):
                k = int(inner[0].sum())
                li = torch.tensor(np.stack([np.flatnonzero(row == 1) for row in kappa[loc]]).reshape(B, k)
                                  if all((row == 1).sum() == k for row in kappa[loc]) else np.zeros((0, 0), int),
                                  device="cuda")
                if li.numel():
                    Aii = torch.gather(torch.gather(A, 1, li.unsqueeze(2).expand(B, k, m)), 2,
                                       li.unsqueeze(1).expand(B, k, k))
                    kept[-1] += (torch.gather(t, 1, li), torch.linalg.cholesky(Aii))
                else:
                    kept[-1] += (None, [(t[q][inner[q]], torch.linalg.cholesky(A[q][inner[q]][:, inner[q]]))
                                        for q in range(B)])
    if n_c:
        uc = torch.linalg.solve(Ac, rc)
        for t, ct, phi, *_ in kept:
            v.index_add_(0, t.reshape(-1), (weight[t] * (phi @ uc[ct])).reshape(t.numel(), -1))
    r1 = r - _stiff_apply(case, sig.reshape((case["ne"],) * d + (1,)), _grid(case, v)).reshape(r.shape)
    for _, _, _, *inside in kept:
        if not inside:
            continue
        if inside[0] is not None:
            v[inside[0].reshape(-1)] += torch.cholesky_solve(r1[inside[0]], inside[1]).reshape(inside[0].numel(), -1)
        else:
            for ti, L in inside[1]:
                if ti.numel():
                    v[ti] += torch.cholesky_solve(r1[ti], L)
    return v


def exact(case, seed):
    sub, n_sub, cell = _partition(case)
    sigma = _sigma(case, seed, cell)
    kind, d = case["kind"], case["dim"]
    sig = torch.tensor(sigma, device="cuda").reshape((case["ne"],) * d + (1,))
    flat = _shape(case)
    if kind == "apply":
        r = _normal(case, seed, 1).reshape(flat[0], -1) * _free(case).unsqueeze(1)
        z = _exact_apply(case, sigma, sub, n_sub, r)
        return None if z is None else z.reshape(flat)
    if kind == "matvec":
        return _stiff_apply(case, sig, _grid(case, _normal(case, seed, 1))).reshape(flat)
    if kind == "rhs":
        f = _grid(case, _normal(case, seed, 1))
        for ax in range(d):   # the consistent mass matrix: (h / 6) [1 4 1] along every axis
            n1 = f.shape[ax]
            g = 4 * f
            g.narrow(ax, 0, n1 - 1).add_(f.narrow(ax, 1, n1 - 1))
            g.narrow(ax, 1, n1 - 1).add_(f.narrow(ax, 0, n1 - 1))
            f = g / (6 * case["ne"])
        return (f * _grid(case, _free(case))).reshape(flat)
    if kind == "solve":
        x = _exact_solve(case, sig, _grid(case, _load(case, seed)))
        return {"x": x.reshape(flat), "iters": None}
    if kind == "elem_grad":
        u, lam = _grid(case, _field(case, seed, 1)), _grid(case, _field(case, seed, 3))
    else:
        u = _exact_solve(case, sig, _grid(case, _load(case, seed)))
        lam = _exact_solve(case, sig, u - 0.05 * _grid(case, _field(case, seed, 3)))
    K = _stiffness(d, 1.0 / case["ne"])
    c = _corners(d)
    g = torch.zeros_like(u[_window(case, c[0])])
    for a in range(len(c)):
        t = torch.zeros_like(g)
        for b in range(len(c)):
            t += K[a, b] * u[_window(case, c[b])]
        g += lam[_window(case, c[a])] * t
    g = -g.sum(-1).reshape(-1)
    return g if kind == "elem_grad" else {"sigma": g.cpu(), "b": lam.reshape(flat)}
