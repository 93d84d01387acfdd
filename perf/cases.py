"""Timed cases of the solver, through its public Python entry points.

Three kinds of pass:

  solve    the operator and the preconditioner are set up (a program keeps both for a
           network it solves again and again); one pass is one pcg_solve with every array on
           the device
  request  one network from host arrays to the solution in host memory: assembly, operator,
           preconditioner, PCG
  serve    a stream of requests through spnet.Server, submitted at once and waited for

The networks are those of paper_2207_07488_gb300.networks at the sizes of its workloads.
A case fixes the geometry of its network; the seed gives the per-edge material weights
U[0.1, 1] (so every seed has another K, other star factors and another coarse matrix) and
the load cases.  Solves run to a relative residual of 1e-11 rather than the default 1e-8,
so that two correct solvers agree to far more digits than 1e-8 would pin down: 1e-12 for the
structural model, whose solution is further from its residual, and 1e-10 on the grid, where
the rounding of the residual ends a little below that.
"""
from __future__ import annotations

import functools
import math
import time
from dataclasses import replace

import numpy as np
import torch

from paper_2207_07488_gb300 import networks as nw
from paper_2207_07488_gb300 import spnet

MAXIT = 4000


def _case(name, kind, net, size, nH, model="scalar", precision="mixed", nrhs=1, stars="interior",
          patch="element", coarse="q1"):
    return {"name": name, "kind": kind, "net": net, "size": size, "nH": nH, "model": model,
            "precision": precision, "nrhs": nrhs, "stars": stars, "patch": patch, "coarse": coarse}


def _rtol(c):
    return 1e-12 if c["model"] == "truss3" else 1e-10 if c["net"] == "grid" else 1e-11


def listed():
    return [
        # the 2D workload (1000 fibres): the smallest call, a chain of short kernels
        _case("solve_2d_1k", "solve", "fiber2d", 1000, 8),
        # a 3D network nearer the size where fibre networks percolate, three load cases
        _case("solve_3d_28k_k3", "solve", "fiber3d", 28000, 11, nrhs=3),
        # the 3D workload (40000 fibres, H = 1/16), the main path: mixed precision, one load
        _case("solve_3d_40k", "solve", "fiber3d", 40000, 16),
        # the same solved by plain FP64 PCG, the arm the mixed path is compared with
        _case("solve_3d_40k_fp64", "solve", "fiber3d", 40000, 16, precision="fp64"),
        # the same with 32 load cases stepped together
        _case("solve_3d_40k_k32", "solve", "fiber3d", 40000, 16, nrhs=32),
        # a large 2D network (about 330000 nodes, 300 a coarse element), a ragged block of loads
        _case("solve_2d_10k_k7", "solve", "fiber2d", 10000, 33, nrhs=7),
        # the structural workload: three components a node, stars of up to 3400 dofs
        _case("solve_truss_40k", "solve", "truss3d", 40000, 12, model="truss3"),
        # the heat experiment of the paper's grid, FP64, a star at every mesh node, support patches
        _case("solve_grid_512", "solve", "grid", 9, 32, precision="fp64", stars="all", patch="support"),
        # a request on the 3D workload from host arrays to host arrays: set-up and solve
        _case("request_3d_40k", "request", "fiber3d", 40000, 16),
        # a 2D request with five load cases: the set-up of large stars weighs most
        _case("request_2d_6k_k5", "request", "fiber2d", 6000, 20, nrhs=5),
        # a structural request
        _case("request_truss_40k", "request", "truss3d", 40000, 12, model="truss3"),
        # the serving stream: requests of mixed dimension, size and number of loads, four in flight
        _case("serve_mixed", "serve", "stream", 12, 0),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["solve", "solve", "solve", "request", "request", "serve"])
    if kind == "serve":
        c = _case("", "serve", "stream", rng.randint(4, 12), rng.randint(1, 999))
        del c["name"]
        return c
    net = rng.choice(["fiber2d", "fiber2d", "fiber3d", "fiber3d", "truss3d", "grid"])
    model, stars, patch, coarse = "scalar", "interior", "element", "q1"
    precision = rng.choice(["mixed", "mixed", "mixed", "fp64"])
    most = 32
    if net == "fiber2d":
        size = log_int(500, 10000)
        nodes = 0.0032 * size ** 2
        nH = max(2, int(round(math.sqrt(nodes / rng.uniform(100, 350)))))
    elif net == "fiber3d":
        size = log_int(500, 40000)
        if 16000 < size < 27000:  # at percolation the rounding of the residual ends above 1e-11
            size += 11000
        nodes = 172461 * (size / 40000) ** 2.2
        nH = max(2, int(round((nodes / rng.uniform(40, 300)) ** (1 / 3))))
    elif net == "truss3d":
        size = rng.randint(32000, 40000)
        model, nodes, nH = "truss3", 3 * 172461, rng.randint(10, 12)
        most = 2
    else:
        size = rng.randint(6, 9)
        nodes, nH = 4.0 ** size, 2 ** (size - 4)
        stars, patch = "all", "support"
    if net in ("fiber2d", "fiber3d") and rng.random() < 0.2:
        coarse, stars = "p1", "all"
    cost = 40 if precision == "fp64" else 10
    most = max(1, min(most, int(172461 * 320 / (cost * max(nodes, 1)))))
    nrhs = 1 if rng.random() < 0.4 else rng.randint(1, most)
    c = _case("", kind, net, size, nH, model, precision, nrhs, stars, patch, coarse)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

@functools.lru_cache(maxsize=32)
def _network(net, size):
    if net == "fiber2d":
        return nw.fiber_network_2d(size, 0.1, 1000 + size)
    if net == "fiber3d":
        return nw.fiber_network_3d(size, 0.1, 0.004, 2000 + size)
    if net == "truss3d":
        return nw.fiber_network_3d(size, 0.1, 0.004, 3000 + size, keep="clamped_x")
    raise ValueError(net)


def _share(net):
    """A node's share of the total edge length (half of its edges' lengths)."""
    d = np.linalg.norm(net.coords[net.edges[:, 1]] - net.coords[net.edges[:, 0]], axis=1)
    m = np.bincount(net.edges[:, 0], d, net.n_nodes) + np.bincount(net.edges[:, 1], d, net.n_nodes)
    return m / m.sum()


def _problem(c, seed):
    """The networks.Problem of a case and its loads F (nrhs, n_dof) and boundary values G."""
    rng = np.random.default_rng([seed, 17])
    H = 1.0 / c["nH"]
    if c["net"] == "grid":
        p = nw.grid_heat_problem(c["size"], H, star_set=c["stars"], patch=c["patch"])
        p.net = replace(p.net, cond=p.net.cond * rng.uniform(0.1, 1.0, p.net.n_edges))
        F = p.f * rng.uniform(0.0, 2.0, (c["nrhs"], p.n_dof))
        return p, F, np.tile(p.dirichlet_vals, (c["nrhs"], 1))
    net = _network(c["net"], c["size"])
    w = rng.uniform(0.1, 1.0, net.n_edges)
    net = replace(net, cond=net.cond * w, stiff=net.stiff * w)
    if c["model"] == "truss3":  # pulled by 0.01 in x (the workload), a different pull in each load case
        p = nw.truss_band_problem(net, H, star_set=c["stars"])
        F = np.zeros((c["nrhs"], p.n_dof))
    else:  # 0 and 1 on the bands, a source spread over the fibres by length
        p = nw.scalar_band_problem(net, H, star_set=c["stars"])
        F = 100.0 * _share(net) * rng.uniform(0.0, 2.0, (c["nrhs"], p.n_dof))
    p.patch, p.coarse = c["patch"], c["coarse"]
    G = p.dirichlet_vals * rng.uniform(0.5, 1.5, (c["nrhs"], 1))
    return p, F, G


def _stream_cases(c):
    """The requests of a stream: 2D and 3D in turn, fibre counts spread over the serving range,
    1 to 8 load cases each."""
    n, out = c["size"], []
    for i in range(n):
        frac = (i * 7 % n) / max(1, n - 1)
        jit = (c["nH"] * 31 + i * 13) % 97
        if i % 2:
            size = int(3000 * 5.0 ** frac) + jit
            nodes = 172461 * (size / 40000) ** 2.2
            nH = max(2, int(round((nodes / 300) ** (1 / 3))))
        else:
            size = int(700 * 6.0 ** frac) + jit
            nH = max(2, int(round(math.sqrt(0.0032 * size ** 2 / 300))))
        out.append(_case("", "request", "fiber3d" if i % 2 else "fiber2d", size, nH, nrhs=1 + (i * 5) % 8))
    return out


def _setup(p, c, device):
    op = spnet.Operator.from_problem(p, device=device)
    pc = spnet.Preconditioner(op, p.H, p.gamma_faces,
                              precision=spnet.PREC_FP64 if c["precision"] == "fp64" else spnet.PREC_MIXED,
                              star_set=spnet.STARS_ALL if c["stars"] == "all" else spnet.STARS_INTERIOR,
                              batch_rhs=c["nrhs"], patch=c["patch"], coarse=c["coarse"])
    return op, pc


def prepare(case, seed):
    if case["kind"] == "serve":
        reqs = [_problem(c, seed + 1000 * i) for i, c in enumerate(_stream_cases(case))]
        return {"case": case, "reqs": reqs, "server": spnet.Server(max_inflight=4)}
    p, F, G = _problem(case, seed)
    if case["nrhs"] == 1:
        F, G = F[0], G[0]
    state = {"case": case, "problem": p}
    if case["kind"] == "request":
        return dict(state, f=np.ascontiguousarray(F), g=np.ascontiguousarray(G))
    op, pc = _setup(p, case, True)
    return dict(state, op=op, pc=pc, f=torch.from_numpy(np.ascontiguousarray(F)).cuda(),
                g=torch.from_numpy(np.ascontiguousarray(G)).cuda())


def run(state):
    case = state["case"]
    if case["kind"] == "serve":
        server = state["server"]
        tickets = [server.submit(p, F, G, rtol=1e-11, maxit=MAXIT, batch_rhs=len(F)) for p, F, G in state["reqs"]]
        out = []
        for t in tickets:
            x, res = server.wait(t)
            if res["status"] != spnet.OK:
                raise RuntimeError(res["message"])
            out.append(x)
        return out
    if case["kind"] == "request":
        op, pc = _setup(state["problem"], case, False)
        u, _ = spnet.pcg_solve(op, pc, state["f"], state["g"], rtol=_rtol(case), maxit=MAXIT)
        pc.close()
        op.close()
        return u
    u, _ = spnet.pcg_solve(state["op"], state["pc"], state["f"], state["g"], rtol=_rtol(case), maxit=MAXIT)
    return u


def _sizes(case):
    """(dofs, entries of K) of a case."""
    if case["net"] == "grid":
        n = 2 ** case["size"] + 1
        return n * n, n * n + 4 * n * (n - 1)
    net = _network(case["net"], case["size"])
    nd = 3 if case["model"] == "truss3" else 1
    return nd * net.n_nodes, nd * nd * (net.n_nodes + 2 * net.n_edges)


def work(case):
    """K (values, columns, row pointers), loads and boundary data read once, solutions written
    once, and one product with K per load case: the lower end of any iteration."""
    cases = _stream_cases(case) if case["kind"] == "serve" else [case]
    b = f = 0
    for c in cases:
        n, nnz = _sizes(c)
        b += 12 * nnz + 8 * n + 16 * n * c["nrhs"]
        f += 2 * nnz * c["nrhs"]
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# the solutions in plain torch: K from the edge list, Jacobi-preconditioned CG in 64 bits
# ---------------------------------------------------------------------------

def _stiffness(p):
    net, n = p.net, p.net.n_nodes
    i, j = net.edges[:, 0], net.edges[:, 1]
    if p.ndof == 1:
        rows = np.concatenate([i, j, i, j])
        cols = np.concatenate([j, i, i, j])
        vals = np.concatenate([-net.cond, -net.cond, net.cond, net.cond])
    else:
        B = net.stiff[:, None, None] * (net.dirs[:, :, None] * net.dirs[:, None, :] + 0.1 * np.eye(3))
        r3, c3 = [], []
        for a, b in ((i, j), (j, i), (i, i), (j, j)):
            r3.append(np.broadcast_to(3 * a[:, None, None] + np.arange(3)[:, None], B.shape).ravel())
            c3.append(np.broadcast_to(3 * b[:, None, None] + np.arange(3)[None, :], B.shape).ravel())
        rows, cols = np.concatenate(r3), np.concatenate(c3)
        vals = np.concatenate([-B.ravel(), -B.ravel(), B.ravel(), B.ravel()])
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    ij = torch.from_numpy(np.stack([rows, cols])).to(dev)
    return torch.sparse_coo_tensor(ij, torch.from_numpy(vals).to(dev), (n * p.ndof,) * 2).coalesce()


def _solve(p, F, G, until):
    """Solutions (nrhs, n_dof), or None if CG is not done by the time `until`."""
    K = _stiffness(p)
    dev, n = K.device, K.shape[0]
    free = torch.ones(n, dtype=torch.bool, device=dev)
    free[torch.from_numpy(p.dirichlet_dofs).to(dev)] = False
    u = torch.zeros(n, len(F), dtype=torch.float64, device=dev)
    u[torch.from_numpy(p.dirichlet_dofs).to(dev)] = torch.from_numpy(np.ascontiguousarray(G.T)).to(dev)
    ij, v = K.indices(), K.values()
    diag = torch.zeros(n, dtype=torch.float64, device=dev)
    on = ij[0] == ij[1]
    diag[ij[0][on]] = v[on]
    idx = torch.cumsum(free, 0) - 1
    keep = free[ij[0]] & free[ij[1]]
    nf = int(free.sum())
    A = torch.sparse_coo_tensor(idx[ij[:, keep]], v[keep], (nf, nf)).coalesce().to_sparse_csr()
    b = torch.from_numpy(np.ascontiguousarray(F.T)).to(dev)[free] - torch.sparse.mm(K, u)[free]
    minv = (1.0 / diag[free])[:, None]
    x = torch.zeros_like(b)
    bb = (b * minv * b).sum(0)
    for _ in range(3):  # restarted from the recomputed residual
        r = b - A @ x
        z = minv * r
        q = z.clone()
        rz = (r * z).sum(0)
        while True:
            for _ in range(100):
                w = A @ q
                a = rz / (q * w).sum(0).clamp_min(1e-300)
                x += a * q
                r -= a * w
                z = minv * r
                new = (r * z).sum(0)
                q = z + (new / rz.clamp_min(1e-300)) * q
                rz = new
            if bool((rz <= 1e-28 * bb).all()):
                break
            if time.time() > until:
                return None
    u[free] = x
    return u.T.contiguous()


def exact(case, seed):
    until = time.time() + 14.0
    if case["kind"] == "serve":
        reqs = [_problem(c, seed + 1000 * i) for i, c in enumerate(_stream_cases(case))]
        return [_solve(*q, until) for q in reqs]
    p, F, G = _problem(case, seed)
    u = _solve(p, F, G, until)
    return u if u is None or case["nrhs"] > 1 else u[0]
