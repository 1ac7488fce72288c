"""Timed cases: the calls a user of the library makes, over the sizes of the workloads, the paper's
table rows and the serving pool.

A case is a dict of plain values.  ``call`` says which entry points a pass goes through:

* ``solve``   ``Problem.solve_device`` on a factored problem (a repeated solve request);
* ``cg``      ``Problem.solve_cg_device`` (the paper's comparison solver);
* ``factor``  ``Problem.factor`` and then one ``Problem.solve_device`` (new operators, one request);
* ``cold``    ``Problem`` (setup and assembly), ``factor`` and ``solve`` on host arrays;
* ``serve``   ``Server.submit`` / ``Server.wait`` of a burst of requests on two problems.

The problem (mesh, kernel, decomposition) follows from the case, the loads and the Dirichlet data
from the seed.  The mixed solves are refined to 1e-10, the tolerance of the FP64 path's PCG, so that
two correct builds agree to the digits of an FP64 result.

The constant kernel on the interval (1-D) and on the l-infinity ball reproduces polynomials exactly
at the nodes of a uniform mesh (quadratics in 1-D, cubics in 2-D, delta a whole number of cells):
those cases are manufactured (Sec. 6.2 of the paper) with random polynomials, so their exact nodal
solution is the polynomial.  The other kernels get N(0,1) load vectors, as the workloads do; their
discrete solution needs the singular pair quadrature of the whole mesh and a dense or banded FP64
factorization, minutes in numpy, so they have no exact().
"""
import collections
import math

import numpy as np
import torch

import workloads as W
from paper_2306_00094_gb300 import binding

KERNELS = {"const_1d": W.KERNEL_CONST_LINF, "const_linf": W.KERNEL_CONST_LINF, "const_l2": W.KERNEL_CONST_L2,
           "fractional": W.KERNEL_FRACTIONAL, "peridynamic": W.KERNEL_PERIDYNAMIC}
SERVE_COUNTS = (1, 5, 12, 3, 32, 8)      # right-hand sides of the requests of one burst


def _case(name, call, kernel, N, k, delta_cells, nrhs, precision=1, precond=1, s=0.5, mesh="grid"):
    """N cells per unit length, k parts per side (k parts in all in 1-D and on an irregular mesh)."""
    c = dict(call=call, kernel=kernel, N=N, k=k, delta_cells=delta_cells, nrhs=nrhs, precision=precision,
             precond=precond, s=s, mesh=mesh)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest request: the 1-D workload (1000 cells, 4 parts, one load), where launches
        # and latency count
        _case("solve_1d", "solve", "const_1d", 1000, 4, 100.0, 1),
        # a warm request on the 2-D constant-kernel workload (16129 dofs, 8 loads)
        _case("solve_const_l2", "solve", "const_l2", 128, 4, 12.8, 8),
        # the fractional workload with the most loads one request carries (64)
        _case("solve_fractional", "solve", "fractional", 96, 6, 19.2, 64),
        # the benchmark's workload: peridynamics, 130050 dofs, 8 x 8 jittered parts, 16 loads, the
        # preconditioner on the tensor cores
        _case("solve_peridynamic", "solve", "peridynamic", 256, 8, 3.0, 16, precond=2),
        # irregular nodes and diagonals with graph-grown parts, odd sizes and an odd load count
        _case("solve_irregular", "solve", "const_l2", 101, 13, 10.1, 5, mesh="irregular"),
        # the paper's 6 x 6 table row (62001 dofs, one load, Dirichlet data) in plain FP64
        _case("solve_row_fp64", "solve", "const_linf", 250, 6, 2.0, 1, precision=0),
        # its 12 x 12 row (249001 dofs, 144 parts, one load) in the mixed mode
        _case("solve_row_12x12", "solve", "const_linf", 500, 12, 4.0, 1),
        # new FP32 operators (a changed material) on peridynamic parts of the benchmark's size
        _case("factor_peridynamic", "factor", "peridynamic", 128, 4, 3.0, 2),
        # new FP64 operators on the 6 x 6 table row
        _case("factor_row_fp64", "factor", "const_linf", 250, 6, 2.0, 1, precision=0),
        # a first request from host arrays: setup, assembly of a singular kernel, factorization, solve
        _case("cold_fractional", "cold", "fractional", 64, 4, 6.4, 4),
        # the paper's comparison solver on the 6 x 6 table row
        _case("cg_row", "cg", "const_linf", 250, 6, 2.0, 1, precision=0),
        # a burst of requests of 1 to 32 loads on two problems of the serving pool
        _case("serve_burst", "serve", "fractional", 64, 8, 6.4, sum(SERVE_COUNTS)),
    ]


def draw(rng):
    """One case of the ranges the listed ones stand for."""
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    call = rng.choice(["solve", "solve", "solve", "solve", "factor", "cold", "cg"])
    if call == "solve" and rng.random() < 0.2:
        K = rng.randint(2, 9)
        per = logint(40, 400)                                   # cells per part
        return _case(None, call, "const_1d", per * K + rng.randint(0, K - 1), K, float(rng.randint(2, per // 3)),
                     logint(1, 16), precision=rng.choice([0, 1]))
    kernel = rng.choice(["const_linf", "const_l2", "fractional", "peridynamic"])
    per = rng.randint(12, 32)                                   # cells per side of a part
    k = rng.randint(2, 4 if call in ("factor", "cold") else (6 if kernel == "peridynamic" else 8))
    N = per * k + rng.randint(0, k - 1)
    if kernel == "const_linf":
        delta = float(rng.randint(2, 4))
    elif kernel == "peridynamic":
        delta = 3.0
    else:
        delta = round(rng.uniform(2.0, min(8.0, per / 2.5)), 1)
    precision = rng.choice([0, 1, 1])
    mesh = "irregular" if kernel == "const_l2" and rng.random() < 0.4 and N <= 128 else "grid"
    nrhs = logint(1, {"solve": 8 if precision == 0 else 64, "factor": 8, "cold": 8, "cg": 8}[call])
    return _case(None, call, kernel, N, k * k if mesh == "irregular" else k, delta, nrhs, precision=precision,
                 precond=rng.choice([1, 2]), s=rng.choice([0.4, 0.5]), mesh=mesh)


# ------------------------------------------------------------------------------ problems

def _workload(case):
    dim = 1 if case["kernel"] == "const_1d" else 2
    N, k = case["N"], case["k"]
    delta = case["delta_cells"] / N
    kern = W.Kernel(KERNELS[case["kernel"]], delta, s=case["s"] if case["kernel"] == "fractional" else 0.0)
    kern.scale = W.default_scale(kern, dim)
    m = W.collar_cells(delta, N)
    if case["mesh"] == "irregular":
        mesh = W.unstructured_mesh(N, m, seed=11)
        labels, K = W.graph_labels(mesh, k, seed=11), k
    else:
        mesh = W.make_mesh(dim, N, m)
        if dim == 1:
            labels, K = W.rect_labels(mesh, k), k
        elif case["kernel"] == "peridynamic":
            labels, K = W.rect_labels(mesh, k, k, jitter=0.2, seed=4), k * k
        else:
            labels, K = W.rect_labels(mesh, k, k), k * k
    return W.Workload(case["kernel"], mesh, kern, labels, K, np.zeros((mesh.n_nodes * kern.ncomp, 0)), 1)


def _options(case):
    if case["precision"] == 0:
        return binding.default_options(precision=0, max_it=20000)
    return binding.default_options(precision=1, refine_tol=1e-10, precond_fp16=case["precond"])


_context = None
_held = collections.OrderedDict()       # the last case's workload and factored problem, as a program keeps them


def _ctx():
    global _context
    if _context is None:
        _context = binding.Context()
    return _context


def _hold(key, make):
    if key not in _held:
        _held.clear()
        _held[key] = make()
    return _held[key]


def _key(case):
    return tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "nrhs")))


def _problem(w, case):
    p = binding.Problem.from_workload(_ctx(), w)
    p.set_options(_options(case))
    return p


def _make(case):
    if case["call"] == "serve":
        other = _case(None, "solve", "const_l2", 2 * case["N"], 3, 3.0, 1)
        made = []
        for c in (case, other):
            w = _workload(c)
            p = _problem(w, c)
            p.factor(2)
            made.append((w, p))
        return made, binding.Server(_ctx(), hbm_budget=0, max_slots=4)
    w = _workload(case)
    if case["call"] == "cold":
        return w, None
    p = _problem(w, case)
    if case["call"] == "cg":
        p.cg_prepare()
    elif case["call"] == "solve":
        p.factor(1 if case["precision"] == 0 else 2)
    return w, p


# ------------------------------------------------------------------------------ loads

def _polynomial(case, seed):
    """A random polynomial per load at the nodes of the mesh (1-D: quadratic, 2-D: cubic) and the
    nodal load f of the nonlocal problem it solves (the kernel constants make the operator -2 u''
    in 1-D and -Laplace u in 2-D on these): arrays (nrhs, nodes)."""
    rng = np.random.default_rng([seed, case["N"], case["k"]])
    N = case["N"]
    m = W.collar_cells(case["delta_cells"] / N, N)
    x = (np.arange(N + 2 * m + 1) - m) / N
    if case["kernel"] == "const_1d":
        a, b, c = rng.uniform(-1.0, 1.0, (3, case["nrhs"], 1))
        return a * x * x + b * x + c, np.broadcast_to(-4.0 * a, (case["nrhs"], x.size)).copy()
    X, Y = np.tile(x, x.size), np.repeat(x, x.size)
    powers = [(i, j) for i in range(4) for j in range(4 - i)]
    u, f = np.zeros((case["nrhs"], X.size)), np.zeros((case["nrhs"], X.size))
    for i, j in powers:
        a = rng.uniform(-1.0, 1.0, (case["nrhs"], 1))
        u += a * X ** i * Y ** j
        if i >= 2:
            f -= a * (i * (i - 1) * X ** (i - 2) * Y ** j)
        if j >= 2:
            f -= a * (j * (j - 1) * X ** i * Y ** (j - 2))
    return u, f


def _manufactured(case):
    return case["kernel"] in ("const_1d", "const_linf")


def _loads(case, w, seed, nrhs):
    """(rhs, rhs_kind, g) as (nrhs, dofs) arrays."""
    if _manufactured(case):
        u, f = _polynomial(case, seed)
        return f, 0, u
    rng = np.random.default_rng([seed, nrhs])
    return rng.standard_normal((nrhs, w.mesh.n_nodes * w.kernel.ncomp)), 1, None


def prepare(case, seed):
    held = _hold(_key(case), lambda: _make(case))
    if case["call"] == "serve":
        made, server = held
        requests = []
        for i, n in enumerate(SERVE_COUNTS):
            w, p = made[i % 2]
            requests.append((p, np.asfortranarray(_loads(case, w, seed + 1000 * i, n)[0].T)))
        return dict(call="serve", server=server, requests=requests)
    w, p = held
    rhs, kind, g = _loads(case, w, seed, case["nrhs"])
    if case["call"] == "cold":
        return dict(call="cold", case=case, w=w, rhs=np.asfortranarray(rhs.T), kind=kind,
                    g=None if g is None else np.asfortranarray(g.T))
    dev = lambda a: None if a is None else torch.from_numpy(a).cuda()
    d_rhs = dev(rhs)
    return dict(call=case["call"], p=p, mask=1 if case["precision"] == 0 else 2, rhs=d_rhs, kind=kind, g=dev(g),
                out=torch.empty_like(d_rhs))


def run(state):
    call = state["call"]
    if call == "serve":
        tickets = [state["server"].submit(p, rhs, 1) for p, rhs in state["requests"]]
        return [state["server"].wait(t)[0] for t in tickets]
    if call == "cold":
        case = state["case"]
        p = _problem(state["w"], case)
        p.factor(1 if case["precision"] == 0 else 2)
        u, _ = p.solve(state["rhs"], state["kind"], state["g"])
        p.close()
        return u
    p = state["p"]
    if call == "cg":
        p.solve_cg_device(state["rhs"], state["kind"], state["out"], state["g"])
        return state["out"]
    if call == "factor":
        p.factor(state["mask"])
    p.solve_device(state["rhs"], state["kind"], state["out"], state["g"])
    return state["out"]


def exact(case, seed):
    if not _manufactured(case):
        return None
    u, _ = _polynomial(case, seed)
    return np.asfortranarray(u.T) if case["call"] == "cold" else torch.from_numpy(u)


def work(case):
    """The least a pass moves and computes: loads in and solution out, and the operators of the
    interface (Gamma_k, about 4 (N/k) delta_cells dofs of a part) read once and applied once; a
    factorization reads every A^k (FP64) once, writes its operators once and needs n_k^3 / 3
    multiply-adds; a cold request also forms A^k; the CG reads the matrix rows (about
    (2 delta_cells + 1)^2 entries per dof) once."""
    if case["call"] == "serve":
        return {k: work(dict(case, call="solve"))[k] + work(dict(case, call="solve", kernel="const_l2", N=2 * case["N"], k=3,
                                                                 delta_cells=3.0))[k] for k in ("bytes", "flops")}
    nc = 2 if case["kernel"] == "peridynamic" else 1
    dim = 1 if case["kernel"] == "const_1d" else 2
    N, dc, R = case["N"], case["delta_cells"], case["nrhs"]
    K = case["k"] if dim == 1 or case["mesh"] == "irregular" else case["k"] ** 2
    s = N / (K if dim == 1 else math.sqrt(K))
    n_k, n_g = nc * (s + dc) ** dim, nc * ((s + dc) ** dim - max(0.0, s - dc) ** dim)
    es = 8 if case["precision"] == 0 else 4
    dofs = nc * (N + 2 * math.ceil(dc) + 1) ** dim
    vectors = 8.0 * dofs * R * (3 if _manufactured(case) else 2)
    if case["call"] == "cg":
        nnz = dofs * nc * (2 * dc + 1) ** dim
        return {"bytes": vectors + 12.0 * nnz, "flops": 2.0 * nnz * R}
    bytes_, flops = vectors + K * n_g ** 2 * es, 2.0 * K * n_g ** 2 * R
    if case["call"] in ("factor", "cold"):
        bytes_ += K * n_k ** 2 * (8 + es)
        flops += K * n_k ** 3 * 2.0 / 3.0
    if case["call"] == "cold":
        bytes_ += K * n_k ** 2 * 8
    return {"bytes": bytes_, "flops": flops}
