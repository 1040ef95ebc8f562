"""The measured cases: what a user of the library has it do, through its public entry points.

One pass is one of these calls (the "kind" of a case):

* ``step``: factorize a system and solve it with the factor as GMRES' preconditioner
  (``ifmm_factor`` + ``bem_gmres``), the whole job of one geometry, for the Laplace kernel in
  FP64 and in the reduced-precision modes, and for the Helmholtz kernel (``wavenumber`` > 0);
* ``batch``: the same for several independent problems at once
  (``ifmm_factor_batched`` + ``bem_gmres_batched``);
* ``solve``: apply a factor that is kept (``ifmm_solve``) to several right-hand sides;
* ``bd``: the block-diagonal preconditioner and GMRES with it (``ifmm_bd_factor`` + ``bem_gmres``);
* ``matvec``: one product with the system matrix (``bem_matvec``) as the FP64 or float-pair
  direct sum or through the FMM representation;
* ``mlp``: the rank predictor's inference and one full-batch gradient
  (``ifmm_mlp_forward`` + ``ifmm_mlp_grad``).

Trees, colorings and right-hand sides are in hand before the call, as for a user who solves on a
geometry; so is the factor of a ``solve``.  Surfaces, sizes, depths and truncations follow the
package's named workloads and its batch generator.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_1905_10602_gb300 import ifmm
from paper_1905_10602_gb300.workloads import batch_workloads, helmholtz_source_rhs, point_source_rhs, surface

RESTART, MAXIT = 30, 500


def _step(name, shape, n, depth, order, eps, sigma, precision, arith, wavenumber=0.0, tol=1e-8):
    return {"name": name, "kind": "step", "shape": shape, "n": n, "depth": depth, "order": order, "eps": eps,
            "sigma": sigma, "precision": precision, "arith": arith, "wavenumber": wavenumber, "tol": tol}


def listed():
    return [
        # the smallest job: a 2,048-point sphere in plain FP64, where launches and latency count
        _step("step-sphere2k-fp64", "sphere", 2048, 3, 3, 1e-6, 6, "fp64", "fp64"),
        # an ordinary FP64 job at the tighter truncation
        _step("step-sphere8k-fp64", "sphere", 8192, 4, 4, 1e-8, 3, "fp64", "fp64"),
        # an ordinary mixed-precision job of an odd size: ragged leaves and random spacing
        _step("step-torus20k-fp32", "torus", 20011, 5, 4, 1e-6, 3, "fp32", "df"),
        # the headline job: 131,072 points, mixed precision
        _step("step-bumpy131k-fp32", "bumpy", 131072, 6, 4, 1e-6, 3, "fp32", "df"),
        # an acoustic job: the complex Helmholtz kernel
        _step("step-helmholtz3k-fp32", "sphere", 3072, 3, 4, 1e-6, 3, "fp32", "fp64", wavenumber=8.0),
        # independent problems together, shapes and sizes mixed as the batch generator draws them
        {"name": "batch8", "kind": "batch", "count": 8, "nmax": 24576, "mix": 5, "eps": 1e-6, "tol": 1e-8},
        # the preconditioner applied in a user's own iteration, an odd size and a few right-hand sides
        {"name": "solve-bumpy12k-fp64", "kind": "solve", "shape": "bumpy", "n": 12289, "depth": 4, "order": 4,
         "eps": 1e-6, "sigma": 3, "nrhs": 4},
        # the cheap preconditioner of a well-conditioned system
        {"name": "bd-bumpy65k", "kind": "bd", "shape": "bumpy", "n": 65536, "depth": 5, "level": 5, "tol": 1e-8},
        # one product with the matrix: the large float-pair sum, an odd FP64 sum, the FMM
        {"name": "matvec-df-131k", "kind": "matvec", "shape": "bumpy", "n": 131072, "depth": 6, "arith": "df",
         "order": 0},
        {"name": "matvec-fp64-10k", "kind": "matvec", "shape": "torus", "n": 10007, "depth": 4, "arith": "fp64",
         "order": 0},
        {"name": "matvec-fmm-65k", "kind": "matvec", "shape": "torus", "n": 65536, "depth": 6, "arith": "fmm",
         "order": 4},
        # the rank predictor: inference and the gradient over a training set
        {"name": "mlp-65k", "kind": "mlp", "n": 65536},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _depth(n):
    return int(min(6, max(2, round(math.log(n / 32.0, 4)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "batch", "solve", "bd", "matvec", "matvec", "mlp"])
    shape = rng.choice(["sphere", "torus", "bumpy"])
    if kind == "step":
        mode = rng.choice(["fp64", "fp32", "fp32", "bf16", "helmholtz"])
        if mode == "helmholtz":
            n = _log_uniform(rng, 600, 3000)
            c = _step("", "sphere", n, _depth(n), 4, 1e-6, 3, "fp32", "fp64", wavenumber=round(rng.uniform(2, 8), 2))
        elif mode == "fp64":
            sigma = rng.choice([3, 6])
            n = _log_uniform(rng, 1024, 7000 if sigma == 3 else 2500)
            c = _step("", shape, n, _depth(n), rng.choice([3, 4]), rng.choice([1e-6, 1e-8]), sigma, "fp64",
                      rng.choice(["fp64", "df"]))
        else:
            # bfloat16 operands make a coarser preconditioner: the residual is asked for further down
            n = _log_uniform(rng, 2048, 100000)
            c = _step("", shape, n, _depth(n), rng.choice([3, 4]), 1e-6, 3, mode, "df",
                      tol=1e-8 if mode == "fp32" else 1e-10)
        del c["name"]
        return c
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(2, 8), "nmax": _log_uniform(rng, 6000, 24576),
                "mix": rng.randint(6, 9999), "eps": 1e-6, "tol": 1e-8}
    if kind == "solve":
        n = _log_uniform(rng, 1024, 12289)
        return {"kind": "solve", "shape": shape, "n": n, "depth": _depth(n), "order": rng.choice([3, 4]),
                "eps": rng.choice([1e-6, 1e-8]), "sigma": 3, "nrhs": rng.randint(1, 8)}
    if kind == "bd":
        n = _log_uniform(rng, 2048, 65536)
        d = _depth(n)
        return {"kind": "bd", "shape": shape, "n": n, "depth": d, "level": rng.choice([d, d - 1]), "tol": 1e-8}
    if kind == "matvec":
        arith = rng.choice(["df", "fp64", "fmm"])
        n = _log_uniform(rng, 1024, {"df": 131072, "fp64": 32768, "fmm": 65536}[arith])
        return {"kind": "matvec", "shape": shape, "n": n, "depth": _depth(n), "arith": arith,
                "order": rng.choice([3, 4]) if arith == "fmm" else 0}
    return {"kind": "mlp", "n": _log_uniform(rng, 256, 65536)}


# ---------------------------------------------------------------- inputs
def _source(seed):
    """A point source away from every surface: inside the sphere-like ones, in the torus' hole."""
    return tuple(np.random.default_rng([seed, 7]).uniform(-0.3, 0.3, 3))


def _points(case, seed):
    return surface(case["shape"], case["n"], seed)


def _batch(case, seed):
    """The problems of a batch: shapes and sizes (folded into [4096, nmax]) of the generator's, points of the seed."""
    out = []
    for k, w in enumerate(batch_workloads(case["count"], case["mix"], 4, case["eps"])):
        n = w.n
        while n > case["nmax"]:
            n = max(4096, n // 2)
        out.append((w.shape, n, _depth(n), seed * 1000 + k))
    return out


def _kernel(case):
    n = case["n"]
    if case.get("wavenumber"):
        return ifmm.helmholtz_kernel(n, case["wavenumber"])
    return ifmm.default_kernel(n, case.get("arith", "df"), case.get("order", 0) if case["kind"] == "matvec" else 0)


def _mlp_inputs(case, seed):
    """Weights of a He initialisation, and predictor inputs and targets in the ranges of a factorization's events."""
    g = np.random.default_rng(seed)
    dims, w = [9, 64, 64, 64, 1], []
    for a, b in zip(dims[:-1], dims[1:]):
        w += [g.uniform(-1, 1, a * b) * math.sqrt(6.0 / a), g.uniform(-0.1, 0.1, b)]
    n = case["n"]
    x = np.empty((n, 9))
    x[:, :3] = g.uniform(-1, 1, (n, 3))                      # cell centre
    x[:, 3] = g.integers(1, 256, n) / 256.0                  # block size
    x[:, 4] = g.integers(2, 7, n) / 10.0                     # level
    x[:, 5] = g.integers(0, 65, n) / 64.0                    # current rank
    x[:, 6] = g.integers(0, 2048, n) / 1024.0                # fill-in rows
    x[:, 7] = g.integers(0, 4, n) / 3.0                      # offset to the eliminated neighbour
    x[:, 8] = g.choice([-4.0, -6.0, -8.0], n) / 10.0         # log10(eps) / 10
    t = g.integers(0, 65, n) / 64.0
    return tuple(np.ascontiguousarray(v, dtype=np.float32) for v in (np.concatenate(w), x, t))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        return {"case": case, "mlp": _mlp_inputs(case, seed)}
    if kind == "batch":
        trees, bs = [], []
        for shape, n, depth, s in _batch(case, seed):
            pts = surface(shape, n, s)
            t = ifmm.ifmm_build_tree(pts, depth)
            ifmm.ifmm_color(t, 3)
            trees.append(t)
            bs.append(point_source_rhs(pts, _source(seed)))
        return {"case": case, "trees": trees, "bs": bs, "kernels": [ifmm.default_kernel(t.n, "df") for t in trees]}
    pts = _points(case, seed)
    tree = ifmm.ifmm_build_tree(pts, case["depth"])
    ifmm.ifmm_color(tree, case.get("sigma", 3))
    state = {"case": case, "tree": tree, "kernel": _kernel(case)}
    if kind == "matvec":
        state["x"] = torch.from_numpy(np.random.default_rng(seed).standard_normal(case["n"])).cuda()
    elif kind == "solve":
        state["x"] = torch.from_numpy(np.random.default_rng(seed).standard_normal((case["nrhs"], case["n"]))).cuda()
        state["fact"] = ifmm.ifmm_factor(tree, case["order"], case["eps"], kernel=state["kernel"], precision="fp64")
    elif case.get("wavenumber"):
        state["b"] = torch.from_numpy(helmholtz_source_rhs(pts, case["wavenumber"], _source(seed))).cuda()
    else:
        state["b"] = torch.from_numpy(point_source_rhs(pts, _source(seed))).cuda()
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "mlp":
        w, x, t = state["mlp"]
        y = ifmm.ifmm_mlp_forward(w, x)
        loss, g = ifmm.ifmm_mlp_grad(w, x, t)
        return {"y": y, "loss": np.float32(loss), "grad": g}
    if kind == "batch":
        facts = ifmm.ifmm_factor_batched(state["trees"], 4, case["eps"], precision="fp32", kernels=state["kernels"])
        xs, _, _ = ifmm.bem_gmres_batched(state["trees"], state["bs"], facts, RESTART, case["tol"], MAXIT,
                                          kernels=state["kernels"])
        return {"x": xs}
    if kind == "matvec":
        return {"y": ifmm.bem_matvec(state["tree"], state["x"], kernel=state["kernel"])}
    if kind == "solve":
        return {"v": ifmm.ifmm_solve(state["fact"], state["x"])}
    if kind == "bd":
        fact = ifmm.ifmm_bd_factor(state["tree"], case["level"], kernel=state["kernel"])
    else:
        fact = ifmm.ifmm_factor(state["tree"], case["order"], case["eps"], kernel=state["kernel"],
                                precision=case["precision"])
    x, _, _ = ifmm.bem_gmres(state["tree"], state["b"], precond=fact, restart=RESTART, tol=case["tol"], maxit=MAXIT,
                             kernel=state["kernel"])
    return {"x": x}


# ---------------------------------------------------------------- work
# Operations of a factorization per point and of a factor's application, from the operation counts that the library
# reports (about 23 MFLOP per point at order 4 and eps = 1e-6, three times that at 1e-8; complex: four times).
def _factor_flops(n, order, eps, dof=1):
    return n * 2.3e7 * (order / 4.0) ** 3 * (3.0 if eps < 1e-7 else 1.0) * dof ** 3


def work(case):
    """What a pass cannot do without: inputs and results once, and the operations of the method."""
    kind, n = case["kind"], case.get("n", 0)
    pair = 20.0  # operations of one ordered pair of a direct sum
    if kind == "mlp":
        macs = 9 * 64 + 64 * 64 * 2 + 64
        return {"bytes": 4.0 * (n * (2 * 9 + 2) + 3 * 9025), "flops": 2.0 * n * macs * 4}
    if kind == "matvec":
        if case["arith"] == "fmm":
            # leaf near field over ~9 neighbours of n / 4^depth points and 64 coefficients over ~27 translations a cell
            cells, rc = 1.3 * 4.0 ** case["depth"] * 4, case["order"] ** 3
            return {"bytes": n * 40.0, "flops": 10 * n * n / cells * pair + cells * 27 * 2 * rc * rc + 4.0 * n * rc}
        return {"bytes": n * 40.0, "flops": pair * n * n}
    if kind == "batch":
        ns = [s[1] for s in _batch(case, 1)]
        return {"bytes": 40.0 * sum(ns), "flops": sum(_factor_flops(m, 4, case["eps"]) + 3 * pair * m * m for m in ns)}
    if kind == "solve":
        coeff = 4200.0 * (case["order"] / 4.0) ** 3 * (1.5 if case["eps"] < 1e-7 else 1.0)  # of the factor, per point
        return {"bytes": n * (8 * coeff + 16.0 * case["nrhs"]), "flops": 2.0 * coeff * n * case["nrhs"]}
    if kind == "bd":
        m = max(1.0, n / (3.2 * 4.0 ** case["level"]))  # points of a block
        return {"bytes": n * 40.0, "flops": 2.0 * n * m * m + 9 * pair * n * n}
    dof = 2 if case["wavenumber"] else 1
    return {"bytes": n * 40.0 * dof,
            "flops": _factor_flops(n, case["order"], case["eps"], dof) + 3 * pair * (4.0 if dof == 2 else 1.0) * n * n}


# ---------------------------------------------------------------- 64-bit values
def _matrix_rows(p, i0, i1, scale, diag, wavenumber=0.0):
    """Rows [i0, i1) of the system matrix of the points p (torch, CUDA, float64)."""
    r = torch.zeros((i1 - i0, p.shape[0]), dtype=torch.float64, device=p.device)
    for d in range(3):
        r += (p[i0:i1, d:d + 1] - p[None, :, d]) ** 2
    r.sqrt_()
    rows = torch.arange(i1 - i0, device=p.device)
    r[rows, rows + i0] = 1.0
    if wavenumber:
        m = torch.polar(scale / r, wavenumber * r)
    else:
        m = scale / r
    m[rows, rows + i0] = diag
    return m


def _matrix(pts, scale, diag, wavenumber=0.0):
    p = torch.from_numpy(pts).cuda()
    n = p.shape[0]
    a = torch.empty((n, n), dtype=torch.complex128 if wavenumber else torch.float64, device="cuda")
    for i in range(0, n, 1024):
        j = min(n, i + 1024)
        a[i:j] = _matrix_rows(p, i, j, scale, diag, wavenumber)
    return a


def _dense_solve(a, b):
    """x with a x = b: directly, or by GMRES to the rounding level where the matrix is large."""
    if a.shape[0] <= 6144:
        return torch.linalg.solve(a, b)
    x, bn = torch.zeros_like(b), b.norm()
    r = b.clone()
    for _ in range(12):
        beta = r.norm()
        if beta <= 3e-15 * bn:
            break
        basis, h, m = [r / beta], torch.zeros((41, 40), dtype=b.dtype, device=b.device), 0
        for j in range(40):
            w = a @ basis[j]
            q = torch.stack(basis)
            for _ in range(2):
                c = q.conj() @ w
                w = w - q.T @ c
                h[:j + 1, j] += c
            nw = w.norm()
            h[j + 1, j] = nw
            m = j + 1
            e = torch.zeros(m + 1, dtype=b.dtype, device=b.device)
            e[0] = beta
            y = torch.linalg.lstsq(h[:m + 1, :m], e[:, None]).solution[:, 0]
            if (h[:m + 1, :m] @ y - e).norm() <= 1e-15 * bn or nw == 0:
                break
            basis.append(w / nw)
        x = x + torch.stack(basis[:m]).T @ y
        r = b - a @ x
    return x


def _mlp_exact(case, seed):
    w, x, t = (torch.from_numpy(v).double() for v in _mlp_inputs(case, seed))
    w.requires_grad_(True)
    dims, o, h = [9, 64, 64, 64, 1], 0, x
    for i, (a, b) in enumerate(zip(dims[:-1], dims[1:])):
        h = h @ w[o:o + a * b].view(a, b) + w[o + a * b:o + a * b + b]
        o += a * b + b
        h = torch.relu(h) if i < 3 else h
    y = h[:, 0]
    loss = ((y - t) ** 2).mean() / 2
    loss.backward()
    return {"y": y.detach(), "loss": loss.detach(), "grad": w.grad}


def exact(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        return _mlp_exact(case, seed)
    if kind == "solve":
        return None  # the factor is an approximation: its application has no value of its own in 64 bits
    if kind == "batch":
        xs = []
        for shape, n, _, s in _batch(case, seed):
            pts = surface(shape, n, s)
            a = _matrix(pts, 1.0 / n, 0.5 + 1.0 / math.sqrt(n))
            xs.append(_dense_solve(a, torch.from_numpy(point_source_rhs(pts, _source(seed))).cuda()))
            del a
        return {"x": xs}
    n = case["n"]
    pts = _points(case, seed)
    if kind == "matvec":
        if case["arith"] == "fmm":
            return None  # the FMM matrix is an approximation of the direct sum
        p = torch.from_numpy(pts).cuda()
        x = torch.from_numpy(np.random.default_rng(seed).standard_normal(n)).cuda()
        y = torch.empty_like(x)
        for i in range(0, n, 1024):
            j = min(n, i + 1024)
            y[i:j] = _matrix_rows(p, i, j, 1.0 / n, 0.5 + 1.0 / math.sqrt(n)) @ x
        return {"y": y}
    if case.get("wavenumber"):
        k = _helmholtz_diag(n, case["wavenumber"])
        a = _matrix(pts, 1.0 / n, k, case["wavenumber"])
        b = helmholtz_source_rhs(pts, case["wavenumber"], _source(seed))
    else:
        a = _matrix(pts, 1.0 / n, 0.5 + 1.0 / math.sqrt(n))
        b = point_source_rhs(pts, _source(seed))
    return {"x": _dense_solve(a, torch.from_numpy(b).cuda())}


def _helmholtz_diag(n, k):
    """Diagonal of the Helmholtz matrix: 0.5 plus the kernel integrated over a disk panel of radius 2 / sqrt(n)."""
    rho = 2.0 / math.sqrt(n)
    return complex(0.5 + math.sin(k * rho) / (2.0 * k), (1.0 - math.cos(k * rho)) / (2.0 * k))
