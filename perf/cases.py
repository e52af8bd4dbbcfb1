"""Workloads for timing the library: what a program that uses it calls, from
the smallest grids of the test-suite to the largest benchmark grid, through
the public entry points.

A case is a plain dict.  `op` says which entry point a pass calls:

  spmv     y = A x on the fine grid                       (hpg_spmv)
  smooth   symmetric Gauss-Seidel sweeps on a given z     (hpg_mg_smooth)
  vcycle   one multigrid V-cycle from z = 0               (hpg_mg_vcycle)
  vbatch   the V-cycle of several right-hand sides        (hpg_mg_vcycle_batch)
  solve    a whole GMRES-IR solve                         (hpg_gmres_ir_solve)
  bsolve   several systems, several right-hand sides each, in one call
                                                          (hpg_batch_solve)
  adjoint  differentiable solve, forward and backward     (adjoint.solve)

`exact` restates the operators in plain torch on the natural grid, in 64 bits;
solves are given a right-hand side made from a known solution.
"""

import math

import torch

import paper_2507_11512_gb300 as hpg
from paper_2507_11512_gb300 import adjoint, batch

DEV = "cuda"
BATCH_EDGES = (24, 32, 48, 64, 96)
BASES = {"fp64": hpg.HPG_FP64, "fp32": hpg.HPG_FP32, "bf16": hpg.HPG_BF16, "fp16": hpg.HPG_FP16}


def _case(op, dims, name=None, **kw):
    c = {"op": op, "nx": dims[0], "ny": dims[1], "nz": dims[2], "beta": 0.5, "levels": 4}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the preconditioner on the smallest grid of the test-suite: launches and latency only
        _case("vcycle", (16, 16, 16), "vcycle_16_fp64", prec="fp64"),
        # a standalone smoother call on an odd grid (no coarse level exists), from a given iterate
        _case("smooth", (33, 17, 24), "smooth_33x17x24_fp32", prec="fp32", sweeps=1),
        # the FP64 operator on a ragged grid: what a caller's own residual check costs
        _case("spmv", (82, 78, 84), "spmv_82x78x84_fp64", prec="fp64"),
        # the Arnoldi product of the benchmark grid
        _case("spmv", (128, 128, 128), "spmv_128_fp32", prec="fp32"),
        # the preconditioner of the benchmark grid
        _case("vcycle", (128, 128, 128), "vcycle_128_fp32", prec="fp32"),
        # the preconditioner in FP64 (the FP64-only comparison solve, FP64 adjoints)
        _case("vcycle", (96, 96, 96), "vcycle_96_fp64", prec="fp64"),
        # the preconditioner of the largest benchmark grid
        _case("vcycle", (320, 320, 320), "vcycle_320_fp32", prec="fp32"),
        # the preconditioner of the batched workload's largest system
        _case("vbatch", (96, 96, 96), "vcycle_96_rhs8", nrhs=8, beta=0.6),
        # the smallest whole solve: plain FP64 GMRES(30)
        _case("solve", (16, 16, 16), "solve_16_fp64", basis="fp64", restart=30, tol=1e-11),
        # the benchmark solve (FP32 inner GMRES(30), FP64 refinement), run two digits further
        # than its 1e-9 so that the solution itself is determined to 1e-9
        _case("solve", (128, 128, 128), "solve_128_mxp", basis="fp32", restart=30, tol=1e-11),
        # one system of each edge of the batched workload, 8 right-hand sides each, one call
        {"name": "solve_batch_5x8", "op": "bsolve", "systems": 5, "first": 0, "nrhs": 8,
         "beta": 0.4, "restart": 30, "tol": 1e-12},
        # the differentiable workload: new per-cell scales on each state, gradients to b and
        # theta (the scaled operator amplifies a residual by several thousand)
        _case("adjoint", (96, 96, 96), "adjoint_96", tol=1e-13),
    ]


def _edges(rng, lo, hi):
    """Three edges whose product is spread over its logarithm; half of the
    grids coarsen three times, the others have any edges."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    e = [n * math.exp(rng.uniform(-0.35, 0.35)) for _ in range(3)]
    if rng.random() < 0.5:
        return [max(8, 8 * round(v / 8)) for v in e]
    return [max(3, round(v)) for v in e]


def draw(rng):
    op = rng.choice(["spmv", "smooth", "vcycle", "vcycle", "vbatch", "solve", "bsolve", "adjoint"])
    beta = rng.choice([0.0, 0.5, round(rng.uniform(-0.75, 0.75), 3)])
    if op in ("spmv", "smooth", "vcycle"):
        prec = rng.choice(["fp32", "fp32", "fp64"])
        c = _case(op, _edges(rng, 12, 200), prec=prec, beta=beta)
        if op == "smooth":
            c["sweeps"] = rng.choice([1, 2, 3])
        return c
    if op == "vbatch":
        return _case(op, _edges(rng, 12, 90), nrhs=rng.choice([2, 4, 8]), beta=beta)
    if op == "solve":
        basis = rng.choice(["fp32", "bf16", "fp16", "fp64"])
        e = [max(8, 8 * round(v / 8)) for v in _edges(rng, 12, 100)]
        return _case(op, e, basis=basis, restart=rng.choice([20, 30, 50]), tol=1e-12, beta=beta)
    if op == "bsolve":
        return {"op": "bsolve", "systems": rng.randint(2, 5), "first": rng.randint(0, 4),
                "nrhs": rng.choice([2, 4, 8]), "beta": round(rng.uniform(0.25, 0.75), 3),
                "restart": 30, "tol": 1e-12}
    e = [max(8, 8 * round(v / 8)) for v in _edges(rng, 12, 80)]
    return _case(op, e, tol=1e-13, beta=beta)


# ------------------------------------------- the operators in plain torch, 64 bits
def _coef(beta, dx, dy, dz):
    return -1.0 + beta * float(dx + dy + dz) / 3.0


def _grid(v, dims):
    return v.view(dims[2], dims[1], dims[0])


def _apply(x, dims, beta, theta=None, transpose=False):
    """A x (or A^T x) of a natural-order FP64 vector."""
    nx, ny, nz = dims
    b = -beta if transpose else beta
    xp = torch.nn.functional.pad(_grid(x, dims), (1, 1, 1, 1, 1, 1))
    y = 26.0 * x if theta is None else 26.0 * theta * x
    y = _grid(y.clone(), dims)
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                if dx or dy or dz:
                    y += _coef(b, dx, dy, dz) * xp[1 + dz:1 + dz + nz, 1 + dy:1 + dy + ny,
                                                   1 + dx:1 + dx + nx]
    return y.reshape(-1)


def _phase(zp, r, dims, beta, colour):
    """One Gauss-Seidel colour phase on the padded grid zp (coordinates with
    the colour's bit set are even)."""
    st = [1 - ((colour >> a) & 1) for a in range(3)]
    n = [(dims[a] - st[a] + 1) // 2 for a in range(3)]
    if min(n) < 1:
        return

    def at(dx, dy, dz):
        s = [slice(1 + st[a] + d, 1 + st[a] + d + 2 * n[a] - 1, 2)
             for a, d in enumerate((dx, dy, dz))]
        return zp[s[2], s[1], s[0]]

    acc = r[st[2]::2, st[1]::2, st[0]::2].clone()
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                if dx or dy or dz:
                    acc -= _coef(beta, dx, dy, dz) * at(dx, dy, dz)
    at(0, 0, 0).copy_(acc / 26.0)


def _sweeps(r, z, dims, beta, count):
    """`count` symmetric sweeps on z; natural order."""
    zp = torch.nn.functional.pad(_grid(z, dims), (1, 1, 1, 1, 1, 1))
    rg = _grid(r, dims)
    for _ in range(count):
        for c in list(range(8)) + list(range(6, -1, -1)):
            _phase(zp, rg, dims, beta, c)
    return zp[1:-1, 1:-1, 1:-1].reshape(-1)


def _vcycle(r, dims, beta, levels):
    z = _sweeps(r, torch.zeros_like(r), dims, beta, 1)
    if levels == 1 or any(d % 2 for d in dims):
        return z
    half = [d // 2 for d in dims]
    d = _grid(r - _apply(z, dims, beta), dims)
    zc = _vcycle(d[::2, ::2, ::2].reshape(-1), half, beta, levels - 1)
    z = z.clone()
    _grid(z, dims)[::2, ::2, ::2] += _grid(zc, half)
    return _sweeps(r, z, dims, beta, 1)


def _storage(v, dims):
    """A natural-order vector in the documented colour-blocked storage order."""
    g = _grid(v, dims)
    out = []
    for c in range(8):
        st = [1 - ((c >> a) & 1) for a in range(3)]
        blk = g[st[2]::2, st[1]::2, st[0]::2].reshape(-1)
        out += [blk, blk.new_zeros(-blk.numel() % 32)]
    return torch.cat(out)


# ------------------------------------------------------------------- the cases
def _dims(case):
    return (case["nx"], case["ny"], case["nz"])


def _count(case):
    return case["nx"] * case["ny"] * case["nz"]


def _dtype(case):
    return torch.float64 if case["prec"] == "fp64" else torch.float32


def _systems(case):
    return [BATCH_EDGES[(case["first"] + i) % 5] for i in range(case["systems"])]


def _normal(gen, *shape):
    return torch.randn(*shape, dtype=torch.float64, device=DEV, generator=gen)


def _inputs(case, seed):
    """The vectors of a case, natural order, FP64 on the GPU, from the seed."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    op = case["op"]
    if op == "bsolve":
        # right-hand sides of about N(0, 1)
        return [[_normal(gen, e ** 3) / 26.0 for _ in range(case["nrhs"])]
                for e in _systems(case)]
    n = _count(case)
    if op == "vbatch":
        return _normal(gen, case["nrhs"], n).to(torch.float32)
    if op == "solve":
        # b = A * 1 + noise of about 1e-3
        return 1.0 + _normal(gen, n) * (1e-3 / 26.0)
    if op == "adjoint":
        theta = 0.9 + 0.2 * torch.rand(n, dtype=torch.float64, device=DEV, generator=gen)
        return theta, _normal(gen, n) / 26.0, _normal(gen, n) / 13.0
    r = _normal(gen, n).to(_dtype(case))
    return (r, _normal(gen, n).to(_dtype(case))) if op == "smooth" else r


def prepare(case, seed):
    op = case["op"]
    v = _inputs(case, seed)
    if op == "bsolve":
        probs = [hpg.Problem(e, e, e, beta=case["beta"]) for e in _systems(case)]
        Bs = [torch.stack([_apply(x, (e, e, e), case["beta"]) for x in xs])
              for e, xs in zip(_systems(case), v)]
        return {"case": case, "Bs": Bs, "probs": probs,
                "solver": batch.BatchSolver(probs, case["nrhs"], restart=case["restart"])}
    dims = _dims(case)
    if op == "adjoint":
        theta, x, lam = v
        b = _apply(x, dims, case["beta"], theta)
        # dL/dx = 2 (x - target) = A^T lam
        target = x - 0.5 * _apply(lam, dims, case["beta"], theta, transpose=True)
        return {"case": case, "b": b, "theta": theta, "target": target}
    p = hpg.Problem(*dims, beta=case["beta"], levels=case["levels"])
    if op == "solve":
        return {"case": case, "p": p, "b": _apply(v, dims, case["beta"])}
    if op == "vbatch":
        st = torch.empty(p.n_store(), case["nrhs"], dtype=torch.float32, device=DEV)
        batch.permute_batch(p.h, 0, 0, case["nrhs"], v, st)
        return {"case": case, "p": p, "r": st}
    if op == "smooth":
        return {"case": case, "p": p, "r": p.to_storage(v[0]), "z": p.to_storage(v[1])}
    return {"case": case, "p": p, "r": p.to_storage(v)}


def run(state):
    case = state["case"]
    op = case["op"]
    if op == "spmv":
        return state["p"].spmv(state["r"])
    if op == "vcycle":
        return state["p"].vcycle(state["r"])
    if op == "smooth":
        return state["p"].smooth(state["r"], state["z"].clone(), sweeps=case["sweeps"])
    if op == "vbatch":
        z = torch.empty_like(state["r"])
        batch.vcycle_batch(state["p"].h, 0, state["r"], z)
        return z
    if op == "solve":
        basis = BASES[case["basis"]]
        inner = hpg.HPG_FP64 if case["basis"] == "fp64" else hpg.HPG_FP32
        x, _ = state["p"].solve(state["b"], tol=case["tol"], restart=case["restart"],
                                inner=inner, basis=basis)
        return x
    if op == "bsolve":
        Xs = [torch.zeros_like(b) for b in state["Bs"]]
        state["solver"].solve(state["Bs"], Xs, tol=case["tol"])
        return Xs
    b = state["b"].detach().requires_grad_()
    theta = state["theta"].detach().requires_grad_()
    x = adjoint.solve(b, theta, _dims(case), beta=case["beta"], tol=case["tol"],
                      levels=case["levels"])
    ((x - state["target"]) ** 2).sum().backward()
    return {"x": x.detach(), "grad_b": b.grad, "grad_theta": theta.grad}


def exact(case, seed):
    op = case["op"]
    v = _inputs(case, seed)
    if op == "bsolve":
        return [torch.stack(xs) for xs in v]
    if op == "solve":
        return v
    if op == "adjoint":
        _, x, lam = v
        return {"x": x, "grad_b": lam, "grad_theta": -26.0 * lam * x}
    dims, beta = _dims(case), case["beta"]
    if op == "spmv":
        return _storage(_apply(v.double(), dims, beta), dims)
    if op == "vcycle":
        return _storage(_vcycle(v.double(), dims, beta, case["levels"]), dims)
    if op == "smooth":
        return _storage(_sweeps(v[0].double(), v[1].double(), dims, beta, case["sweeps"]), dims)
    return torch.stack([_storage(_vcycle(r.double(), dims, beta, case["levels"]), dims)
                        for r in v], dim=1)


def _vcycle_flops(dims, levels):
    """Two symmetric sweeps (15 of 16 half-sweep phases each), the residual at
    the coarse points and the correction per level; one sweep on the last."""
    total = 0.0
    for l in range(levels):
        n = dims[0] * dims[1] * dims[2]
        last = l == levels - 1 or any(d % 2 for d in dims)
        total += (1 if last else 2) * (15.0 / 8.0) * 53.0 * n + (0.0 if last else 55.0 * n / 8.0)
        if last:
            return total
        dims = [d // 2 for d in dims]
    return total


def work(case):
    """Bytes: the operator is defined by its grid, beta and theta, so a pass
    reads its input vectors once and writes its result once; a solve also
    streams the Krylov basis that its inner steps span (three times per step,
    as classical Gram-Schmidt with reorthogonalisation needs)."""
    op = case["op"]
    if op == "bsolve":
        bytes_ = flops = 0.0
        for e in _systems(case):
            c = _case("solve", (e, e, e), basis="fp32", restart=case["restart"], tol=case["tol"])
            w = work(c)
            bytes_ += w["bytes"] * case["nrhs"]
            flops += w["flops"] * case["nrhs"]
        return {"bytes": bytes_, "flops": flops}
    n, dims = float(_count(case)), _dims(case)
    if op in ("spmv", "smooth", "vcycle"):
        s = 8 if case["prec"] == "fp64" else 4
        if op == "spmv":
            return {"bytes": 2 * s * n, "flops": 54 * n}
        if op == "smooth":
            return {"bytes": 3 * s * n, "flops": case["sweeps"] * (15.0 / 8.0) * 53 * n}
        return {"bytes": 2 * s * n, "flops": _vcycle_flops(dims, case["levels"])}
    if op == "vbatch":
        return {"bytes": 2 * 4 * n * case["nrhs"],
                "flops": case["nrhs"] * _vcycle_flops(dims, case["levels"])}
    # inner steps to the tolerance grow about linearly with the mean edge
    steps = (0.14 if op == "solve" else 0.16) * n ** (1 / 3) * -math.log10(case["tol"]) + 4
    m = min(steps, case.get("restart", 30))
    q = {"fp64": 8, "fp32": 4}.get(case.get("basis", "fp32"), 2)
    s = 8 if q == 8 else 4
    step_bytes = n * (3 * q * m / 2 + 8 * s)
    step_flops = _vcycle_flops(dims, case["levels"]) + 54 * n + 8 * n * m / 2
    k = 2 if op == "adjoint" else 1
    return {"bytes": k * (steps * step_bytes + 24 * n), "flops": k * steps * step_flops}
