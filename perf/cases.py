"""The workloads this framework is timed on: assembling the subdomains' dual operators F_i and applying them.

A case names a problem (`problem` and its sizes, built by `synth` and factorised on the host, as the README's
example does) and what the program does with it (`call`):

  step      Plan.assemble, then one Plan.apply: the numeric stage after new values, in FP64 or with `digits` 8-bit digits on
            the tensor cores (`digits` = 0: FP64; -1: a variant per subdomain, as the learned selector picks them)
  apply     one product q = F lambda of a dual solver's iteration; `form`: "fp64", "fixed", "mixed" or "digits" (from the
            digit form that the program keeps beside F)
  refresh   Plan.prepare_digits, then Plan.apply_digits: the first product after an assembly
  implicit  ImplicitPlan.apply: the same product by two sparse triangular solves, without F

Problems: "heat2d" (k x k squares on a lattice, sizes drawn between kmin and kmax; a 1 x 1 lattice is the single square
whose boundary nodes are all glued), "heat3d" (a cube cut into parts^3 subdomains of k^3 elements), "elasticity" (uneven
cubes on a lattice) and "mixed" (squares and elasticity cubes in one batch).
"""
import functools
import math

import numpy as np
import torch

import synth
from paper_2509_21037_gb300 import host, implicit, sc

DEV = "cuda"


def listed():
    square = {"problem": "heat2d", "nx": 1, "ny": 1, "kmin": 16, "kmax": 16, "mesh": 0}
    squares = {"problem": "heat2d", "nx": 6, "ny": 6, "kmin": 32, "kmax": 96, "mesh": 0}
    cube = {"problem": "heat3d", "parts": 4, "k": 16}
    cubes = {"problem": "elasticity", "nx": 2, "ny": 2, "nz": 2, "kmin": 8, "kmax": 16, "mesh": 1}
    lattice = {"problem": "elasticity", "nx": 4, "ny": 4, "nz": 4, "kmin": 8, "kmax": 16, "mesh": 0}
    mixed = {"problem": "mixed", "nx": 4, "ny": 4, "nz": 1, "kmin": 32, "kmax": 96, "k3min": 8, "k3max": 14, "mesh": 0}
    return [
        # one small subdomain: what a first try or a coarse model costs, all latency
        {"name": "step_square", "call": "step", "digits": 0, **square},
        # a plane domain cut into uneven squares: sparse factors, few multipliers per subdomain
        {"name": "step_squares", "call": "step", "digits": 0, **squares},
        # the benchmark's batch: 64 floating subdomains of a 3D heat cube, FP64
        {"name": "step_cube", "call": "step", "digits": 0, **cube},
        # a few uneven elasticity subdomains: three multipliers per glued node, long supernodes
        {"name": "step_elasticity", "call": "step", "digits": 0, **cubes},
        # the benchmark's batch in split precision at the FP64 path's accuracy
        {"name": "step_cube_7digits", "call": "step", "digits": 7, **cube},
        # a mixed batch with a variant per subdomain: FP64, 7 and 5 digits side by side
        {"name": "step_mixed_variants", "call": "step", "digits": -1, **mixed},
        # a dual solver's iteration on the assembled operators, FP64
        {"name": "apply_cube", "call": "apply", "form": "fp64", **cube},
        # the same without a digit form, tiles split between the FP64 and the integer pipes
        {"name": "apply_elasticity_mixed", "call": "apply", "form": "mixed", **lattice},
        # the solver's default product, from the digit form, on operators far larger than L2
        {"name": "apply_elasticity_digits", "call": "apply", "form": "digits", **lattice},
        # a solver that gets a new F for every few products: the digit form is made again
        {"name": "refresh_cube", "call": "refresh", **cube},
        # the operator without assembly: too few iterations to pay for it
        {"name": "implicit_cube", "call": "implicit", **cube},
        # the same on subdomains of very different sizes and depths
        {"name": "implicit_mixed", "call": "implicit", **mixed},
    ]


def _log(rng, lo, hi):
    """A whole number between lo and hi, spread over their logarithm."""
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo - 0.49), math.log(hi + 0.49))))))


def draw(rng):
    kind = rng.choice(("heat2d", "heat3d", "elasticity", "mixed"))
    c = {"problem": kind}
    if kind == "heat2d":
        lo = _log(rng, 4, 64)
        c.update(nx=rng.randint(1, 6), ny=rng.randint(1, 6), kmin=lo, kmax=rng.randint(lo, min(96, 3 * lo)))
    elif kind == "heat3d":
        c.update(parts=rng.randint(2, 4), k=_log(rng, 3, 16))
    elif kind == "elasticity":
        lo = _log(rng, 3, 12)
        c.update(nx=2, ny=rng.randint(1, 2), nz=rng.randint(1, 2), kmin=lo, kmax=rng.randint(lo, min(15, 2 * lo)))
    else:
        lo, lo3 = _log(rng, 8, 64), _log(rng, 3, 10)
        c.update(nx=rng.randint(2, 4), ny=rng.randint(1, 4), nz=1, kmin=lo, kmax=rng.randint(lo, min(96, 3 * lo)),
                 k3min=lo3, k3max=rng.randint(lo3, min(14, 2 * lo3)))
    if kind != "heat3d":
        c["mesh"] = rng.randint(0, 10 ** 6)
    c["call"] = rng.choice(("step", "step", "step", "apply", "apply", "refresh", "implicit", "implicit"))
    if c["call"] == "step":
        c["digits"] = rng.choice((0, 0, 5, 6, 7, -1))
    if c["call"] == "apply":
        c["form"] = rng.choice(("fp64", "fixed", "mixed", "digits", "digits"))
    return c


# ---- the problem: meshes, gluing and host factors (the same for every seed; kept, as a program keeps its mesh) ----

_FACTORS = {}


def _sizes(rng, count, lo, hi):
    return [rng.randint(lo, hi) for _ in range(count)]


def _mesh(c):
    if c["problem"] == "heat3d":
        return synth.cube_heat_3d(c["parts"], c["k"])
    if c["problem"] == "elasticity":
        return synth.elasticity_cubes((c["nx"], c["ny"], c["nz"]), c["kmin"], c["kmax"], c["mesh"])
    if c["problem"] == "mixed":
        return synth.mixed_batch((c["nx"], c["ny"]), (c["kmin"], c["kmax"]), (c["nx"], 2, c["nz"]),
                                 (c["k3min"], c["k3max"]), c["mesh"])
    if c["nx"] * c["ny"] == 1:
        return synth.single_heat_2d(c["kmin"])
    # the squares of a mixed batch, without its cubes
    both = synth.mixed_batch((c["nx"], c["ny"]), (c["kmin"], c["kmax"]), (2, 1, 1), (3, 3), c["mesh"])
    subs = [s for s in both.subdomains if s.ndpn == 1]
    return synth.Problem("squares", subs, 1 + max(int(s.lambda_map.max()) for s in subs), c["mesh"])


@functools.lru_cache(maxsize=32)
def _problem(key):
    p = _mesh(dict(key))
    new = {s.key: s for s in p.subdomains if s.key not in _FACTORS}
    for s, f in zip(new.values(), host.factorize_problem(list(new.values())) if new else []):
        _FACTORS[s.key] = f.L
    fs = [host.permute_bt(s, _FACTORS[s.key]) for s in p.subdomains]
    # a variant per subdomain as the learned selector picks them: FP64 for small ones, 5 digits for most, 7 for some
    slices = [0 if s.ndpn == 1 and max(s.grid) <= 64 else 7 if i % 6 == 5 else 5 for i, s in enumerate(p.subdomains)]
    return fs, p.n_dual, slices


def _of(case):
    return _problem(tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "call", "digits", "form"))))


def _plan(case):
    fs, n_dual, slices = _of(case)
    digits = case.get("digits", 0)
    if digits < 0:
        return sc.Plan(fs, n_dual, sub_slices=slices)
    return sc.Plan(fs, n_dual, precision=1 if digits else 0, n_slices=digits)


# ---- the inputs, from the seed alone ----

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _lambda(case, seed):
    return torch.randn(_of(case)[1], dtype=torch.float64, device=DEV, generator=_gen(seed))


def _factors(case, seed):
    """Values of all L_i: every subdomain has its own conductivity or stiffness, log-uniform in [1/2, 2]."""
    fs = _of(case)[0]
    coef = np.exp2(np.random.default_rng(seed).uniform(-1.0, 1.0, len(fs)))
    L = torch.from_numpy(sc.concat_L_values(fs)).to(DEV)
    at = 0
    for f, c in zip(fs, coef):
        L[at:at + f.L.nnz] *= math.sqrt(c)
        at += f.L.nnz
    return L


def _tiles(case):
    """Of every stored 32 x 32 tile, in the order of F: subdomain, I, J."""
    sub, I, J = [], [], []
    for i, f in enumerate(_of(case)[0]):
        r, c = np.tril_indices((f.m + 31) // 32)
        sub.append(np.full(len(r), i)), I.append(r), J.append(c)
    return tuple(torch.from_numpy(np.concatenate(x)).to(DEV) for x in (sub, I, J))


def _operators(case, seed):
    """Operators F_i in their packed layout: symmetric, the tiles falling off away from the diagonal."""
    sub, I, J = _tiles(case)
    T = torch.randn((len(I), 32, 32), dtype=torch.float64, device=DEV, generator=_gen(seed + 1))   # [tile][column][row]
    T /= (1.0 + (I - J).double())[:, None, None]
    on = I == J
    T[on] = T[on] + T[on].transpose(1, 2)
    T[on] += 8.0 * torch.eye(32, dtype=torch.float64, device=DEV)
    m = torch.tensor([f.m for f in _of(case)[0]], device=DEV)[sub]
    at = torch.arange(32, device=DEV)
    T *= (32 * J[:, None] + at < m[:, None])[:, :, None]
    T *= (32 * I[:, None] + at < m[:, None])[:, None, :]
    return T.reshape(-1)


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.call, s.form = case["call"], case.get("form")
    s.lam = _lambda(case, seed)
    s.q = torch.empty_like(s.lam)
    if s.call == "implicit":
        fs, n_dual, _ = _of(case)
        s.plan = implicit.ImplicitPlan(fs, n_dual).upload(DEV)
        s.L = _factors(case, seed)
        return s
    s.plan = _plan(case).upload(DEV)
    if s.call == "step":
        s.L = _factors(case, seed)
        s.F = s.plan.new_F(DEV)
    else:
        s.F = _operators(case, seed)
        s.Fd = s.plan.prepare_digits(s.F) if s.call == "refresh" or s.form == "digits" else None
    return s


def run(s):
    if s.call == "step":
        s.plan.assemble(s.L, s.F)
        s.plan.apply(s.F, s.lam, s.q)
        return {"F": s.F, "q": s.q}
    if s.call == "implicit":
        s.plan.apply(s.L, s.lam, s.q)
        return {"q": s.q}
    if s.call == "refresh":
        s.plan.prepare_digits(s.F, s.Fd)
    if s.call == "refresh" or s.form == "digits":
        s.plan.apply_digits(s.Fd, s.lam, s.q)
    elif s.form == "fixed":
        s.plan.apply_fixed(s.F, s.lam, s.q)
    elif s.form == "mixed":
        s.plan.apply_mixed(s.F, s.lam, s.q, fp64_quarters=1)
    else:
        s.plan.apply(s.F, s.lam, s.q)
    return {"q": s.q}


def work(case):
    fs, n_dual, _ = _of(case)
    nnz, stored = sum(f.L.nnz for f in fs), sum(f.m * (f.m + 1) // 2 for f in fs)
    if case["call"] == "implicit":
        # L's values once (both solves), lambda and q; a multiply-add per entry and solve
        return {"bytes": 8 * nnz + 16 * n_dual, "flops": 4 * nnz}
    if case["call"] == "step":
        # L in and F out, F's useful arithmetic as the plan counts it, and the product on F
        st = _plan(case).stats
        return {"bytes": 8 * nnz + 8 * stored + 16 * n_dual, "flops": st.flops_trsm + st.flops_syrk + 4 * stored}
    return {"bytes": 8 * stored + 16 * n_dual, "flops": 4 * stored}


# ---- the same in plain torch, 64 bits ----

def _product(case, T, lam):
    """q = sum_i scatter(F_i gather(lambda)) from the packed tiles T."""
    fs, n_dual, _ = _of(case)
    sub, I, J = _tiles(case)
    first = np.concatenate([[0], np.cumsum([(f.m + 31) // 32 for f in fs])])
    to = np.full((int(first[-1]), 32), n_dual)                       # multiplier of every padded local row
    for f, a in zip(fs, first):
        to[a:].reshape(-1)[:f.m] = f.lambda_map
    to, first = torch.from_numpy(to).to(DEV), torch.from_numpy(first).to(DEV)
    x = torch.cat([lam, lam.new_zeros(1)])[to]
    y = torch.zeros_like(x)
    off = I > J
    T = T.view(-1, 32, 32)
    y.index_add_(0, first[sub] + I, torch.einsum("tcr,tc->tr", T, x[first[sub] + J]))
    y.index_add_(0, (first[sub] + J)[off], torch.einsum("tcr,tr->tc", T[off], x[(first[sub] + I)[off]]))
    return lam.new_zeros(n_dual + 1).index_add_(0, to.reshape(-1), y.reshape(-1))[:n_dual]


def _dense(f, values):
    """L_i and B_i^T as dense matrices."""
    col = torch.from_numpy(np.repeat(np.arange(f.n), np.diff(f.L.colptr))).to(DEV)
    L = torch.zeros((f.n, f.n), dtype=torch.float64, device=DEV)
    L[torch.from_numpy(f.L.rowind.astype(np.int64)).to(DEV), col] = values
    B = torch.zeros((f.n, f.m), dtype=torch.float64, device=DEV)
    at = np.repeat(np.arange(f.m), np.diff(f.bt_colptr))
    B[torch.from_numpy(f.bt_rowind.astype(np.int64)).to(DEV), torch.from_numpy(at).to(DEV)] = \
        torch.from_numpy(f.bt_sign.astype(np.float64)).to(DEV)
    return L, B


def exact(case, seed):
    fs, n_dual, _ = _of(case)
    lam = _lambda(case, seed)
    if case["call"] in ("apply", "refresh"):
        return {"q": _product(case, _operators(case, seed), lam)}
    if sum(f.n * f.n * (f.m if case["call"] == "step" else 64) for f in fs) > 1.2e13:
        return None
    values = _factors(case, seed)
    tiles, at, q = [], 0, torch.zeros(n_dual, dtype=torch.float64, device=DEV)
    for f in fs:
        if f.m:
            L, B = _dense(f, values[at:at + f.L.nnz])
            if case["call"] == "implicit":
                to = torch.from_numpy(f.lambda_map.astype(np.int64)).to(DEV)
                y = torch.linalg.solve_triangular(L, (B @ lam[to])[:, None], upper=False)
                q.index_add_(0, to, (B.T @ torch.linalg.solve_triangular(L.T, y, upper=True))[:, 0])
            else:
                Y = torch.linalg.solve_triangular(L, B, upper=False)
                nt = (f.m + 31) // 32
                A = torch.zeros((32 * nt, 32 * nt), dtype=torch.float64, device=DEV)
                A[:f.m, :f.m] = Y.T @ Y
                I, J = torch.tril_indices(nt, nt, device=DEV)
                tiles.append(A.view(nt, 32, nt, 32).permute(0, 2, 3, 1)[I, J].reshape(-1))
        at += f.L.nnz
    if case["call"] == "implicit":
        return {"q": q}
    F = torch.cat(tiles)
    return {"F": F, "q": _product(case, F, lam)}
