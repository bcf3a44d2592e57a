"""The branches of the tiered implicit product that small batches do not reach: pieces with more supernodes than
shared memory holds, with more levels, tiers with more pieces than SMs and separators of more than 32 columns
in them, and trees cut into several tiers.  The plan is checked on the CPU to have what the case is for."""
import dataclasses
import functools

import numpy as np
import pytest

import implicit_emulator as ie
import synth
from paper_2509_21037_gb300 import host, implicit, sc
from test_implicit_tiers import PIECE

SMEM_SNS, SMEM_LEVELS, SMS = 768, 63, 152        # kTierSns, kTierLevs, kCtaSlots in sc_implicit.cu


def _chain(n, seed):
    """A tridiagonal factor in its natural order: n - 1 supernodes, one to a level, glued at both ends."""
    rng = np.random.default_rng(seed)
    colptr = np.minimum(2 * np.arange(n + 1), 2 * n - 1).astype(np.int64)
    rowind = np.stack([np.arange(n), np.arange(n) + 1], 1).reshape(-1)[:2 * n - 1].astype(np.int32)
    values = np.stack([1.0 + rng.random(n), rng.uniform(-1, 1, n)], 1).reshape(-1)[:2 * n - 1].copy()
    L = host.HostFactor(n, colptr, rowind, values, np.arange(n, dtype=np.int32))
    return host.FactoredSubdomain(L, np.array([0, 1, 2, 3], np.int32), np.array([0, n // 2, n - 1], np.int32),
                                  np.array([1, -1, 1], np.int8), np.arange(3, dtype=np.int32))


def _star(leaves, seed):
    """One-column supernodes without children under a root of three columns: two levels, every leaf glued."""
    rng = np.random.default_rng(seed)
    cols = [[c, leaves, leaves + 1, leaves + 2] for c in range(leaves)] + \
           [list(range(leaves + k, leaves + 3)) for k in range(3)]
    colptr = np.cumsum([0] + [len(c) for c in cols]).astype(np.int64)
    rowind = np.concatenate(cols).astype(np.int32)
    values = rng.uniform(-1, 1, len(rowind)) / leaves
    values[colptr[:-1]] = 1.0 + rng.random(len(cols))
    L = host.HostFactor(leaves + 3, colptr, rowind, values, np.arange(leaves + 3, dtype=np.int32))
    m = 7
    rows = [np.arange(j, leaves, m, dtype=np.int32) for j in range(m)]
    ptr = np.cumsum([0] + [len(r) for r in rows]).astype(np.int32)
    sign = rng.choice(np.array([-1, 1], np.int8), leaves)
    return host.FactoredSubdomain(L, ptr, np.concatenate(rows), sign, np.arange(m, dtype=np.int32))


def _copies(f, count):
    return [dataclasses.replace(f, lambda_map=(f.lambda_map * 0 + np.arange(f.m) + i * f.m).astype(np.int32))
            for i in range(count)]


@functools.lru_cache(maxsize=None)
def _batch(name):
    if name == "long":             # 200 levels of one supernode, descriptors in shared memory
        return [_chain(201, 1)]
    if name == "longer":           # and 899: neither fits
        return [_chain(900, 2)]
    if name == "many":             # more supernodes than shared memory holds, few levels, two CTAs to an SM
        return _copies(_star(1000, 3), 400)
    if name == "wide":             # separators of 147 columns and, two to a level, of 63; two CTAs to an SM
        return _copies(host.factorize_problem(synth.elasticity_cubes((2, 2, 2), 6, 6, 1).subdomains)[0], 400)
    return host.factorize_problem(synth.cube_heat_3d(parts=2, k=16).subdomains)      # "tiers"


NAMES = ["long", "longer", "many", "wide", "tiers"]


def _pieces(ip):
    blob = ip.export_plan()
    tail = blob[ie.HEADER.itemsize:ie.HEADER.itemsize + 16].view("<i8")
    return blob[int(tail[0]):int(tail[0]) + int(tail[1]) * PIECE.itemsize].view(PIECE)


@pytest.mark.parametrize("name", NAMES)
def test_the_plan_has_what_the_case_is_for(name):
    fs = _batch(name)
    ip = implicit.ImplicitPlan(fs, 1 + max(int(f.lambda_map.max()) for f in fs))
    T, pieces = ie.export_plan(ip), _pieces(ip)
    sns = [int(T["levptr"][p["lev_lo"] + p["n_lev"]] - T["levptr"][p["lev_lo"]]) for p in pieces]
    levels = int(pieces["n_lev"].max())
    if name == "long":
        assert SMEM_LEVELS < levels and max(sns) <= SMEM_SNS
    elif name == "longer":
        assert SMEM_LEVELS < levels and max(sns) > SMEM_SNS
    elif name == "many":
        assert levels <= SMEM_LEVELS and max(sns) > SMEM_SNS and len(pieces) == len(fs) > SMS
    elif name == "wide":
        assert len(pieces) == len(fs) > SMS
        p = pieces[0]
        per = [T["sns"]["ns"][T["levptr"][l]:T["levptr"][l + 1]] for l in range(p["lev_lo"], p["lev_lo"] + p["n_lev"])]
        assert any((x > 32).sum() == 2 for x in per) and any((x > 64).sum() == 1 for x in per)
    else:
        per_sub = [sum(p["sub"] == i for p in pieces) for i in range(len(fs))]
        assert min(per_sub) > 2 and max(int(x) for x in T["sns"]["ns"]) > 64


def _exact(f, lam):
    """B L^-T L^-1 B^T lambda with the factor as it is, by scipy's sparse triangular solves."""
    import scipy.sparse as sp
    from scipy.sparse.linalg import spsolve_triangular
    L = sp.csc_matrix((f.L.values, f.L.rowind, f.L.colptr), shape=(f.n, f.n))
    B = sp.csc_matrix((f.bt_sign.astype(float), f.bt_rowind, f.bt_colptr), shape=(f.n, f.m))
    y = spsolve_triangular(L.tocsr(), B @ lam, lower=True)
    return B.T @ spsolve_triangular(L.T.tocsr(), y, lower=False)


@pytest.mark.gpu
@pytest.mark.parametrize("name", NAMES)
def test_product(name):
    torch = pytest.importorskip("torch")
    fs = _batch(name)
    n_dual = 1 + max(int(f.lambda_map.max()) for f in fs)
    lam = np.random.default_rng(3).standard_normal(n_dual)
    ip = implicit.ImplicitPlan(fs, n_dual).upload("cuda")
    ip.ws.fill_(0xff)
    q = torch.full((n_dual,), float("nan"), dtype=torch.float64, device="cuda")
    ip.apply(torch.from_numpy(sc.concat_L_values(fs)).cuda(), torch.from_numpy(lam).cuda(), q)
    assert ip.device_status() == 0
    q = q.cpu().numpy()
    want = np.zeros(n_dual)
    memo = {}
    for f in fs[:3] + fs[-2:] if len(fs) > 100 else fs:
        want[f.lambda_map] += _exact(f, lam[f.lambda_map])
        memo.update({int(k): 1 for k in f.lambda_map})
    at = np.array(sorted(memo))
    assert np.all(np.isfinite(q))
    # two solves with the same FP64 factor: each within a few hundred roundings of the exact one (test_gpu_implicit's bound)
    assert np.linalg.norm(q[at] - want[at]) <= 1e-12 * np.linalg.norm(want[at])
