"""Batches of so many tiles that the fixed-point products hand their runs out in rounds (64 tiles and more to every
resident warp): just below the line, just above it, and three rounds."""
import dataclasses

import numpy as np
import pytest

import synth
from paper_2509_21037_gb300 import host, sc

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
WARPS = 152 * 6 * 4                              # resident warps of the fixed-point kernel


@pytest.mark.parametrize("per_warp", [63.9, 64.1, 97.0])
def test_rounds_of_runs(per_warp):
    f = host.factorize_problem(synth.elasticity_cubes((2, 2, 2), 8, 8, 1).subdomains)[0]
    nt = -(-f.m // 32)
    count = int(per_warp * WARPS / (nt * (nt + 1) // 2))
    fs = [dataclasses.replace(f, lambda_map=(np.arange(f.m) + (i % 16) * f.m).astype(np.int32)) for i in range(count)]
    n_dual = 16 * f.m
    plan = sc.Plan(fs, n_dual).upload("cuda")
    tiles = int(plan.sizes.F_doubles) // 1024
    # tiles per resident warp: below two rounds of 32, or from there on
    assert (tiles // WARPS >= 64) == (per_warp > 64)
    gen = torch.Generator(device="cuda").manual_seed(3)
    F = torch.randn(int(plan.sizes.F_doubles), dtype=torch.float64, device="cuda", generator=gen)
    lam = torch.randn(n_dual, dtype=torch.float64, device="cuda", generator=gen)
    want, q = torch.empty_like(lam), torch.empty_like(lam)
    plan.apply(F, lam, want)
    # test_gpu_apply_digits's bound between two products of the same F
    for quarters in (0, 1, 2):
        q.fill_(float("nan"))
        plan.apply_mixed(F, lam, q, fp64_quarters=quarters)
        assert float((q - want).norm() / want.norm()) <= 1e-14
