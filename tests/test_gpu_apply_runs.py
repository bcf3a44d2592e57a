"""The explicit products cut the stored tiles into one run per warp: runs of one tile, runs that start and
end inside a row block or a subdomain, more warps than tiles, and an F that is only 8-byte aligned."""
import numpy as np
import pytest

import oracle
import synth
from paper_2509_21037_gb300 import host, sc

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("offset", [0, 1])              # doubles past a 16-byte boundary
@pytest.mark.parametrize("name", ["one", "few", "many"])
def test_runs_of_tiles(name, offset):
    if name == "one":
        subs = [synth.chain_1d(5, [5])]                 # a single tile with one live entry
    elif name == "few":
        subs = synth.mixed_batch((3, 2), (5, 20), (2, 1, 1), (2, 3), 1).subdomains
    else:
        subs = synth.cube_heat_3d(parts=3, k=8).subdomains      # 2000 tiles and more
    fs = host.factorize_problem(subs)
    n_dual = 1 + max(int(f.lambda_map.max()) for f in fs)
    plan = sc.Plan(fs, n_dual).upload("cuda")
    L = torch.from_numpy(sc.concat_L_values(fs)).cuda()
    F = torch.empty(plan.sizes.F_doubles + offset, dtype=torch.float64, device="cuda")[offset:]
    plan.assemble(L, F)
    lam = torch.from_numpy(np.random.default_rng(2).standard_normal(n_dual)).cuda()
    qo = oracle.apply_dual([plan.export(F, i).cpu().numpy() for i in range(plan.nsub)],
                           [f.lambda_map for f in fs], lam.cpu().numpy(), n_dual)
    q = torch.empty_like(lam)
    # an FP64 sum of up to 1700 terms of one sign or the other: well within 1e-14 of the norm (test_gpu_apply_digits's bound)
    for run in [lambda: plan.apply(F, lam, q), lambda: plan.apply_fixed(F, lam, q)] + \
               [lambda k=k: plan.apply_mixed(F, lam, q, fp64_quarters=k) for k in (1, 2, 3, 4)] + \
               [lambda: plan.apply_digits(plan.prepare_digits(F), lam, q)]:
        q.fill_(float("nan"))
        run()
        assert np.linalg.norm(q.cpu().numpy() - qo) <= 1e-14 * np.linalg.norm(qo)
