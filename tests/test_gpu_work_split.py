"""How the assembly shares its work out (columns per TRSM warp, CTAs per
SYRK task) follows the batch's sizes, and must not show in the results: every
entry of Y and of F is one chain of operations in a fixed order, so a
subdomain alone (narrow parts, shared tasks) and among many (wide parts, one CTA
per task) gives the same bits."""
import numpy as np
import pytest

import oracle
import synth
from paper_2509_21037_gb300 import abi, host, sc

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _subdomains(name):
    if name == "single":                       # one multiplier, and a whole chunk of a chain
        return [synth.chain_1d(40, [40]), synth.chain_1d(70, list(range(1, 33)))]
    if name == "square":
        return synth.single_heat_2d(21).subdomains          # 84 columns: a ragged last chunk
    if name == "cubes":
        return synth.cube_heat_3d(parts=2, k=7).subdomains  # supernodes of 64 columns
    return synth.elasticity_cubes((2, 2, 1), 3, 6, 5).subdomains


@pytest.mark.parametrize("digits,bound", [(0, 1e-12), (7, 1e-12), (5, 1.8e-9)])   # test_gpu_parity's and test_gpu_fullsize's bounds
@pytest.mark.parametrize("name", ["single", "square", "cubes", "elasticity"])
def test_the_split_of_the_work_does_not_show(name, digits, bound):
    subs = _subdomains(name)
    fs = host.factorize_problem(subs)
    n_dual = 1 + max(int(f.lambda_map.max()) for f in fs)
    Fo = oracle.dual_operators(subs)
    copies = 400 // len(fs) + 1

    def assemble(batch, **kw):
        plan = sc.Plan(batch, n_dual, precision=int(digits > 0), n_slices=digits, **kw).upload("cuda")
        F = plan.new_F("cuda")
        F.fill_(float("nan"))
        plan.assemble(torch.from_numpy(sc.concat_L_values(batch)).cuda(), F)
        assert plan.device_status() == abi.SC_OK
        return plan, F

    many, Fm = assemble(fs * copies)
    queue, Fq = assemble(fs * copies, persistent=True)
    assert torch.equal(Fm, Fq)
    for i, f in enumerate(fs):
        one, F1 = assemble([f])
        a, b = (int(many.F_offsets[k]) for k in (i, i + 1))
        assert torch.equal(F1, Fm[a:b])
        last = int(many.F_offsets[-1]) - int(many.F_offsets[len(fs)]) + a
        assert torch.equal(F1, Fm[last:last + b - a])
        assert oracle.relative_frobenius(one.export(F1, 0).cpu().numpy(), Fo[i]) <= bound
