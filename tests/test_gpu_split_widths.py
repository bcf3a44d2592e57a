"""The split-precision TRSM takes 8 columns, 16 or the whole chunk of 32 to a CTA by the batch's sizes: the same bits from
all three, and from the oracle what the digits promise."""
import numpy as np
import pytest

import oracle
import plan_emulator as pe
import synth
from paper_2509_21037_gb300 import abi, host, sc

SLOTS = 4 * 152


def _width(plan):
    """Columns per warp of the plan's one variant group (the planner's rule, from the exported tables)."""
    T = pe.export_plan(plan)
    cost, width, below = [], 0.0, 0.0
    for t in T["trsm"]:
        c = 1e3 * float(t["list_len"])
        for si in T["trsm_list"][t["list_off"]:t["list_off"] + t["list_len"]]:
            s = T["sns"][si]
            for kb in range(0, int(s["ns"]), 32):
                kw, nr = min(32, int(s["ns"]) - kb), int(s["ns"] + s["rs"])
                if min(int(s["jhi"]), int(t["c_lo"] + t["w"]), int(T["cuts"][s["cut_off"] + kb // 32])) > \
                        max(int(s["jlo"]), int(t["c_lo"])):
                    c += 32 * (kw * kw + 2 * kw * (nr - kb - kw))
                    width, below = width + kw, below + kw * (nr - kb - kw)
        cost.append(c)
    r = max(cost) * SLOTS / sum(cost)
    return r, below / width


@pytest.mark.gpu
@pytest.mark.parametrize("digits,bound", [(7, 1e-12), (6, 5e-10), (5, 1.8e-9), (4, 4.7e-7), (3, 1.2e-4)])   # 2^(-8 S) times 2e3, or 1e-12
def test_widths_agree(digits, bound):
    torch = pytest.importorskip("torch")
    # 3000 dofs: separators of up to 300 columns, blocks of one to 32 columns, chunks of 32 and of 24 columns
    subs = synth.elasticity_cubes((2, 2, 1), 9, 9, 1).subdomains[:1]
    fs = host.factorize_problem(subs)
    n_dual = 1 + max(int(f.lambda_map.max()) for f in fs)

    def assemble(batch):
        plan = sc.Plan(batch, n_dual, precision=1, n_slices=digits).upload("cuda")
        F = plan.new_F("cuda")
        F.fill_(float("nan"))
        plan.assemble(torch.from_numpy(sc.concat_L_values(batch)).cuda(), F)
        assert plan.device_status() == abi.SC_OK
        return plan, F

    one, F1 = assemble(fs[:1])
    r, b = _width(one)
    assert r > 4                                              # two columns to a warp
    some, Fs = assemble(fs * 20)
    r, b = _width(some)
    assert r <= 4 and 300 * r > b                             # four
    many, Fm = assemble(fs * 100)
    r, b = _width(many)
    assert max(300 * r, 180) <= b and r <= 1                  # the whole chunk
    n = int(one.F_offsets[1])
    for i in (0, 7, 19):
        assert torch.equal(F1, Fs[i * n:(i + 1) * n]) and torch.equal(F1, Fm[i * n:(i + 1) * n])
    Fo = oracle.dual_operators(subs, refine=1)
    assert oracle.relative_frobenius(many.export(Fm, 99).cpu().numpy(), Fo[0]) <= bound
