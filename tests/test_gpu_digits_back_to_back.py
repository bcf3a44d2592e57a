"""The digit-form product is launched while the kernel that writes lambda's digits still runs: calls that follow one
another without a synchronisation, each with another lambda in the same scratch, must each use their own."""
import numpy as np
import pytest

import synth
from paper_2509_21037_gb300 import host, sc

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("name", ["few", "many"])
def test_each_call_uses_its_own_lambda(name, captured):
    prob = synth.cube_heat_3d(parts=2, k=4) if name == "few" else synth.cube_heat_3d(parts=4, k=10)
    fs = host.factorize_problem(prob.subdomains)
    plan = sc.Plan(fs, prob.n_dual).upload("cuda")
    F = plan.new_F("cuda")
    plan.assemble(torch.from_numpy(sc.concat_L_values(fs)).cuda(), F)
    Fd = plan.prepare_digits(F)
    rng = np.random.default_rng(9)
    # magnitudes apart, so that a block of another call's digits is off by many orders
    lams = [torch.from_numpy(rng.standard_normal(prob.n_dual) * 10.0 ** (3 * k)).cuda() for k in (0, 2, -2, 1, -1, 0)]
    want = [torch.empty_like(l) for l in lams]
    got = [torch.full_like(l, float("nan")) for l in lams]
    for l, w in zip(lams, want):
        plan.apply(F, l, w)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())

    def calls():
        for l, g in zip(lams, got):
            plan.apply_digits(Fd, l, g, stream=s)

    if captured:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            calls()
        with torch.cuda.stream(s):
            for _ in range(5):
                g.replay()
    else:
        for _ in range(5):
            calls()
    s.synchronize()
    assert plan.digits_status(Fd) == 0
    for w, g in zip(want, got):      # test_gpu_apply_digits's bound between the two products
        assert float((g - w).norm() / w.norm()) <= 1e-14
