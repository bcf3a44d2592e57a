"""The split-precision TRSM on factors whose rows differ by hundreds of orders of magnitude: L(r, p) / L(p, p) may leave
FP64's range although no product of the substitution does, because the column is zero at p or small there."""
import numpy as np
import pytest

from paper_2509_21037_gb300 import abi, host, sc

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _dense(n, glued, exponents, seeds):
    """A dense factor (one supernode) with its rows scaled by powers of two, right-hand sides e_j times a seed."""
    rng = np.random.default_rng(n)
    A = np.tril(rng.uniform(-1, 1, (n, n))) / n + np.diag(1 + rng.random(n))
    D = np.ldexp(1.0, exponents)
    colptr = np.cumsum([0] + [n - c for c in range(n)]).astype(np.int64)
    rowind = np.concatenate([np.arange(c, n) for c in range(n)]).astype(np.int32)
    L = host.HostFactor(n, colptr, rowind, np.concatenate([(A[c:, c] * D[c:]) for c in range(n)]),
                        np.arange(n, dtype=np.int32))
    m = len(glued)
    f = host.FactoredSubdomain(L, np.arange(m + 1, dtype=np.int32), np.array(glued, np.int32), np.ones(m, np.int8),
                               np.arange(m, dtype=np.int32), bt_val=np.array(seeds))
    # Y of the scaled factor is Y of A times seed / D[glued]: column by column, rows unchanged
    E = np.zeros((n, m))
    E[glued, np.arange(m)] = 1.0
    Y = np.linalg.solve(A, E) * (np.array(seeds) / D[glued])
    return f, Y.T @ Y


@pytest.mark.parametrize("digits,bound", [(7, 1e-12), (6, 5e-10), (5, 1.8e-9), (3, 1.2e-4)])
@pytest.mark.parametrize("case", ["above", "below"])
@pytest.mark.parametrize("n", [12, 40])
@pytest.mark.parametrize("copies", [1, 400])                # two and four columns to a warp
def test_row_scales(n, case, copies, digits, bound):
    glued = [n // 2, n - 1]
    up = np.arange(n) >= n // 2
    if case == "above":       # zero rows of 2^-540 over rows of 2^500
        f, F = _dense(n, glued, np.where(up, 500, -540), [1.0, 1.0])
    else:                     # rows of 2^540 over rows of 2^-500, the right-hand side as large as its rows
        glued = [1, n - 1]
        f, F = _dense(n, glued, np.where(up, -500, 540), [2.0 ** 540, 2.0 ** -500])
    plan = sc.Plan([f] * copies, 2, precision=1, n_slices=digits).upload("cuda")
    G = plan.new_F("cuda")
    plan.assemble(torch.from_numpy(sc.concat_L_values([f] * copies)).cuda(), G)
    assert plan.device_status() == abi.SC_OK
    scale = 2.0 ** 1000 if case == "above" else 1.0
    for i in (0, copies - 1):
        got = plan.export(G, i).cpu().numpy()
        # 7 and 5 digits: test_gpu_work_split's bounds; else 2^(-8 S) times the same factor 2e3
        assert np.linalg.norm(got * scale - F * scale) <= bound * np.linalg.norm(F * scale)
