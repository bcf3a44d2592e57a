"""The implicit apply's tiered schedule: the pieces' partition on the CPU, the product on the GPU."""
import numpy as np
import pytest

import implicit_emulator as ie
import oracle
import synth
from paper_2509_21037_gb300 import host, implicit, sc

PIECE = np.dtype([("sub", "<i4"), ("lev_lo", "<i4"), ("n_lev", "<i4"), ("s_lo", "<i4"), ("s_hi", "<i4"), ("pad", "<i4")])


def _problem(name):
    if name == "small":           # a few dofs each: one tier
        return synth.cube_heat_3d(parts=2, k=3)
    if name == "squares":         # deep trees of supernodes of one to four columns
        return synth.mixed_batch((3, 2), (20, 64), (2, 1, 1), (2, 2), 3)
    if name == "cube":            # separators of 81 columns, small subtrees that share pieces
        return synth.cube_heat_3d(parts=2, k=8)
    # separators of 33 .. 300 columns, the last block of 32 not full
    return synth.elasticity_cubes((2, 2, 1), 5, 9, 4)


NAMES = ["small", "squares", "cube", "elasticity"]


@pytest.mark.parametrize("name", NAMES)
def test_pieces_partition_the_tree(name):
    """Every level of every subdomain lies in one piece and every scatter entry in the piece of its row;
    pieces of one tier share no rows and update rows of their own or of later tiers only."""
    prob = _problem(name)
    fs = host.factorize_problem(prob.subdomains)
    ip = implicit.ImplicitPlan(fs, prob.n_dual)
    T = ie.export_plan(ip)
    tail = ip.export_plan()[ie.HEADER.itemsize:ie.HEADER.itemsize + 16].view("<i8")
    pieces = ip.export_plan()[int(tail[0]):int(tail[0]) + int(tail[1]) * PIECE.itemsize].view(PIECE)
    lev, sns = T["levptr"], T["sns"]
    levels = sorted(l for p in pieces for l in range(p["lev_lo"], p["lev_lo"] + p["n_lev"]))
    assert levels == sorted(l for sd in T["subs"] for l in range(sd["lev_lo"], sd["lev_lo"] + sd["n_lev"]))
    entries = sorted(e for p in pieces for e in range(p["s_lo"], p["s_hi"]))
    assert entries == list(range(len(T["sent"])))
    for i, sd in enumerate(T["subs"]):
        owner, start = np.full(int(sd["n"]), -1), {}
        mine = [k for k, p in enumerate(pieces) if p["sub"] == i]
        for k in mine:
            p = pieces[k]
            for s in range(lev[p["lev_lo"]], lev[p["lev_lo"] + p["n_lev"]]):
                c0, ns = int(sns[s]["c0"]), int(sns[s]["ns"])
                assert np.all(owner[c0:c0 + ns] == -1)
                owner[c0:c0 + ns] = k
                start.update({c: l for l in range(p["lev_lo"], p["lev_lo"] + p["n_lev"])
                              for c in range(c0, c0 + ns) if lev[l] <= s < lev[l + 1]})
        for k in mine:
            p = pieces[k]
            assert all(owner[e["r"]] == k for e in T["sent"][p["s_lo"]:p["s_hi"]])
            for s in range(lev[p["lev_lo"]], lev[p["lev_lo"] + p["n_lev"]]):
                sn = sns[s]
                R = T["rows"][sn["rows_off"]:sn["rows_off"] + sn["rs"]]
                # in the piece: a later level; outside: another piece whose levels come later (a later tier)
                assert all(start[int(r)] > start[int(sn["c0"])] for r in R)
                assert all(owner[r] == k or pieces[owner[r]]["lev_lo"] > p["lev_lo"] for r in R)
                assert all(owner[r] == k or owner[r] > k for r in R)     # pieces are stored tier by tier


@pytest.mark.gpu
@pytest.mark.parametrize("name", NAMES)
def test_tiered_product(name):
    torch = pytest.importorskip("torch")
    prob = _problem(name)
    fs = host.factorize_problem(prob.subdomains)
    lam = torch.from_numpy(np.random.default_rng(6).standard_normal(prob.n_dual)).cuda()
    L = torch.from_numpy(sc.concat_L_values(fs)).cuda()
    q = []
    for kw in ({}, {"cluster_min_work": 1 << 60}):           # tiered, and one CTA per subdomain
        ip = implicit.ImplicitPlan(fs, prob.n_dual, **kw).upload("cuda")
        ip.ws.fill_(0xff)                                    # the workspace's contents do not matter
        out = torch.full_like(lam, float("nan"))
        ip.apply(L, lam, out)
        assert ip.device_status() == 0
        q.append(out.cpu().numpy())
    qo = oracle.apply_dual(oracle.dual_operators(prob.subdomains, refine=1), [s.lambda_map for s in prob.subdomains],
                           lam.cpu().numpy(), prob.n_dual)
    for v in q:
        assert np.linalg.norm(v - qo) <= 1e-12 * np.linalg.norm(qo)      # test_gpu_implicit's bound
