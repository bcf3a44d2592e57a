"""The tables and the sharing of work that the assembly and product kernels use, replayed on the CPU."""
import numpy as np
import pytest

import parts_emulator as pa
import plan_emulator as pe
import synth
from paper_2509_21037_gb300 import host, sc
from test_abi import edge_batch


def _factors(name):
    if name == "holes":           # unglued subdomains first, last and between others
        fs = host.factorize_problem(edge_batch().subdomains)
        assert fs[0].m == 0
        return [fs[0], fs[3], fs[0], fs[0], fs[1], fs[0]]
    if name == "squares":
        return host.factorize_problem(synth.mixed_batch((2, 2), (20, 33), (1, 1, 1), (2, 2), 3).subdomains)
    return host.factorize_problem(synth.cube_heat_3d(parts=2, k=6).subdomains[:2])   # supernodes of up to 49 columns


NAMES = ["holes", "squares", "cubes"]


def _plan(fs, **kw):
    return sc.Plan(fs, 1 + max([int(f.lambda_map.max()) for f in fs if f.m], default=0), **kw)


@pytest.mark.parametrize("name", NAMES)
@pytest.mark.parametrize("digits", [0, 7])
def test_seeds_of_every_column(name, digits):
    fs = _factors(name)
    plan = _plan(fs, precision=int(digits > 0), n_slices=digits)
    T = pe.export_plan(plan)
    seeds = pa.seed_table(plan, T)
    assert len(seeds) == sum(f.m for f in fs) + 1
    assert seeds[0] == 0 and seeds[-1] == len(T["seeds"]) and np.all(np.diff(seeds) >= 0)
    for f, sd in zip(fs, T["subs"]):
        perm = T["perm"][sd["col_off"]:sd["col_off"] + f.m]
        for q in range(f.m):
            e = T["seeds"][seeds[sd["col_off"] + q]:seeds[sd["col_off"] + q + 1]]
            j = perm[q]
            assert np.array_equal(e["value"], f.bt_sign[f.bt_colptr[j]:f.bt_colptr[j + 1]])
    for t in T["trsm"]:
        c = int(T["subs"][t["sub"]]["col_off"]) + int(t["c_lo"])
        assert (seeds[c], seeds[c + t["w"]]) == (t["seed_lo"], t["seed_hi"])


def _assembled(T, plan, Lv):
    invd = np.zeros(int(T["header"]["n_cols"]))
    invd[T["active"]] = 1.0 / Lv[T["lcp"][T["active"]]]
    return invd, pe.emulate_assembly(T, plan.sizes, plan.stats, Lv)


@pytest.mark.parametrize("name", NAMES)
def test_parts_pieces_and_numbered_rows(name):
    """Every width of a part, flat and whole-row updates, and every sharing of the SYRK give the task by task result."""
    fs = _factors(name)
    plan = _plan(fs)
    T, Lv = pe.export_plan(plan), sc.concat_L_values(fs)
    seeds = pa.seed_table(plan, T)
    invd, F = _assembled(T, plan, Lv)
    Ys = {}
    for width in (1, 2, 4, 8, 16):
        Y = np.full(int(plan.stats.y_doubles), np.nan)
        for t in T["trsm"]:
            for lo, hi in pa.part_columns(t, width):
                if lo < hi:
                    pa.trsm_part(T, seeds, t, lo, hi, Lv, invd, Y, flat=width >= 16)
        assert not np.isnan(Y).any()
        Ys[width] = Y
    scale = np.abs(Ys[16]).max()
    assert all(np.abs(Y - Ys[16]).max() <= 1e-13 * scale for Y in Ys.values())     # the same chains, dot products apart
    for ctas in (1, 4, 8):
        for t in T["syrk"]:
            sd = T["subs"][t["sub"]]
            acc = pa.syrk_task(T, t, Ys[2], ctas)
            perm = T["perm"][sd["col_off"]:sd["col_off"] + sd["m"]]
            for r in range(32):
                for c in range(32 if t["q1"] != t["q2"] else r + 1):
                    j1, j2 = 32 * t["q1"] + r, 32 * t["q2"] + c
                    if j1 < sd["m"] and j2 < sd["m"]:
                        hi, lo = max(perm[j1], perm[j2]), min(perm[j1], perm[j2])
                        I, J = hi // 32, lo // 32
                        want = F[sd["F_off"] + (I * (I + 1) // 2 + J) * 1024 + hi % 32 + 32 * (lo % 32)]
                        assert abs(acc[r, c] - want) <= 1e-12 * np.abs(F).max()


@pytest.mark.parametrize("name", NAMES)
def test_units_of_digit_rows(name):
    fs = _factors(name)
    plan = _plan(fs, precision=1, n_slices=7)
    T = pe.export_plan(plan)
    layout = pe.check_split_layout(T, plan.sizes, plan.stats, sub_var=[7] * len(fs))
    for t in T["syrk"]:
        pa.syrk_units(T, t, layout["yd_plane"])


@pytest.mark.parametrize("name", NAMES)
def test_runs_visit_every_tile_once(name):
    fs = _factors(name)
    plan = _plan(fs)
    T = pe.export_plan(plan)
    n = int(plan.sizes.F_doubles) // 1024
    want = [(i, I, J) for i, sd in enumerate(T["subs"]) for I in range(sd["nt"]) for J in range(I + 1)]
    assert len(want) == n
    for warps in {1, 3, 4, n - 1, n, n + 5, 1824} - {0}:
        assert pa.walk_runs(T, n, warps) == want
