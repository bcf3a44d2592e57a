"""CPU replay of how the assembly and product kernels share a plan's work out, beside tests/plan_emulator.py's tasks:
the seeds of every sorted column, the FP64 TRSM's parts of 1 .. 16 columns, both
SYRKs' rows numbered through across supernodes and their 8x8 pieces, and the products' runs of tiles.  Index
arithmetic as in csrc/sc_trsm.cuh, sc_kernels.cu, sc_split.cu, sc_tiles.cuh and sc_apply_fixed.cu, values in FP64."""
import numpy as np

import plan_emulator as pe

SYRK_BATCH = 64          # kSyrkBatch


def seed_table(plan, T) -> np.ndarray:
    """The section behind the numbered ones: the first seed of every sorted column of the batch, and the end."""
    blob = np.zeros(plan.sizes.plan_bytes, np.uint8)
    plan.lib.sc_export_plan(plan.h, blob.ctypes.data, blob.size)
    off, nb = blob[pe.HEADER.itemsize:pe.HEADER.itemsize + 16].view("<u8")
    assert off % 256 == 0 and off + nb <= blob.size
    last = max(int(a) + int(b) for a, b in zip(T["header"]["sec_off"], T["header"]["sec_bytes"]))
    assert off >= last
    return blob[int(off):int(off + nb)].view("<i4")


def part_columns(t, width):
    """The columns of each part of a TRSM task (kChunk / width parts; the last ones may have none)."""
    c_end = int(t["c_lo"] + t["w"])
    for part in range(32 // width):
        lo = int(t["c_lo"]) + part * width
        yield lo, min(lo + width, c_end)


def tri_at(row, p):
    return p * 31 - p * (p - 1) // 2 + row - p - 1


def trsm_part(T, seeds, t, c_lo, c_hi, Lv, invd, Y, flat):
    """One part by one warp.  flat: the update's (row, column) pairs numbered row by row over all lanes, else
    32 / wk whole rows at a time."""
    sns = T["sns"]
    lst = T["trsm_list"][t["list_off"]:t["list_off"] + t["list_len"]]
    hit = [s for s in (sns[si] for si in lst) if max(s["jlo"], c_lo) < min(s["jhi"], c_hi)]
    for s in hit:
        a, b, ws = max(int(s["jlo"]), c_lo), min(int(s["jhi"]), c_hi), int(s["jhi"] - s["jlo"])
        for r in range(s["ns"]):
            o = int(s["y_off"]) + r * ws - int(s["jlo"])
            Y[o + a:o + b] = 0.0
    col0 = int(T["subs"][t["sub"]]["col_off"])
    for e in T["seeds"][seeds[col0 + c_lo]:seeds[col0 + c_hi]]:
        Y[e["y_off"]] = e["value"]
    for s in hit:
        a, b, ws = max(int(s["jlo"]), c_lo), min(int(s["jhi"]), c_hi), int(s["jhi"] - s["jlo"])
        ns, nr = int(s["ns"]), int(s["ns"] + s["rs"])
        colsh = a - int(s["jlo"])
        rm = T["rmap"][s["rmap_off"]:s["rmap_off"] + s["rs"]]
        row = lambda p: (int(s["y_off"]) + p * ws if p < ns else int(rm[p - ns])) + colsh
        lc = int(T["lcp"][s["lcp_off"]])                    # panel row t of column kb at lc + t
        for kb in range(0, ns, 32):
            kw, below = min(32, ns - kb), kb + min(32, ns - kb)
            wk = min(b, int(T["cuts"][s["cut_off"] + kb // 32])) - a
            if wk > 0:
                # the block's triangle, column by column, as it is staged
                tri = np.full(496, np.nan)
                o = lc + kb
                for p in range(kw):
                    for r in range(p + 1, kw):
                        assert o + r == T["lcp"][s["lcp_off"] + kb + p] + r - p
                        tri[tri_at(r, p)] = Lv[o + r]
                    o += nr - (kb + p) - 1
                X = np.stack([Y[row(kb + q):row(kb + q) + wk] for q in range(kw)])
                for p in range(kw):
                    X[p] *= invd[s["lcp_off"] + kb + p]
                    for r in range(p + 1, kw):
                        X[r] -= tri[tri_at(r, p)] * X[p]
                for q in range(kw):
                    Y[row(kb + q):row(kb + q) + wk] = X[q]
                # offsets of a row below from column to column
                step = np.concatenate([[0], np.cumsum([nr - (kb + q) - 1 for q in range(kw - 1)])]).astype(np.int64)
                assert np.array_equal(lc + step + (nr - 1), T["lcp"][s["lcp_off"] + kb + np.arange(kw)] + nr - 1 - kb -
                                      np.arange(kw))
                done = np.zeros((nr - below, wk), int)
                dp = 32 // wk
                for lane in range(32):
                    p, cl, dc = below + lane // wk, lane % wk, 32 - dp * wk
                    if not flat and lane >= dp * wk:
                        p = nr
                    while p < nr:
                        done[p - below, cl] += 1
                        Y[row(p) + cl] -= Lv[lc + step + p] @ X[:, cl]
                        p += dp
                        if flat:
                            cl += dc
                            if cl >= wk:
                                cl, p = cl - wk, p + 1
                assert np.all(done == 1)
            lc += 32 * (nr - kb) - 16 * 33


def syrk_rows(T, t, unit):
    """The live rows of a SYRK task in batches of 64 listed supernodes: per batch (row or unit start of every
    supernode, its first 32-row block); unit = 1 (FP64 rows) or 8 (digit rows)."""
    lst = T["syrk_list"][t["list_off"]:t["list_off"] + t["list_len"]]
    j1 = int(t["q1"]) * 32
    for l0 in range(0, len(lst), SYRK_BATCH):
        start, first = [0], []
        part = [T["sns"][si] for si in lst[l0:l0 + SYRK_BATCH]]
        for s in part:
            nb, b = (int(s["ns"]) + 31) // 32, 0
            while b < nb and T["cuts"][s["cut_off"] + b] <= j1:
                b += 1
            start.append(start[-1] + (max(0, int(s["ns"]) - 32 * b) + unit - 1) // unit)
            first.append(b)
        yield part, np.array(start + [start[-1]] * (SYRK_BATCH + 1 - len(start))), first


def find(start, g):
    """The last supernode that starts at or before row g, as the kernels search for it."""
    e, h = 0, SYRK_BATCH // 2
    while h >= 1:
        if start[e + h] <= g:
            e += h
        h //= 2
    return e


def syrk_pieces(diag, ctas):
    """(row piece, column piece) lists of every warp of a task's CTAs; a row piece is 8 rows, a column piece
    8 columns (4 with eight CTAs)."""
    if ctas == 1:
        code = [0x073, 0x1fb, 0x062, 0x05a]
        return [[((code[w] >> 4 * i) & 3, (code[w] >> (4 * i + 2)) & 3) for i in range(3 if w < 2 else 2)] if diag else
                [(2 * (w >> 1) + (i >> 1), 2 * (w & 1) + (i & 1)) for i in range(4)] for w in range(4)]
    cols = 4 if ctas == 4 else 8
    out = []
    for u in range(4 * ctas):
        if not diag:
            out.append([(u // cols, u % cols)])
            continue
        r = 0
        while r < 4 and u >= (r + 1) * (r + 2) // 2 * (cols // 4):
            r += 1
        out.append([(r, u - r * (r + 1) // 2 * (cols // 4))] if r < 4 else [])
    return out


def syrk_task(T, t, Y, ctas):
    """The 32x32 block of one FP64 task: every piece over the numbered rows that are live on it."""
    diag = t["q1"] == t["q2"]
    j1, j2 = int(t["q1"]) * 32, int(t["q2"]) * 32
    acc, owner = np.zeros((32, 32)), np.zeros((32, 32), int)
    cw = 8 if ctas <= 4 else 4
    for pieces in syrk_pieces(diag, ctas):
        for rb, cb in pieces:
            owner[8 * rb:8 * rb + 8, cw * cb:cw * cb + cw] += 1
    low = np.tril(np.ones((32, 32), bool)) if diag else np.ones((32, 32), bool)
    assert owner.max() == 1 and np.all(owner[low] == 1)
    for part, start, first in syrk_rows(T, t, 1):
        for g in range(start[-1]):
            e = find(start, g)
            s, r = part[e], g - int(start[e])
            ws = int(s["jhi"] - s["jlo"])
            off = int(s["y_off"]) + (32 * first[e] + r) * ws - int(s["jlo"])
            hi, lo = min(int(s["jhi"]), int(T["cuts"][s["cut_off"] + first[e] + r // 32])), int(s["jlo"])
            a1, b1, a2, b2 = max(lo - j1, 0), min(hi - j1, 32), max(lo - j2, 0), min(hi - j2, 32)
            A, B = np.zeros(32), np.zeros(32)
            A[a1:b1], B[a2:b2] = Y[off + j1 + a1:off + j1 + b1], Y[off + j2 + a2:off + j2 + b2]
            assert not np.isnan(A).any() and not np.isnan(B).any()
            for pieces in syrk_pieces(diag, ctas):
                for rb, cb in pieces:
                    r0, c0 = 8 * rb, cw * cb
                    if a1 < r0 + 8 and b1 > r0 and a2 < c0 + cw and b2 > c0:
                        acc[r0:r0 + 8, c0:c0 + cw] += np.outer(A[r0:r0 + 8], B[c0:c0 + cw])
    return np.where(low, acc, 0.0)


def syrk_units(T, t, yd_plane):
    """The split SYRK's 16-byte copies: every live row of every listed supernode in exactly one unit of 8, inside the
    supernode's digit block."""
    seen = set()
    for part, start, first in syrk_rows(T, t, 8):
        for u in range(start[-1]):
            e = find(start, u)
            s, npad = part[e], (int(part[e]["ns"]) + 31) // 32 * 32
            k = 32 * first[e] + 8 * (u - int(start[e]))
            assert k < int(s["ns"]) <= npad and k + 8 <= npad
            for q in (int(t["q1"]), int(t["q2"])):
                for j in range(max(32 * q, int(s["jlo"])), min(32 * q + 32, int(s["jhi"]))):
                    o = int(s["yd_off"]) - int(s["jlo"]) * npad + 32 * first[e] + 8 * (u - int(start[e])) + j * npad
                    assert o % 8 == 0 and o == int(s["yd_off"]) + (j - int(s["jlo"])) * npad + k
                    assert 0 <= o and o + 8 <= yd_plane
            seen.update((int(s["yd_off"]), k + i) for i in range(8) if k + i < s["ns"])
    lst = T["syrk_list"][t["list_off"]:t["list_off"] + t["list_len"]]
    want = {(int(T["sns"][si]["yd_off"]), k) for si in lst for k in range(T["sns"][si]["ns"])
            if int(t["q1"]) * 32 < T["cuts"][T["sns"][si]["cut_off"] + k // 32]}
    assert want <= seen and all(any(x[0] == y[0] and x[1] // 32 == y[1] // 32 for y in want) for x in seen)


def tile_at(T, t0):
    """(task, J) of tile t0 by the warp's 32-way search."""
    tile0 = lambda k: int(T["subs"][T["apply"][k]["sub"]]["F_off"]) // 1024 + int(T["apply"][k]["I"]) * (
        int(T["apply"][k]["I"]) + 1) // 2
    lo, hi = 0, len(T["apply"]) - 1
    while lo < hi:
        step = (hi - lo + 31) // 32
        lo += step * sum(lo + (lane + 1) * step <= hi and tile0(lo + (lane + 1) * step) <= t0 for lane in range(32))
        hi = min(lo + step - 1, hi)
    return lo, t0 - tile0(lo)


def walk_runs(T, n_tiles, warps):
    """(subdomain, I, J) of every tile as the warps' runs visit them, in storage order."""
    out = []
    for w in range(warps):
        t0, t1 = n_tiles * w // warps, n_tiles * (w + 1) // warps
        if t0 >= t1:
            continue
        task, J = tile_at(T, t0)
        for t in range(t0, t1):
            a = T["apply"][task]
            out.append((int(a["sub"]), int(a["I"]), J))
            if t + 1 < t1:
                J += 1
                if J > a["I"]:
                    task, J = task + 1, 0
    return out
