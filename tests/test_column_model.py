"""A CPU model of the batched kernels' window: edit-distance columns in
difference form instead of GenASM's error rows, against the CPU oracle.

Row d of GenASM's table says where D(i, j) <= d, with D(i, j) the fewest edits
that align the pattern suffix of j + 1 bases with a prefix of the text from
column i (text end free). The model keeps D's vertical and horizontal
differences, one bit vector each per column (Myers 1999, Hyyro 2003), and
walks the traceback on three facts about an active cell with D(i, j) = d:
M is possible iff the bases match, S iff D(i+1, j-1) = d - 1 (diagonal
difference 1), I iff the vertical and D iff the horizontal difference is +1.
Every walk stays on such exact cells, so the edges are those that the rows
d and d - 1 show. Lengths, geometries and priority orders are the kernels' own
range; outputs must be the oracle's, element by element.
"""
from __future__ import annotations

import random

import numpy as np
import pytest

import oracle
from paper_2203_15561_gb300 import datagen

M, S, I, D = 0, 1, 2, 3
OPS = {M: 7, S: 8, I: 1, D: 2}


def columns(P, T):
    """Per text column i: (D0, VP, HP); and d_min = D(0, wp - 1)."""
    wp, wt = len(P), len(T)
    full = (1 << wp) - 1
    eq = {c: sum(1 << j for j in range(wp) if P[wp - 1 - j] == c) for c in set(P) | set(T)}
    vp, vn, out = full, 0, [None] * wt
    for i in range(wt - 1, -1, -1):
        e = eq[T[i]]
        d0 = ((((e & vp) + vp) ^ vp) | e | vn) & full
        hp = (vn | ~(d0 | vp)) & full
        hn = vp & d0
        hps, hns = (hp << 1) & full, (hn << 1) & full
        vp, vn = (hns | ~(d0 | hps)) & full, hps & d0
        out[i] = (d0, vp, hp)
    return out, bin(vp).count("1") - bin(vn).count("1")


def locate(P, T, S, k):
    """(leftmost start with the fewest edits among 0..min(S, L), its edits), or None."""
    wp, L = len(P), len(T)
    best = None
    if S >= L and wp <= k:
        best = (wp, L)
    cols = [None] * L
    full = (1 << wp) - 1
    eq = {c: sum(1 << j for j in range(wp) if P[wp - 1 - j] == c) for c in set(P) | set(T)}
    vp, vn, score, top = full, 0, wp, 1 << (wp - 1)
    for i in range(L - 1, -1, -1):
        e = eq[T[i]]
        d0 = ((((e & vp) + vp) ^ vp) | e | vn) & full
        hp = (vn | ~(d0 | vp)) & full
        hn = vp & d0
        score += bool(hp & top) - bool(hn & top)
        hps, hns = (hp << 1) & full, (hn << 1) & full
        vp, vn = (hns | ~(d0 | hps)) & full, hps & d0
        if i <= S and score <= k and (best is None or score <= best[0]):
            best = (score, i)
    return best


def align(read, ref, W, O, k, order=(M, S, I, D), span=0):
    """(status, dist, ref_start, ref_end, runs, windows, cells)."""
    pp = pt = dist = windows = cells = 0
    start, runs = 0, []
    k = min(k, W)

    def put(op, n):
        if n and runs and runs[-1][0] == op:
            runs[-1][1] += n
        elif n:
            runs.append([op, n])

    if span and read:
        L = min(len(ref), span + W)
        found = locate(read[:W], ref[:L], min(span, L), k)
        if found is None:
            return 1, -1, -1, -1, [], 0, 0
        start = pt = found[1]
        cells = L * (found[0] + 1)
    while pp < len(read):
        P, T = read[pp:pp + W], ref[pt:pt + W]
        wp, wt = len(P), len(T)
        last = pp + wp == len(read)
        cols, dmin = columns(P, T)
        if dmin > k:
            return 1, -1, -1, -1, [], windows, cells
        cp = ct = edits = 0
        while cp < wp if last else (cp < W - O and ct < W - O):
            j = wp - 1 - cp
            if ct == wt:
                code = I
            else:
                d0, vp, hp = cols[ct]
                can = {M: P[cp] == T[ct], S: not d0 >> j & 1, I: vp >> j & 1, D: hp >> j & 1}
                code = next(c for c in order if can[c])
            put(OPS[code], 1)
            edits += code != M
            cp += code != D
            ct += code != I
        if last:
            assert edits == dmin
        dist += edits
        windows += 1
        cells += wt * (dmin + 1)
        pp += cp
        pt += ct
    return 0, dist, start, pt, [n << 4 | op for op, n in runs], windows, cells


def pairs(seed, n, max_len):
    rnd = random.Random(seed)
    rs = lambda L: "".join(rnd.choice("ACGT") for _ in range(L))  # noqa: E731
    out = [("A", ""), ("ACGT", ""), ("A" * 70, "A" * 64), ("ACGT" * 20, "T" * 90), ("A", "A"),
           ("A" * 64, "A" * 200), ("C" * 130, "A" * 130)]
    for _ in range(n):
        read = rs(rnd.randint(1, max_len))
        ref = list(read)
        for _ in range(rnd.randint(0, max(1, len(read) // rnd.choice([3, 8, 20])))):
            x = rnd.randrange(len(ref) + 1)
            u = rnd.random()
            if u < 0.3 and x < len(ref):
                ref[x] = rnd.choice("ACGT")
            elif u < 0.65:
                ref[x:x] = rs(rnd.choice([1, 1, 2, 9, 25]))
            else:
                del ref[x:x + rnd.choice([1, 1, 2, 9, 25])]
        ref = rs(rnd.choice([0, 0, 5, 60])) + "".join(ref) + rs(rnd.choice([0, 20]))
        out.append((read, ref if rnd.random() < 0.85 else rs(rnd.randint(0, max_len))))
    return out


def check(ps, W, O, k, order="MSID", spans=None):
    b = datagen.from_pairs(ps)
    ref = oracle.align(b, W=W, O=O, k=k, tb_order=order, start_span=spans)
    for p, (r, f) in enumerate(ps):
        got = align(r, f, W, O, k, ["MSID".index(c) for c in order],
                    0 if spans is None else int(spans[p]))
        want = (ref.status[p], ref.dist[p], ref.ref_start[p] if spans is not None else got[2],
                ref.ref_consumed[p], [int(x) for x in ref.runs(p)])
        assert got[:4] == tuple(int(x) for x in want[:4]), (p, r, f)
        assert got[4] == want[4], (p, r, f)
        if got[0] == 0:
            assert got[5:] == (int(ref.n_windows[p]), int(ref.cells[p])), (p, r, f)


@pytest.mark.parametrize("W,O,k", [(64, 24, 64), (64, 24, 12), (64, 0, 64), (64, 63, 64), (33, 12, 33),
                                   (32, 12, 32), (17, 5, 9), (1, 0, 1), (2, 1, 2), (65, 24, 65),
                                   (96, 36, 96), (97, 10, 97), (128, 48, 128), (128, 127, 40)])
def test_columns_match_oracle(W, O, k):
    check(pairs(W * 131 + O, 60, 400 if W - O > 8 else 140), W, O, k)


@pytest.mark.parametrize("order", ["MISD", "MDSI", "DIMS", "SDIM", "IDSM", "DSIM"])
def test_columns_orders_match_oracle(order):
    for W, O in ((64, 24), (31, 7), (100, 30)):
        check(pairs(sum(map(ord, order)) + W, 40, 300), W, O, W, order)


@pytest.mark.parametrize("W,O,k", [(64, 24, 64), (64, 16, 10), (32, 8, 32), (128, 48, 128), (70, 0, 70)])
def test_columns_free_start_matches_oracle(W, O, k):
    ps = pairs(W + 7 * O, 60, 300)
    rnd = np.random.default_rng(W)
    spans = np.array([int(rnd.choice([0, 1, 60, 200, 10_000])) for _ in ps], dtype=np.uint32)
    check(ps, W, O, k, spans=spans)
