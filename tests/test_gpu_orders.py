"""GPU parity of the traceback's priority orders over the batched kernel's forms: all
24 orders (M first or behind insertions and deletions), reads of no, few and many
errors so that runs of matches are longer and shorter than the walk looks ahead,
repeats that let insertions and deletions compete with matches, every width of a
vector, and batches whose tables hold fewer columns than a window walks."""
from __future__ import annotations

import itertools
import random

import numpy as np
import pytest

import oracle
from paper_2203_15561_gb300 import datagen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2203_15561_gb300.pipeline import DeviceBatch  # noqa: E402

ORDERS = ["".join(o) for o in itertools.permutations("MSID")]


def pairs(seed, n, lo, hi):
    rnd = random.Random(seed)
    rs = lambda L: "".join(rnd.choices("ACGT", k=L))  # noqa: E731
    out = []
    for q in range(n):
        read = rs(rnd.randint(lo, hi))
        if q % 4 == 1:  # repeats of one to three bases
            read = "".join(rnd.choice(["A", "AC", "GGT"]) * rnd.randint(1, 9) for _ in range(len(read) // 8 + 1))
        ref = list(read)
        for _ in range([0, len(read) // 15, 1, len(read) // 60][q % 4]):
            x = rnd.randrange(len(ref) + 1)
            ref[x:x + 1] = rnd.choice(["", rnd.choice("ACGT"), rs(2), rs(9)])
        out.append((read, "".join(ref) + rs(rnd.choice([0, 3, 40]))))
    return out


def check(base, n, W, O, k, order):
    m = len(base)
    ref = oracle.align(datagen.from_pairs(base), W=W, O=O, k=k, tb_order=order)
    db = DeviceBatch(datagen.from_pairs([base[q % m] for q in range(n)]), W=W, O=O, k=k)
    db.pack()
    db.align_order(order)
    got = db.results()
    which = np.arange(n) % m
    for name in ("status", "dist", "ref_consumed", "n_runs"):
        np.testing.assert_array_equal(np.asarray(getattr(got, name)).astype(np.int64),
                                      np.asarray(getattr(ref, name)).astype(np.int64)[which], err_msg=name)
    ok = np.asarray(ref.status)[which] == 0
    for name in ("n_windows", "cells"):
        np.testing.assert_array_equal(np.asarray(getattr(got, name))[ok], np.asarray(getattr(ref, name))[which][ok])
    for p in [*range(min(n, m)), *range(m, n, 97)]:
        assert np.array_equal(got.runs(p), ref.runs(p % m)), f"pair {p}: {got.cigar_str(p)[:120]}"


@pytest.mark.parametrize("order", ORDERS)
def test_orders(order):
    for W, O in [(64, 24), (32, 12), (33, 0), (7, 3), (64, 63), (96, 36), (128, 48)]:
        base = pairs(ORDERS.index(order), 60, 1, 4 * W if W - O > 4 else W + 9)
        check(base, len(base), W, O, W, order)
        check(base, len(base), W, O, max(1, W // 5), order)


@pytest.mark.parametrize("order", ["DIMS", "IMSD", "SDMI", "MDIS"])
@pytest.mark.parametrize("W,O,n", [(64, 24, 20_000), (64, 24, 40_000), (64, 0, 40_000), (32, 12, 40_000),
                                   (32, 0, 40_000), (96, 36, 5_000), (96, 0, 10_000), (128, 48, 5_000),
                                   (128, 0, 10_000)])
def test_orders_of_large_batches(W, O, n, order):
    check(pairs(W + O, 120, W // 2, 3 * W), n, W, O, W, order)
