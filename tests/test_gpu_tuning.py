"""GPU tests of what a stored tuning does to calls that it was not made for: small
batches keep their teams, and an order and turns are taken only by more pairs than
there are lanes, of the kind of lengths they were chosen for. Which way a call went
shows in the launches, and in the queue's counters and the pairs' order at the start
of the workspace."""
from __future__ import annotations

import random

import numpy as np
import pytest

import oracle
from paper_2203_15561_gb300 import datagen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2203_15561_gb300 as ga  # noqa: E402
from paper_2203_15561_gb300.pipeline import DeviceBatch  # noqa: E402

SMS = torch.cuda.get_device_properties(0).multi_processor_count
W, O, K = 64, 24, 64


@pytest.fixture(autouse=True)
def no_stored_tuning():
    yield
    ga.ga_tuning_set(W, O, K, None)


def batch(n, lengths, seed=1):
    rnd = random.Random(seed)
    base = []
    for q in range(60):
        read = "".join(rnd.choices("ACGT", k=lengths[q % len(lengths)]))
        ref = list(read)
        for _ in range(len(read) // 10):
            x = rnd.randrange(len(ref))
            ref[x:x + 1] = rnd.choice(["", "A", "CG"])
        base.append((read, "".join(ref)))
    return datagen.from_pairs([base[q % 60] for q in range(n)])


def align(db, want, tuning=None):
    """Aligns the batch, checks it and returns (launches, pairs that finished in turns)."""
    db.workspace.zero_()
    before = ga.ga_launch_count()
    db.align("batched", tuning=tuning)
    launches = ga.ga_launch_count() - before
    got = db.results()
    np.testing.assert_array_equal(got.dist, want[np.arange(db.n) % 60])
    counters = db.workspace[:20].cpu().numpy().view(np.uint32)
    # [2] the ring's tail: all pairs at first; [3] pairs not finished.
    return launches, int(counters[2]) - int(counters[3]) >= db.n


def prepared(n, lengths):
    b = batch(n, lengths)
    db = DeviceBatch(b, W=W, O=O, k=K)
    db.pack()
    return db, np.asarray(oracle.align(b.slice(0, min(60, n)), W=W, O=O, k=K).dist)


@pytest.mark.parametrize("slice_windows", [2, 64])
def test_stored_turns_leave_other_batches_as_they_are(slice_windows):
    few = prepared(100, [300])
    fewer_than_lanes = prepared(20 * SMS, [300])
    alike = prepared(128 * SMS + 500, [300])
    mixed = prepared(128 * SMS + 500, [100, 200, 900])
    default = [align(*x) for x in (few, fewer_than_lanes, alike, mixed)]
    # A team launch; order and lanes; three launches of ordering, ring and lanes twice.
    assert default == [(1, False), (2, False), (5, True), (5, False)]
    t = ga.ga_tuning(8, 8, 39, 1, 0, slice_windows)
    ga.ga_tuning_set(W, O, K, t)
    assert [align(*x) for x in (few, fewer_than_lanes, alike, mixed)] == default
    # A call that asks for turns itself gets them.
    asked = [align(*x, tuning=t) for x in (few, fewer_than_lanes, alike, mixed)]
    assert asked == [(3, True), (3, True), (5, True), (5, True)]


def handed_out(db):
    """The order in which the last alignment handed the pairs out: "longest" or "index"."""
    order = db.workspace[4352:4352 + 4 * db.n].cpu().numpy().view(np.uint32)
    if np.array_equal(order, np.arange(db.n)):
        return "index"
    assert np.array_equal(np.sort(order), np.arange(db.n))
    rl = np.asarray(db.batch.read_len).astype(np.int64)[order] >> 6
    assert (np.diff(rl) <= 0).all()
    return "longest"


MANY = 128 * SMS + 500  # more pairs than lanes
# (Reads of about one length, but of two buckets of the ordering: longest first is not
# the order of the indexes.)
ALIKE, MIXED = [250, 300], [100, 200, 900]


@pytest.mark.parametrize("n,lengths", [(1, [900]), (100, [300]), (20 * SMS, [100, 900]), (MANY, MIXED), (MANY, ALIKE),
                                       (MANY, [2800]), (MANY, [800, 1500, 2800])])
def test_autotuning_one_batch_leaves_others_as_they_are(n, lengths):
    few = prepared(100, ALIKE)
    db, want = prepared(n, lengths)
    best, ms = db.autotune()
    np.testing.assert_array_equal(db.results().dist, want[np.arange(n) % 60])
    stored = ga.ga_tuning_get(W, O, K)
    assert ms > 0 and (stored.slice_windows, stored.lpt) == (best.slice_windows, best.lpt)
    assert align(*few) == (1, False)
    if n < MANY:  # nothing to choose
        assert (best.lpt, best.slice_windows) == (1, 0)
    for lens in (ALIKE, MIXED):
        d, w = prepared(MANY, lens)
        launches, turns = align(d, w)
        if n == MANY and (lens is ALIKE) == (max(lengths) < 2 * min(lengths)):  # made for it
            alike = lens is ALIKE
            assert turns == (best.slice_windows > 0 or (best.slice_windows == 0 and alike))
            assert handed_out(d) == ("index" if best.lpt < 0 else "longest")
        else:  # as without a stored tuning
            assert turns == (lens is ALIKE) and handed_out(d) == "longest"
    # A call's own tuning is not mixed with the stored one.
    assert align(*few, tuning=ga.ga_tuning(0, 0, 0, 0, 0, 2)) == (3, True) and handed_out(few[0]) == "longest"
