"""GPU tests of what a stored tuning does to calls that it was not made for: small
batches keep their teams, and turns are taken only by more pairs of about one length
than there are lanes. Which way a call went shows in the launches and in the queue's
counters at the start of the workspace."""
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


@pytest.mark.parametrize("n,lengths", [(1, [900]), (100, [300]), (20 * SMS, [100, 900]),
                                       (128 * SMS + 500, [100, 200, 900]), (128 * SMS + 500, [300])])
def test_autotuning_one_batch_leaves_others_as_they_are(n, lengths):
    few = prepared(100, [300])
    mixed = prepared(128 * SMS + 500, [100, 200, 900])
    db, want = prepared(n, lengths)
    best, ms = db.autotune()
    np.testing.assert_array_equal(db.results().dist, want[np.arange(n) % 60])
    stored = ga.ga_tuning_get(W, O, K)
    assert ms > 0 and stored.slice_windows == best.slice_windows and stored.lpt == best.lpt == 1
    if n <= 128 * SMS or len(lengths) > 1:  # no turns to choose
        assert best.slice_windows == 0
    assert best.slice_windows >= 0
    assert align(*few) == (1, False)
    assert align(*mixed) == (5, False)
    assert align(*prepared(128 * SMS + 500, [300])) == (5, True)
