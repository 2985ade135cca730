"""GPU tests of the server's step in its forms: teams of lanes while few pairs are
active, a lane per pair with more than 16 per multiprocessor, vectors of one word
and of two, pairs that change from one form to the other with their saved window
state, and servers of several widths at once. Results have to be the oracle's."""
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

from paper_2203_15561_gb300.serving import Server  # noqa: E402

# More active pairs than teams are made for.
MANY = 16 * torch.cuda.get_device_properties(0).multi_processor_count + 100


def pairs(seed, n, lo, hi):
    rnd = random.Random(seed)
    rs = lambda L: "".join(rnd.choices("ACGT", k=L))  # noqa: E731
    out = []
    for _ in range(n):
        read = rs(rnd.randint(lo, hi))
        ref = list(read)
        for _ in range(len(read) // 12):
            x = rnd.randrange(len(ref))
            ref[x:x + 1] = rnd.choice(["", rnd.choice("ACGT"), rs(2)])
        out.append((read, "".join(ref) + rs(rnd.choice([0, 3, 40])) if rnd.random() < 0.9 else rs(len(read))))
    return out


def many(seed, n, lo, hi):
    base = pairs(seed, 200, lo, hi)
    return datagen.from_pairs([base[q % 200] for q in range(n)])


def check(batch, got, W, O, k):
    ref = oracle.align(batch, W=W, O=O, k=k)
    for name in ("status", "dist", "ref_consumed"):
        np.testing.assert_array_equal(getattr(got, name), getattr(ref, name), err_msg=name)
    for p in range(batch.n_pairs):
        assert np.array_equal(got.runs(p), ref.runs(p)), f"pair {p}"


def finish(server, want, active, limit=20_000):
    got = {}
    for _ in range(limit):
        active.append(server.step())
        for r in server.poll():
            got[r.tag] = r
        if len(got) == want:
            return got
    raise AssertionError(f"{len(got)} of {want} requests")


@pytest.mark.parametrize("W,O", [(32, 12), (17, 4), (33, 9), (48, 18), (64, 24)])
@pytest.mark.parametrize("cap", [False, True])
def test_pairs_change_between_teams_and_lanes(W, O, cap):
    k = W // 4 if cap else W
    server = Server(2 << 30, W=W, O=O, k=k, step_windows=3)
    batches = {0: datagen.from_pairs(pairs(W, 40, 30 * (W - O), 60 * (W - O)))}
    server.submit(batches[0], tag=0)
    active, got = [], {}
    for tag in (1, 2):
        for _ in range(3):  # the long ones by teams
            active.append(server.step())
        batches[tag] = many(W + tag, MANY, 1, 6 * (W - O))  # and with many short ones by lanes
        server.submit(batches[tag], tag=tag)
        for _ in range(2):
            active.append(server.step())
        got.update({r.tag: r for r in server.poll()})
    got.update(finish(server, len(batches) - len(got), active))
    server.close()
    form = [a > MANY - 100 for a in active]
    changes = sum(x != y for x, y in zip(form, form[1:]))
    assert any(form) and changes >= 2, active  # (lanes at least once, and back)
    for tag, b in batches.items():
        check(b, got[tag], W, O, k)


def test_servers_of_several_widths_at_once():
    widths = [(64, 24), (40, 15), (32, 12), (20, 6)]
    servers = [Server(1 << 30, W=W, O=O, k=W, step_windows=2) for W, O in widths]
    batches = [many(W, MANY, 1, 4 * (W - O)) for W, O in widths]
    for s, b in zip(servers, batches):
        s.submit(b, tag=0)
    got = {}
    for _ in range(1000):
        for q, s in enumerate(servers):
            s.step()
            for r in s.poll():
                got[q] = r
        if len(got) == len(servers):
            break
    for q, (W, O) in enumerate(widths):
        check(batches[q], got[q], W, O, W)
        servers[q].close()
