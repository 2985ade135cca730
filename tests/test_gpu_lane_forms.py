"""GPU parity of the launch forms of the batched kernel and of its input and
output stages, at the sizes where they change: widths of a vector word, four
lanes per pair and one, teams, one warp per scheduler and two, the ordering in one
launch and in three, turns of the sliced queue chosen on the device, and the
packer's and the compaction's loops. Outputs are whole numbers and have to be
equal."""
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


def pairs(seed, n, lo, hi):
    rnd = random.Random(seed)
    rs = lambda L: "".join(rnd.choices("ACGT", k=L))  # noqa: E731
    out = []
    for _ in range(n):
        read = rs(rnd.randint(lo, hi))
        ref = list(read)
        for _ in range(len(read) // 12):
            x = rnd.randrange(len(ref) + 1)
            if rnd.random() < 0.4:
                ref[x:x + 1] = rnd.choice("ACGT")
            elif rnd.random() < 0.5:
                ref[x:x] = rs(rnd.choice([1, 1, 2, 12]))
            else:
                del ref[x:x + rnd.choice([1, 1, 2, 12])]
        out.append((read, "".join(ref) + rs(rnd.choice([0, 3, 40]))))
    return out


def check(batch, W, O, k, order="MSID", tuning=None, spans=None):
    db = DeviceBatch(batch, W=W, O=O, k=k)
    ref = oracle.align(batch, W=W, O=O, k=k, tb_order=order, start_span=spans)
    db.pack()
    if spans is not None:
        db.align_locate(spans)
    elif order != "MSID":
        db.align_order(order)
    else:
        db.align("batched", tuning=tuning)
    got = db.results()
    for name in ("status", "dist", "ref_consumed", "n_runs"):
        np.testing.assert_array_equal(np.asarray(getattr(got, name)).astype(np.int64),
                                      np.asarray(getattr(ref, name)).astype(np.int64), err_msg=name)
    ok = np.asarray(ref.status) == 0
    for name in ("n_windows", "cells"):
        np.testing.assert_array_equal(np.asarray(getattr(got, name))[ok], np.asarray(getattr(ref, name))[ok])
    for p in range(batch.n_pairs):
        assert np.array_equal(got.runs(p), ref.runs(p)), f"pair {p}: {got.cigar_str(p)[:120]}"


WIDTHS = [1, 2, 15, 16, 17, 31, 32, 33, 48, 63, 64, 65, 95, 96, 97, 112, 127, 128]


@pytest.mark.parametrize("W", WIDTHS)
def test_widths(W):
    # Every remainder of a vector word, no overlap and the largest; the last pairs
    # end inside a window, at its edge and one base after it.
    for O in sorted({0, 3 * W // 8, W - 1}):
        b = datagen.from_pairs(pairs(W + O, 40, 1, 3 * W + 8 if W - O > 4 else 2 * W + 2))
        check(b, W, O, W)
        check(b, W, O, max(1, W // 4))
        check(b, W, O, W, order="DIMS")
        check(b, W, O, W, spans=np.arange(b.n_pairs, dtype=np.uint32) * 3 % 90)


@pytest.mark.parametrize("W,O,n", [(64, 24, 700), (64, 24, 20_000), (64, 0, 20_000), (64, 24, 40_000),
                                   (32, 12, 40_000), (96, 36, 4_800), (96, 36, 5_000), (128, 48, 5_000),
                                   (128, 0, 10_000), (96, 0, 10_000)])
def test_pairs_per_launch(W, O, n):
    # Reads of one to three windows: one pair per warp and more, one warp per
    # scheduler and two, four lanes per pair (wide windows, up to 4,864 pairs on
    # 152 multiprocessors) and one, warps of 32 pairs and of 16.
    base = pairs(n + W, 500, W // 2, 3 * W)
    check(datagen.from_pairs([base[q % 500] for q in range(n)]), W, O, W)


@pytest.mark.parametrize("W,O", [(64, 24), (32, 12), (40, 3), (64, 63)])
@pytest.mark.parametrize("n", [1, 152, 153, 608, 609, 1216, 1217, 2432, 2433])
def test_teams(W, O, n):
    # A pair by a team of 128, 32, 16 and 8 lanes (on 152 multiprocessors up to
    # 152, 608, 1,216 and 2,432 pairs): reads of few and of many errors, against
    # sequence of their own and of somebody else's, of all lengths at once so that
    # the teams of a warp come to the same places at different times.
    base = pairs(n + W, 60, 1, 400) if W - O > 4 else pairs(n, 30, 1, 100)
    rnd = random.Random(n)
    for read, ref in base[:20]:
        x = rnd.randrange(len(read) + 1)
        base.append((read, read[:x] + rnd.choice("ACGT") + read[x:]))
        base.append((read, base[rnd.randrange(20)][1]))
    b = datagen.from_pairs([base[(q * 7 + q // 100) % len(base)] for q in range(n)])
    check(b, W, O, W)
    check(b, W, O, max(1, W // 5), spans=np.arange(n, dtype=np.uint32) * 3 % 90)


@pytest.mark.parametrize("n", [63, 64, 1024, 1025, 16_384, 16_385, 30_000])
def test_ordering_sizes(n):
    base = pairs(n, 300, 20, 700)
    check(datagen.from_pairs([base[q % 300] for q in range(n)]), 64, 24, 64)


@pytest.mark.parametrize("n,long", [(2_500, 8), (5_000, 700), (20_000, 90)])
def test_few_long_pairs_among_many(n, long):
    # Long pairs that decide how long the batch takes: a few lanes of some warps.
    some = pairs(n, 24, 5_000, 9_000) + pairs(n + 1, 24, 1_500, 5_000)
    rest = pairs(n + 2, 200, 30, 600)
    b = datagen.from_pairs([some[q % 48] if q < long else rest[q % 200] for q in range(n)])
    check(b, 64, 24, 64)
    check(b, 32, 12, 32, spans=np.arange(n, dtype=np.uint32) % 90)


def test_turns_chosen_for_pairs_of_one_length():
    # More pairs than one warp per scheduler holds, all of one length: the sliced
    # queue takes turns of 64 windows (reads of 70 windows have two).
    base = datagen.from_pairs(pairs(5, 40, 2790, 2800))
    n = 20_500
    rl = base.read_len.astype(np.int64)
    order = np.argsort(-rl, kind="stable")
    b = datagen.from_pairs([(base.read(int(order[q % 40])), base.ref(int(order[q % 40]))) for q in range(n)])
    ref = oracle.align(base)
    db = DeviceBatch(b)
    db.run("batched")
    got = db.results()
    want = np.asarray(ref.dist)[order][np.arange(n) % 40]
    np.testing.assert_array_equal(got.dist, want)
    np.testing.assert_array_equal(got.status, 0)
    for p in range(0, n, 17):
        assert np.array_equal(got.runs(p), ref.runs(int(order[p % 40])))


@pytest.mark.parametrize("n", [16 * 64 - 5, 1_000_003, 62_300_000 + 13, 320_000_001])
def test_pack_long_inputs(n):
    # Past the sizes at which a thread packs four chunks at a time, and at which the
    # input counts as far larger than L2, with all byte
    # values among the letters (one in a hundred).
    g = torch.Generator(device="cuda").manual_seed(n)
    letters = torch.tensor(list(b"ACGTacgt"), dtype=torch.uint8, device="cuda")
    a = letters[torch.randint(0, 8, (n,), generator=g, device="cuda")]
    odd = torch.rand(n, generator=g, device="cuda") < 0.01
    a = torch.where(odd, torch.randint(0, 256, (n,), generator=g, device="cuda").to(torch.uint8), a)
    code = torch.zeros(256, dtype=torch.uint8, device="cuda")
    known = torch.zeros(256, dtype=torch.bool, device="cuda")
    for c, v in zip(b"ACGTacgt", (0, 1, 2, 3, 0, 1, 2, 3)):
        code[c], known[c] = v, True
    c = torch.zeros((n + 3) // 4 * 4, dtype=torch.uint8, device="cuda")
    c[:n] = code[a.long()]
    c = c.view(-1, 4)
    want = c[:, 0] | c[:, 1] << 2 | c[:, 2] << 4 | c[:, 3] << 6
    out = torch.full(((n + 3) // 4,), 0xEE, dtype=torch.uint8, device="cuda")
    bad = torch.zeros(1, dtype=torch.int32, device="cuda")
    ga.ga_pack_2bit(a, n, out, bad)
    assert torch.equal(out, want)
    assert int(bad.item()) == int((~known[a.long()]).sum())


@pytest.mark.parametrize("shift", range(1, 16))
def test_pack_at_any_address(shift):
    # Every distance from a 16-byte address, with no, one and many whole blocks and
    # other letters at both ends, against a copy at an aligned address.
    for n in [*range(1, 70), 5 * 4096 + 7, 3_000_017]:
        g = torch.Generator(device="cuda").manual_seed(n + shift)
        a = torch.tensor(list(b"ACGTacgtN"), dtype=torch.uint8, device="cuda")[
            torch.randint(0, 9, (n + shift,), generator=g, device="cuda")][shift:]
        out = [torch.full(((n + 3) // 4 + 4,), 0xEE, dtype=torch.uint8, device="cuda") for _ in range(2)]
        bad = [torch.zeros(1, dtype=torch.int32, device="cuda") for _ in range(2)]
        ga.ga_pack_2bit(a, n, out[0], bad[0])
        ga.ga_pack_2bit(a.clone(), n, out[1], bad[1])
        assert torch.equal(out[0], out[1]) and int(bad[0]) == int(bad[1]), n


@pytest.mark.parametrize("n,most", [(1, 3000), (7, 0), (1023, 20), (1024, 300), (1025, 300), (32_768, 40),
                                    (32_769, 40), (3000, 900), (1_050_000, 3)])
def test_compaction(n, most):
    # One chunk of 1,024 pairs and more, both tile sizes, copies by run and by
    # pair, chunk sums added up and scanned, empty CIGARs, a buffer too small.
    rng = np.random.default_rng(n + most)
    runs = rng.integers(0, most + 1, n).astype(np.int64)
    cap = runs + rng.integers(0, 4, n)
    off = np.concatenate([[0], np.cumsum(cap)]).astype(np.int64)
    src = torch.arange(int(off[-1]) + 1, dtype=torch.int32, device="cuda") * 7 + 3
    d_off = torch.from_numpy(off).cuda()
    d_runs = torch.from_numpy(runs.astype(np.int32)).cuda()
    total = int(runs.sum())
    start = np.concatenate([[0], np.cumsum(runs)])
    pos = np.repeat(off[:-1] - start[:-1], runs) + np.arange(total)
    want = src.cpu().numpy()[pos]
    ws_bytes = ga.ga_cigar_compact_workspace_size(n)
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device="cuda")
    for room in (total + 5, total, max(total - 1, 0)):
        out = torch.full((max(room, 1) + 1,), -9, dtype=torch.int32, device="cuda")
        out_off = torch.full((n + 1,), -9, dtype=torch.int64, device="cuda")
        ga.ga_cigar_compact(src, d_off, d_runs, n, out, room, out_off, ws, ws_bytes)
        np.testing.assert_array_equal(out_off.cpu().numpy(), start)
        got = out.cpu().numpy()
        if room >= total:
            np.testing.assert_array_equal(got[:total], want)
            assert (got[total:] == -9).all()
        else:
            assert (got == -9).all()
