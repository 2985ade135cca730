"""Performance cases of the alignment library: what a read aligner has it do.

Each case is one call (or one burst of calls) that a program makes through the
package's public interface, on sequences already in GPU memory as ASCII, with
the buffers, plan, graph or server that such a program keeps:

  "align"   DeviceBatch: 2-bit packing, then the batched alignment anchored at
            reference base 0 (span false) or with the free-start first window
            over the reference's first 5% (span true), optionally replayed as
            a CUDA graph, with another traceback order, or through the form
            without a workspace; then the CIGARs of all pairs gathered densely
            (ga_cigar_compact), the form in which they leave the GPU;
  "serve"   a Server given a burst of requests on host buffers and stepped
            until every result has been handed out;
  "pack"    ga_pack_2bit alone, as for a reference genome.

Sequences follow the error models of the package's synthetic workloads, drawn
on the GPU: short reads of 1.5-2% substitutions and few indels against a
reference of their own length; long reads of 8-15% errors (substitutions,
deletions and insertions 1:2:3, indel lengths geometric with mean 1.5) against
their true span with a 5% random flank on each side; decoys against unrelated
sequence. All outputs are whole numbers.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2203_15561_gb300 as ga
from paper_2203_15561_gb300 import datagen
from paper_2203_15561_gb300.pipeline import DeviceBatch
from paper_2203_15561_gb300.serving import Server

_ALIGN = {"kind": "align", "W": 64, "O": 24, "k": 64, "span": False, "graph": False, "order": "",
          "noalloc": False, "decoys": 0.0}


def listed():
    return [
        # A mapper verifying one candidate locus of one 10 kb read: the call's latency.
        dict(_ALIGN, name="pair_10kb", n=1, lo=10000, hi=10000, dist="fixed", span=True),
        # A small batch of 100-base reads: launches and latency count.
        dict(_ALIGN, name="short_1k", n=1000, lo=100, hi=100, dist="fixed"),
        # A lane's worth of short and amplicon reads, 100 to 999 bases.
        dict(_ALIGN, name="short_200k", n=200_000, lo=100, hi=999, dist="log"),
        # The benchmark batch: 10,000 reads of 10 kb anchored at reference base 0,
        # replayed from a CUDA graph by a program that reuses its buffers.
        dict(_ALIGN, name="long_10k", n=10_000, lo=10000, hi=10000, dist="fixed", graph=True),
        # The same reads searched for their start in the flank first.
        dict(_ALIGN, name="long_10k_free", n=10_000, lo=10000, hi=10000, dist="fixed", span=True),
        # Chains of a mapper: 2-20 kb reads, a fifth of them against unrelated
        # sequence, with an error cap that turns those away.
        dict(_ALIGN, name="chains_30k", n=30_011, lo=2000, hi=20000, dist="normal", span=True,
             decoys=0.2, k=24),
        # A mixed run, 100 bases to 50 kb: few long reads among many short ones.
        dict(_ALIGN, name="mixed_20k", n=20_000, lo=100, hi=50000, dist="log", span=True),
        # Narrow windows: the quick, less exact setting.
        dict(_ALIGN, name="w32_5k", n=5000, lo=10000, hi=10000, dist="fixed", W=32, O=12, k=32),
        # Windows of 96 and 128 bases: the careful settings.
        dict(_ALIGN, name="w96_4k", n=4000, lo=10000, hi=10000, dist="fixed", W=96, O=36, k=96),
        dict(_ALIGN, name="w128_2k_free", n=2001, lo=10000, hi=10000, dist="fixed", W=128, O=48,
             k=128, span=True),
        # A burst of 16 requests of 1-64 mixed pairs each at an alignment server.
        {"name": "serve_16", "kind": "serve", "requests": 16, "lo": 100, "hi": 50000, "pairs": 64},
        # A gigabase of reference sequence packed to two bits.
        {"name": "pack_1g", "kind": "pack", "n": 1_000_000_007, "offset": 0, "count": True},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    u = rng.random()
    if u < 0.08:
        return {"kind": "pack", "n": _log(rng, 1000, 1_000_000_000), "offset": rng.choice([0, 0, 16, 3]),
                "count": rng.random() < 0.5}
    if u < 0.18:
        return {"kind": "serve", "requests": rng.randint(1, 16), "lo": 100,
                "hi": _log(rng, 1000, 50000), "pairs": rng.randint(1, 64)}
    c = dict(_ALIGN)
    if u < 0.60:
        c["W"] = 64
    elif u < 0.75:
        c["W"] = rng.randint(16, 63)
    else:
        c["W"] = rng.choice([rng.randint(65, 96), rng.randint(97, 128)])
    c["O"] = c["W"] * 3 // 8 if rng.random() < 0.7 else rng.randint(c["W"] // 8, c["W"] * 2 // 3)
    c["k"] = c["W"] if rng.random() < 0.7 else rng.randint(c["W"] // 4, c["W"])
    c["lo"] = _log(rng, 100, 20000)
    c["dist"] = rng.choice(["fixed", "log", "normal"])
    c["hi"] = c["lo"] if c["dist"] == "fixed" else min(50000, c["lo"] * rng.randint(2, 20))
    # At most 40 Mbases of reads (20 in wide windows), at most 100,000 pairs.
    most = (40e6 if c["W"] <= 64 else 20e6) / _mean_len(c)
    c["n"] = _log(rng, 1, max(2, min(100_000, int(most))))
    c["span"] = c["lo"] >= 1000 and rng.random() < 0.6
    c["decoys"] = rng.choice([0.0, 0.0, 0.2])
    v = rng.random()
    if not c["span"]:
        if v < 0.2 and c["W"] <= 64:
            c["graph"] = True
        elif v < 0.4:
            c["order"] = rng.choice(["MISD", "MDSI", "DIMS", "SDIM", "IDSM"])
        elif v < 0.55 and c["W"] <= 64:
            c["noalloc"] = True
    return c


def _mean_len(case):
    lo, hi = case["lo"], case["hi"]
    if hi <= lo:
        return float(lo)
    return (hi - lo) / math.log(hi / lo) if case["dist"] == "log" else (lo + hi) / 2.0


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------


def _lengths(n, lo, hi, dist):
    """Read lengths: the case's own, whatever the seed (a read's real length
    differs from its target by its indels)."""
    rng = np.random.default_rng([n, lo, hi])
    if hi <= lo:
        return np.full(n, lo, dtype=np.int64)
    if dist == "log":
        return np.rint(np.exp(rng.uniform(math.log(lo), math.log(hi), n))).astype(np.int64)
    mid, sd = (lo + hi) / 2.0, (hi - lo) / 12.0
    return np.clip(np.rint(rng.normal(mid, sd, n)), lo, hi).astype(np.int64)


def _starts(lens):
    """4-aligned layout of sequences of these lengths: starts and total characters."""
    pad = (lens + 3) // 4 * 4
    off = torch.zeros(lens.numel() + 1, dtype=torch.int64, device=lens.device)
    torch.cumsum(pad, 0, out=off[1:])
    return off[:-1], int(off[-1])


def _pairs(seed, n, lo, hi, dist, decoys=0.0):
    """n (read, reference) pairs as a host Batch, drawn on the GPU."""
    dev = torch.device("cuda")
    rng = np.random.default_rng([seed, n, lo, hi])
    g = torch.Generator(device=dev)
    g.manual_seed(seed * 1_000_003 + n)
    target = _lengths(n, lo, hi, dist)
    # Reads under 1 kb: short-read model. Longer: 12% errors when all reads are
    # alike, 8-15% by read in a mixed run.
    short = target < 1000
    err = rng.uniform(0.08, 0.15, n) if dist == "log" else np.full(n, 0.12)
    p_sub = np.where(short, 0.015, err / 6)
    r_del = np.where(short, 0.0005, err * 2 / 6 / 1.5)
    r_ins = np.where(short, 0.0005, err * 3 / 6 / 1.5)
    span = np.where(short, target, np.rint(target / (1 - err / 3 + err / 2)).astype(np.int64))
    flank = np.where(short, 0, np.rint(0.05 * span)).astype(np.int64)
    unrelated = rng.random(n) < decoys
    span_d = torch.from_numpy(span).to(dev)
    total = int(span.sum())

    def per_base(values, dtype=torch.float32):
        return torch.repeat_interleave(torch.from_numpy(values).to(dev, dtype), span_d)

    def uniform():
        return torch.rand(total, generator=g, device=dev)

    def codes(m):
        return torch.randint(0, 4, (m,), generator=g, device=dev, dtype=torch.uint8)

    src = codes(total)
    # Deletions: events with geometric lengths (mean 1.5), indels of one base in short reads.
    long_base = per_base(~short, torch.bool)

    def geometric():
        x = 1 + torch.floor(torch.log(uniform().clamp_min(1e-7)) / math.log(1.0 / 3.0)).to(torch.int64)
        return torch.where(long_base, x, torch.ones_like(x))

    at = torch.nonzero(uniform() < per_base(r_del)).squeeze(1)
    gone = torch.zeros(total + 1, dtype=torch.int32, device=dev)
    one = torch.ones_like(at, dtype=torch.int32)
    gone.index_add_(0, at, one)
    gone.index_add_(0, torch.clamp(at + geometric()[at], max=total), -one)
    keep = torch.cumsum(gone[:total], 0) <= 0
    base = torch.where(uniform() < per_base(p_sub), (src + 1 + codes(total) % 3) % 4, src)
    count = torch.where(uniform() < per_base(r_ins), geometric(), 0) + keep
    cum = torch.cumsum(count, 0)
    ends = cum[torch.cumsum(span_d, 0) - 1]
    read_len = torch.diff(ends, prepend=ends.new_zeros(1))
    made = int(ends[-1])
    out = codes(made)  # inserted bases are random
    out[(cum - count)[keep]] = base[keep]
    ascii_of = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device=dev)

    read_off, read_chars = _starts(read_len)
    reads = torch.full((max(read_chars, 4),), ord("A"), dtype=torch.uint8, device=dev)
    shift = torch.repeat_interleave(read_off - (ends - read_len), read_len)
    reads[torch.arange(made, device=dev) + shift] = ascii_of[out.long()]

    flank_d = torch.from_numpy(flank).to(dev)
    ref_len = span_d + 2 * flank_d
    ref_off, ref_chars = _starts(ref_len)
    refs = ascii_of[codes(max(ref_chars, 4)).long()]
    first = torch.cumsum(span_d, 0) - span_d
    shift = torch.repeat_interleave(ref_off + flank_d - first, span_d)
    related = ~per_base(unrelated, torch.bool)
    refs[(torch.arange(total, device=dev) + shift)[related]] = ascii_of[src[related].long()]

    def host(t, dtype=None):
        a = t.cpu().numpy()
        return a if dtype is None else a.astype(dtype)

    return datagen.Batch(host(reads), host(read_off, np.uint64), host(read_len, np.uint32),
                         host(refs), host(ref_off, np.uint64), host(ref_len, np.uint32),
                         np.arange(n, dtype=np.uint64))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "pack":
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        buf = torch.randint(0, 4, (case["n"] + case["offset"],), generator=g, device="cuda",
                            dtype=torch.uint8)
        buf = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device="cuda")[buf.long()] \
            if case["n"] < 50_000_000 else _to_ascii(buf)
        if case["count"]:  # unknown bases, one in a thousand or so
            buf[case["offset"]::997] = ord("N")
        return {"case": case, "ascii": buf, "src": buf[case["offset"]:],
                "packed": torch.zeros((case["n"] + 3) // 4, dtype=torch.uint8, device="cuda"),
                "invalid": torch.zeros(1, dtype=torch.int32, device="cuda")}
    if kind == "serve":
        counts = np.random.default_rng([case["requests"], case["pairs"]]).integers(
            1, case["pairs"] + 1, case["requests"])
        n = int(counts.sum())
        whole = _pairs(seed, n, case["lo"], case["hi"], "log")
        cut = np.concatenate([[0], np.cumsum(counts)])
        # The client's own arrays for the burst's results.
        return {"case": case, "server": Server(1 << 30, step_windows=128),
                "requests": [whole.slice(int(a), int(b)) for a, b in zip(cut[:-1], cut[1:])],
                "cut": cut, "dist": np.zeros(n, np.int32), "status": np.zeros(n, np.int32),
                "ref_consumed": np.zeros(n, np.int32), "n_runs": np.zeros(n, np.int32),
                "runs": np.zeros(_run_room(case, n), np.int32)}
    batch = _pairs(seed, case["n"], case["lo"], case["hi"], case["dist"], case["decoys"])
    db = DeviceBatch(batch, W=case["W"], O=case["O"], k=case["k"])
    st = {"case": case, "db": db}
    if case["span"]:
        db.set_start_span((batch.ref_len.astype(np.int64) + 19) // 20)
    if case["graph"]:
        st["graph"] = db.graph()
    st["cap"] = _run_room(case, db.n)
    st["runs"] = torch.zeros(st["cap"], dtype=torch.int32, device="cuda")
    st["run_off"] = torch.zeros(db.n + 1, dtype=torch.int64, device="cuda")
    st["compact_bytes"] = ga.ga_cigar_compact_workspace_size(db.n)
    st["compact_ws"] = torch.empty(st["compact_bytes"], dtype=torch.uint8, device="cuda")
    return st


def _run_room(case, n):
    """Room for the dense CIGARs: one run per base of the reads' target lengths
    is more than any alignment here makes (indels of mean 1.5, at most 0.7)."""
    return int(_lengths(n, case["lo"], case["hi"], case.get("dist", "log")).sum()) + 16 * n + 1024


def _to_ascii(codes):
    # 0, 1, 2, 3 -> A, C, G, T without an index tensor of eight bytes a base.
    return 65 + 2 * codes + 2 * (codes == 2).to(torch.uint8) + 13 * (codes == 3).to(torch.uint8)


def run(st):
    case = st["case"]
    if case["kind"] == "pack":
        st["invalid"].zero_()
        ga.ga_pack_2bit(st["src"], case["n"], st["packed"], st["invalid"] if case["count"] else None)
        return {"packed": st["packed"], "invalid": st["invalid"]}
    if case["kind"] == "serve":
        server, got = st["server"], {}
        for i, r in enumerate(st["requests"]):
            server.submit(r, tag=i)
        while len(got) < len(st["requests"]):
            server.step()
            for res in server.poll():
                got[res.tag] = res
        at = 0
        for i in range(len(st["requests"])):
            res, a, b = got[i], st["cut"][i], st["cut"][i + 1]
            st["dist"][a:b] = res.dist
            st["status"][a:b] = res.status
            st["ref_consumed"][a:b] = res.ref_consumed
            st["n_runs"][a:b] = np.diff(res.cigar_off)
            st["runs"][at:at + res.cigar.size] = res.cigar.view(np.int32)
            at += res.cigar.size
        return {name: st[name] for name in ("dist", "status", "ref_consumed", "n_runs", "runs")}
    db = st["db"]
    if case["graph"]:
        st["graph"].launch()
    else:
        db.pack()
        if case["span"]:
            db.align_locate(stats=False)
        elif case["order"]:
            db.align_order(case["order"], stats=False)
        elif case["noalloc"]:
            ga.ga_align_batch_noalloc(db.reads, db.read_off, db.read_len, db.refs, db.ref_off,
                                      db.ref_len, db.n, db.W, db.O, db.k, db.dist, db.status,
                                      db.ref_consumed, db.cigar, db.cigar_off, db.n_runs, None, None)
        else:
            db.align("batched", stats=False)
    ga.ga_cigar_compact(db.cigar, db.cigar_off, db.n_runs, db.n, st["runs"], st["cap"],
                        st["run_off"], st["compact_ws"], st["compact_bytes"])
    out = {"dist": db.dist, "status": db.status, "ref_consumed": db.ref_consumed,
           "run_off": st["run_off"], "runs": st["runs"]}
    if case["span"]:
        out["ref_start"] = db.ref_start
    return out


def work(case):
    """Bytes: the ASCII sequences read once, the results written once (about 0.3
    CIGAR runs a read base where the windows follow the read, 0.6 where an
    anchored window meets the random flank, 0.1 in short reads). Operations:
    32-bit integer operations of the windows' edit-distance columns, ten for
    every 32 rows of a column, W columns in each window of W - O bases."""
    if case["kind"] == "pack":
        return {"bytes": 1.25 * case["n"], "flops": 0}
    if case["kind"] == "serve":
        n, lo, hi, W, O = case["requests"] * (case["pairs"] + 1) / 2, case["lo"], case["hi"], 64, 24
        mean, free, long_ = (hi - lo) / math.log(hi / lo), False, hi >= 1000
    else:
        n, W, O = case["n"], case["W"], case["O"]
        mean, free, long_ = _mean_len(case), case["span"], case["hi"] >= 1000
    bases = n * mean
    runs = 0.1 if not long_ else 0.3 if free else 0.6
    ref = bases * (1.08 if long_ else 1.0)
    ops = bases / (W - O) * W * 10 * math.ceil(W / 32)
    return {"bytes": bases + ref + 4 * runs * bases + 20 * n, "flops": ops}


def exact(case, seed):
    """Every output is a whole number and has to be equal: there is no rounding to measure."""
    return None
