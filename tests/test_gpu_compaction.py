"""GPU tests of the CIGAR compaction at the sizes where its launch changes: tiles of
8, 16, 32 and 64 pairs, chunk sums added up by the blocks and scanned, and CIGARs on
both sides of the mean of 64 runs that decides how a tile is copied."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2203_15561_gb300 as ga  # noqa: E402


@pytest.mark.parametrize("n", [1, 1024, 1025, 10_000, 10_001, 20_001, 40_001, 80_001, 262_144, 262_145])
@pytest.mark.parametrize("most", [1, 9, 126, 130, 700])
def test_launch_sizes(n, most):
    if n * most > 20_000_000:
        most = max(1, 20_000_000 // n)
    rng = np.random.default_rng(n + most)
    runs = rng.integers(0, most + 1, n).astype(np.int64)
    runs[rng.random(n) < 0.1] = 0
    if n > 100:  # some tiles of nothing, one of a single long CIGAR
        runs[50:120] = 0
        runs[n - 5] = 5000
    cap = runs + rng.integers(0, 3, n)
    off = np.concatenate([[0], np.cumsum(cap)]).astype(np.int64)
    src = torch.randint(0, 1 << 30, (int(off[-1]) + 1,), dtype=torch.int32, device="cuda",
                        generator=torch.Generator(device="cuda").manual_seed(n))
    total = int(runs.sum())
    start = np.concatenate([[0], np.cumsum(runs)])
    want = src.cpu().numpy()[np.repeat(off[:-1] - start[:-1], runs) + np.arange(total)]
    ws_bytes = ga.ga_cigar_compact_workspace_size(n)
    ws = torch.full((ws_bytes,), 0xEE, dtype=torch.uint8, device="cuda")
    out = torch.full((total + 8,), -9, dtype=torch.int32, device="cuda")
    out_off = torch.full((n + 2,), -9, dtype=torch.int64, device="cuda")
    ga.ga_cigar_compact(src, torch.from_numpy(off).cuda(), torch.from_numpy(runs.astype(np.int32)).cuda(), n, out,
                        total, out_off, ws, ws_bytes)
    np.testing.assert_array_equal(out_off.cpu().numpy()[:-1], start)
    assert int(out_off[-1]) == -9
    np.testing.assert_array_equal(out.cpu().numpy()[:total], want)
    assert (out.cpu().numpy()[total:] == -9).all()
