"""The plan of an uneven batch at the system counts where its form changes: one
cluster up to 65536 systems (a block's threads, all blocks' threads, several
systems per thread), separate launches above; every system solved against the
FP64 oracle, empty ones among them, and invalid ranges skipped and reported.
GPU only."""
import numpy as np
import pytest

import oracle
from paper_2201_03950_gb300 import inputs, trid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nsys", [1, 31, 33, 1023, 1024, 1025, 8191, 8192, 8193, 20000, 65535, 65536,
                                  65537])
def test_system_counts(nsys):
    rng = np.random.default_rng(nsys)
    lens = rng.integers(0, 12, nsys)
    some = rng.integers(0, nsys, 12)
    lens[some] = rng.integers(1, 1500, 12)
    lens[rng.integers(0, nsys)] = 5000
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    a, b, c, d = inputs.dominant_system((int(off[-1]),), seed=nsys, dtype=np.float32)
    t = [torch.from_numpy(v).cuda() for v in (a, b, c, d)]
    ws = torch.full((trid.varlen_workspace_bytes(nsys),), 255, dtype=torch.uint8, device="cuda")
    # the second and third call find the plan of another division of the same rows
    # in the workspace
    for o in (off, np.concatenate([[0], np.cumsum(lens[::-1])]).astype(np.int64), off):
        ref = oracle.solve_varlen(a, b, c, d, o)
        x = t[3].clone()
        trid.solve_varlen(*t[:3], x, torch.from_numpy(o).cuda(), int(lens.max()), workspace=ws)
        assert np.max(np.abs(x.cpu().numpy() - ref)) <= 1e-5 * np.max(np.abs(ref))
    assert trid.device_status() == 0


def test_invalid_ranges_are_skipped_and_reported():
    off = np.array([0, 5, 9, 30, 20, 40, 1000, 45, 50], dtype=np.int64)   # 30..20, 40..1000, 1000..45
    a, b, c, d = inputs.dominant_system((50,), seed=1, dtype=np.float32)
    t = [torch.from_numpy(v).cuda() for v in (a, b, c, d)]
    trid.solve_varlen(*t, torch.from_numpy(off).cuda(), 64)
    assert trid.device_status() == 1
    got = t[3].cpu().numpy()
    for s, e in ((0, 5), (5, 9), (45, 50)):
        ref = oracle.solve_varlen(a[s:e], b[s:e], c[s:e], d[s:e], np.array([0, e - s], dtype=np.int64))
        assert np.max(np.abs(got[s:e] - ref)) <= 1e-5 * np.max(np.abs(ref))
