"""Contiguous systems of up to 256 rows (FP32: 512) that are no whole 16-byte
vectors, brought to shared memory element by element (k_lines_staged) or read
directly (k_lines), against the FP64 oracle: lengths around every change of the lanes
per system, system counts that fill no warp or block, unaligned arrays, stored
and accumulated, with values outside the systems that must not be used.  GPU
only."""
import numpy as np
import pytest

import oracle
from paper_2201_03950_gb300 import inputs, trid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {np.float32: 1e-5, np.float64: 1e-12}


def run(n, nsys, dtype, acc, offset=0):
    total = n * nsys
    a, b, c, d = inputs.dominant_system((total,), seed=n + nsys, dtype=dtype)
    ref = oracle.solve_mesh(a, b, c, d, (n, nsys), 0)
    a.reshape(nsys, n)[:, 0] = np.nan       # not part of the systems
    c.reshape(nsys, n)[:, -1] = np.nan
    guard = 40

    def dev(v):     # with NaN before and behind
        t = torch.full((total + offset + guard,), float("nan"),
                       dtype=torch.float32 if dtype is np.float32 else torch.float64, device="cuda")
        t[offset:offset + total] = torch.from_numpy(v)
        return t, t[offset:offset + total]

    bufs = [dev(v) for v in (a, b, c, d)]
    u0 = inputs.random_rhs((total,), seed=3, dtype=dtype)
    ub = dev(u0)
    views = [v for _, v in bufs]
    out = ub if acc else bufs[3]
    trid.solve(*views, (n, nsys), 0, u=ub[1] if acc else None)
    got = out[1].cpu().numpy().astype(np.float64) - (u0.astype(np.float64) if acc else 0.0)
    rest = torch.cat([out[0][:offset], out[0][offset + total:]])
    assert bool(torch.isnan(rest).all())     # nothing written outside the array
    assert np.max(np.abs(got - ref)) <= TOL[dtype] * np.max(np.abs(ref))


LENGTHS = [1, 2, 3, 5, 7, 9, 13, 15, 17, 31, 33, 63, 65, 101, 127, 129, 201, 250, 255]


@pytest.mark.parametrize("dtype", [np.float32, np.float64], ids=["f32", "f64"])
@pytest.mark.parametrize("acc", [False, True], ids=["store", "acc"])
@pytest.mark.parametrize("n", LENGTHS)
def test_lengths(n, acc, dtype):
    for nsys in (1, 3, 131):
        run(n, nsys, dtype, acc)


@pytest.mark.parametrize("dtype", [np.float32, np.float64], ids=["f32", "f64"])
@pytest.mark.parametrize("n", [4, 8, 16, 64, 128, 256])
def test_unaligned_arrays(n, dtype):
    for acc in (False, True):
        run(n, 70, dtype, acc, offset=1)


@pytest.mark.parametrize("acc", [False, True], ids=["store", "acc"])
@pytest.mark.parametrize("n", [257, 260, 271, 272, 300, 301, 384, 497, 508, 511, 512, 513, 516])
def test_sixteen_rows_per_lane(n, acc):
    for nsys in (1, 2, 5, 131):
        run(n, nsys, np.float32, acc)
    run(n, 9, np.float32, acc, offset=1)
