"""FP64 systems of up to 256 rows in large numbers, solved from both ends
(k_twist), against the FP64 oracle: both forms of access (contiguous whole
vectors, strided), stored and accumulated, at the row counts where the halves
are uneven, empty or whole vectors, with system counts that fill no warp, and
the calls just outside the rule.  Also the reciprocal's range: systems scaled
to the ends of the exponent range.  GPU only."""
import numpy as np
import pytest

import oracle
from paper_2201_03950_gb300 import inputs, trid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def solve(dims, k, acc=False, offset=0):
    n = int(np.prod(dims))
    a, b, c, d = inputs.dominant_system((n,), seed=n + k, dtype=np.float64)
    idx = np.moveaxis(np.arange(n).reshape(dims[::-1]), len(dims) - 1 - k, 0)
    ref = oracle.solve_mesh(a, b, c, d, dims, k)
    a[idx[0].reshape(-1)] = np.nan     # not part of the system, so never used
    c[idx[-1].reshape(-1)] = np.nan

    def dev(v):
        t = torch.empty(n + offset, dtype=torch.float64, device="cuda")[offset:]
        return t.copy_(torch.from_numpy(v))

    ta, tb, tc, td = (dev(v) for v in (a, b, c, d))
    if acc:
        u0 = inputs.random_rhs((n,), seed=5, dtype=np.float64)
        tu = dev(u0)
        trid.solve(ta, tb, tc, td, dims, k, u=tu)
        assert np.array_equal(td.cpu().numpy(), d)
        return tu.cpu().numpy() - u0, ref
    trid.solve(ta, tb, tc, td, dims, k)
    return td.cpu().numpy(), ref


def check(got, ref):
    assert np.all(np.isfinite(got))
    assert np.max(np.abs(got - ref)) <= 1e-13 * np.max(np.abs(ref))


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 8, 9, 15, 16, 31, 100, 129, 255, 256])
@pytest.mark.parametrize("acc", [False, True], ids=["store", "acc"])
def test_strided(n, acc):
    check(*solve((67, n, 69), 1, acc))       # 4623 systems, 67 neighbours
    check(*solve((4609, n), 1, acc))


@pytest.mark.parametrize("n", [4, 8, 12, 16, 20, 100, 252, 256])
@pytest.mark.parametrize("acc", [False, True], ids=["store", "acc"])
def test_contiguous(n, acc):
    check(*solve((n, 6145), 0, acc))


@pytest.mark.parametrize("dims,k", [((254, 6145), 0), ((64, 6143), 0), ((40, 64, 115), 1)])
def test_just_outside(dims, k):
    check(*solve(dims, k))


def test_unaligned_arrays():
    check(*solve((64, 6200), 0, offset=1))   # not 32-byte aligned: the tiled kernel
    check(*solve((71, 64, 70), 1, offset=1))
