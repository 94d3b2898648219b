"""The FP64 reciprocal of the solves over the exponent range: systems scaled to
its ends, where the reciprocal of the pivots falls back to the quotient, give
the oracle's solution; and the reciprocal itself, which systems of one row with
right-hand side 1 return, against the quotient.  GPU only."""
import numpy as np
import pytest

import oracle
from paper_2201_03950_gb300 import inputs, trid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponent", [-1020, -1000, 0, 1000, 1019])
@pytest.mark.parametrize("dims,k", [((40, 60), 0), ((24, 40), 1), ((70, 40, 70), 1), ((700, 9), 0)])
def test_scaled_systems(dims, k, exponent):
    n = int(np.prod(dims))
    a, b, c, d = (v * 2.0 ** exponent
                  for v in inputs.dominant_system((n,), seed=n, dtype=np.float64))
    ref = oracle.solve_mesh(a, b, c, d, dims, k)
    ta, tb, tc, td = (torch.from_numpy(v).cuda() for v in (a, b, c, d))
    trid.solve(ta, tb, tc, td, dims, k)
    got = td.cpu().numpy()
    assert np.all(np.isfinite(got))
    # rounding of the reciprocals by one ulp more or less: a few hundred ulp at most
    assert np.max(np.abs(got - ref)) <= 1e-13 * np.max(np.abs(ref))


def reciprocals(b):
    n = b.size
    zero = torch.zeros(n, dtype=torch.float64, device="cuda")
    x = torch.ones(n, dtype=torch.float64, device="cuda")
    trid.solve(zero, torch.from_numpy(b).cuda(), zero, x, (1, n), 0)
    return x.cpu().numpy()


def test_reciprocal_is_within_one_ulp():
    """The cubic step's error is below 2^-59 before its one rounding, so it is the
    quotient or its neighbour: 0.5 + 2^-7 ulp at most, which rounds otherwise than
    the quotient for at most 2^-6 of all arguments (measured: 3 in 10^4)."""
    rng = np.random.default_rng(0)
    n = 1 << 22
    b = rng.uniform(1.0, 2.0, n) * 2.0 ** rng.integers(-1000, 1001, n) * rng.choice([-1.0, 1.0], n)
    got, ref = reciprocals(b), 1.0 / b
    off = np.abs(got.view(np.int64) - ref.view(np.int64))
    assert off.max() <= 1
    assert np.mean(off != 0) <= 1e-3


def test_reciprocal_of_special_arguments():
    tiny = np.finfo(np.float64).tiny
    b = np.array([1.0, -1.0, 2.0, 0.5, 2.0 ** 1000, 2.0 ** -1000, tiny, -tiny, tiny / 4, 2.0 ** 1023,
                  1.5 * 2.0 ** 1023, np.finfo(np.float64).max, 0.0, -0.0, np.inf, -np.inf, np.nan])
    with np.errstate(divide="ignore", over="ignore"):
        ref = 1.0 / b
    assert np.array_equal(reciprocals(b)[np.isfinite(ref)], ref[np.isfinite(ref)])
    assert not np.any(np.isfinite(reciprocals(b)[~np.isfinite(ref)]))
