"""The FP64 reciprocal of the solves over the exponent range: systems scaled to
its ends, where the reciprocal of the pivots falls back to the quotient, give
the oracle's solution.  GPU only."""
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
