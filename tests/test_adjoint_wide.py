"""Adjoint along strided systems that each span 48 MiB or more, and just less:
32 instead of 16 neighbouring systems per block (k_adjoint_strided), on row
counts of every tile count and neighbour counts that fill no block, sampled
systems against the FP64 oracle.  GPU only."""
import numpy as np
import pytest

import oracle
from graphs import graph_text
from paper_2201_03950_gb300 import trid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

def span(n):   # elements
    return ((51 if n > 128 else 48) << 20) // 4


@pytest.mark.parametrize("n", [3, 8, 9, 17, 40, 100, 256])
@pytest.mark.parametrize("below", [False, True], ids=["wide", "narrower"])
def test_sampled_systems(n, below):
    inner = span(n) // n - 1 if below else span(n) // n + 5
    dims = (inner, n)
    g = torch.Generator(device="cuda").manual_seed(n)

    def rand():
        return torch.rand(inner * n, generator=g, device="cuda")

    a, c = -0.1 - 0.9 * rand(), -0.1 - 0.9 * rand()
    b = a.abs() + c.abs() + 0.5 + rand()
    x, gx = 2 * rand() - 1, 2 * rand() - 1
    got = trid.adjoint(a, b, c, x, gx, dims, 1)
    pick = np.unique(np.concatenate([[0, 15, 16, 31, 32, inner - 1, inner - 2],
                                     np.random.default_rng(n).integers(0, inner, 40)]))
    at = torch.from_numpy(pick).cuda()
    cols = [v.view(n, inner)[:, at].cpu().numpy() for v in (a, b, c, x, gx) + tuple(got)]
    for k in range(len(pick)):
        ref = oracle.adjoint(*(np.ascontiguousarray(v[:, k], dtype=np.float64) for v in cols[:5]))
        for r, v in zip(ref, cols[5:]):
            assert np.max(np.abs(v[:, k] - r)) <= 2e-5 * max(np.max(np.abs(r)), 1e-30)


@pytest.mark.filterwarnings("ignore:DEBUG")
@pytest.mark.parametrize("n,mib,threads", [(256, 50, 512), (256, 52, 1024), (128, 49, 512), (128, 47, 256)])
def test_systems_per_block(n, mib, threads, tmp_path):
    inner = (mib << 20) // 4 // n
    t = [torch.rand(inner * n, device="cuda") + 2 * (k == 1) for k in range(5)]
    text = graph_text(lambda: trid.adjoint(*t, (inner, n), 1), tmp_path / "graph.dot")
    assert f",{threads},0\\>" in text
