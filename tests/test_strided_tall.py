"""Strided FP32 systems of 257 to 1024 rows with 16, 24 or 32 rows per thread
(k_strided), against the FP64 oracle: row counts around every tile height,
system counts on both sides of each choice (8 or 16 systems per block, clusters
instead), neighbours that fill no block, aligned for the clusters and not,
stored and accumulated.  GPU only."""
import numpy as np
import pytest

import oracle
from paper_2201_03950_gb300 import inputs, trid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def run(dims, acc):
    n = int(np.prod(dims))
    a, b, c, d = inputs.dominant_system((n,), seed=n, dtype=np.float32)
    ref = oracle.solve_mesh(a, b, c, d, dims, 1)
    a.reshape(dims[::-1])[..., 0, :] = np.nan      # not part of the systems
    c.reshape(dims[::-1])[..., -1, :] = np.nan
    ta, tb, tc, td = (torch.from_numpy(v).cuda() for v in (a, b, c, d))
    u0 = inputs.random_rhs((n,), seed=2, dtype=np.float32)
    tu = torch.from_numpy(u0).cuda() if acc else None
    got = trid.solve(ta, tb, tc, td, dims, 1, u=tu).cpu().numpy().astype(np.float64)
    if acc:
        assert np.array_equal(td.cpu().numpy(), d)
        got = got - u0
    assert np.max(np.abs(got - ref)) <= 1e-5 * np.max(np.abs(ref))


@pytest.mark.parametrize("acc", [False, True], ids=["store", "acc"])
@pytest.mark.parametrize("n", [257, 300, 496, 512, 513, 700, 768, 769, 1000, 1023, 1024, 1025])
def test_rows(n, acc):
    run((520, n), acc)
    run((37, n, 15), acc)        # rows that are no multiple of 16 bytes, three dimensions


@pytest.mark.parametrize("acc", [False, True], ids=["store", "acc"])
@pytest.mark.parametrize("n", [260, 600, 800])
@pytest.mark.parametrize("nsys", [4, 504, 1216, 1224, 2432, 2436, 4868, 1229, 5001])
def test_system_counts(nsys, n, acc):
    run((nsys, n), acc)


@pytest.mark.parametrize("dims", [(1000, 300), (1024, 700), (1024, 1000), (2048, 900), (4864, 512),
                                  (5000, 600), (37, 800), (1001, 1001), (4700, 200), (4865, 256),
                                  (7400, 250), (9800, 256), (4800, 100)])
def test_stored_and_accumulated_bits_agree(dims):
    """The differentiable ADI recomputes with stored solves what its forward
    accumulated (u = 0 + x), also into an array of another alignment."""
    for dtype, tdt in ((np.float32, torch.float32), (np.float64, torch.float64)):
        n = int(np.prod(dims))
        ta, tb, tc, td = (torch.from_numpy(v).cuda()
                          for v in inputs.dominant_system((n,), seed=n, dtype=dtype))
        for offset in (0, 1):
            u = torch.zeros(n + offset, dtype=tdt, device="cuda")[offset:]
            trid.solve(ta, tb, tc, td, dims, 1, u=u)
            x = trid.solve(ta, tb, tc, td.clone(), dims, 1)
            assert torch.equal(u, x)


@pytest.mark.parametrize("dims", [(64, 700), (2048, 900), (200, 1000)])
def test_checkpoint_spacing_gives_the_same_bits(dims):
    n = dims[0] * dims[1]
    u0 = torch.from_numpy(inputs.target_field(dims, seed=1, dtype=np.float32)).cuda()
    kap = torch.from_numpy(inputs.diffusivity_field(dims, seed=2, dtype=np.float32)).cuda()
    g = torch.from_numpy(inputs.random_rhs((n,), seed=3, dtype=np.float32)).cuda()
    res = []
    for every in (1, 2, 4):
        uT, ck = trid.adi2v_forward(u0, kap, dims, 0.2, 4, every)
        gu, gk, _ = trid.adi2v_backward(g, kap, dims, 0.2, 4, every, ck)
        res.append((uT, gu, gk))
    for r in res[1:]:
        assert all(torch.equal(x, y) for x, y in zip(r, res[0]))
