"""Strided systems longer than 256 rows (y/z axes), FP32: the cluster path
(one CTA per chunk of 256 rows, 512 above 2048, the chunks' responses to the
unknowns outside them joined by a chunk-level solve across the cluster) for up
to 4096 rows, the block per few systems that takes up to 1024 rows when there
are few of them, and the passes beyond.  Whole meshes against the FP64 oracle,
element by element: ragged last chunks of 1, 255 and 4 rows, mesh widths that
leave partial 16-wide strips, several outer slices, accumulate mode, the unread
a of first rows and c of last rows poisoned with NaN.  GPU only."""
import numpy as np
import pytest

import oracle
from graphs import graph_text
from paper_2201_03950_gb300 import inputs, trid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5


def normwise(x, ref):
    x = np.asarray(x, dtype=np.float64)
    ref = np.asarray(ref, dtype=np.float64)
    return float(np.max(np.abs(x - ref)) / max(np.max(np.abs(ref)), 1e-300))


def poison(ta, tc, dims, k):
    total = int(np.prod(dims))
    n = dims[k]
    idx = np.arange(total).reshape(tuple(reversed(dims)))
    ax = len(dims) - 1 - k
    first = np.take(idx, 0, axis=ax).reshape(-1)
    last = np.take(idx, n - 1, axis=ax).reshape(-1)
    ta[torch.from_numpy(first).cuda()] = float("nan")
    tc[torch.from_numpy(last).cuda()] = float("nan")


CASES = [((16, 257), 1), ((32, 512), 1), ((20, 513), 1), ((16, 511), 1), ((48, 769), 1),
         ((16, 8, 300), 2), ((20, 700, 3), 1), ((4, 6, 1030), 2), ((16, 4100), 1),
         ((40, 9000), 1), ((64, 2048), 1), ((16, 3000), 1), ((32, 4096), 1), ((24, 5, 3900), 2)]


@pytest.mark.parametrize("dims,k", CASES, ids=[f"{'x'.join(map(str, d))}-dim{k}" for d, k in CASES])
def test_against_oracle(dims, k):
    total = int(np.prod(dims))
    a, b, c, d = inputs.dominant_system((total,), seed=total % 997, dtype=np.float32)
    ref = oracle.solve_mesh(a, b, c, d, dims, k)
    ta, tb, tc, td = (torch.from_numpy(v).cuda() for v in (a, b, c, d))
    poison(ta, tc, dims, k)
    trid.solve(ta, tb, tc, td, dims, k)
    torch.cuda.synchronize()
    assert normwise(td.cpu().numpy(), ref) <= TOL


@pytest.mark.parametrize("dims,k", [((32, 600), 1), ((16, 4, 1024), 2)], ids=str)
def test_accumulate(dims, k):
    total = int(np.prod(dims))
    a, b, c, d = inputs.dominant_system((total,), seed=5, dtype=np.float32)
    ref = oracle.solve_mesh(a, b, c, d, dims, k)
    u0 = inputs.random_rhs((total,), seed=6, dtype=np.float32)
    ta, tb, tc, td, tu = (torch.from_numpy(v).cuda() for v in (a, b, c, d, u0))
    d0 = td.clone()
    trid.solve(ta, tb, tc, td, dims, k, u=tu)
    torch.cuda.synchronize()
    assert torch.equal(td, d0)
    got = tu.cpu().numpy().astype(np.float64) - u0.astype(np.float64)
    assert normwise(got, ref) <= TOL


def many(n):
    """Systems of n rows enough for clusters: more than two strips of 16 per SM."""
    return 16 * (2 * torch.cuda.get_device_properties(0).multi_processor_count + 1) + 4


@pytest.mark.parametrize("n", [257, 300, 512, 513, 767, 768])
@pytest.mark.parametrize("acc", [False, True], ids=["store", "acc"])
@pytest.mark.filterwarnings("ignore:DEBUG")
def test_clusters_of_two_and_three(n, acc, tmp_path):
    dims = (many(n), n)
    total = dims[0] * n
    a, b, c, d = inputs.dominant_system((total,), seed=n, dtype=np.float32)
    ref = oracle.solve_mesh(a, b, c, d, dims, 1)
    ta, tb, tc, td = (torch.from_numpy(v).cuda() for v in (a, b, c, d))
    poison(ta, tc, dims, 1)
    u = torch.zeros_like(td) if acc else None
    x = td.clone()
    got = trid.solve(ta, tb, tc, x, dims, 1, u=u)
    assert normwise(got.cpu().numpy(), ref) <= TOL
    assert "k_chunk_cluster" in graph_text(lambda: trid.solve(ta, tb, tc, x, dims, 1, u=u),
                                           tmp_path / "graph.dot")


@pytest.mark.parametrize("dims", [(8192, 512), (3000, 1400), (4096, 2048), (4096, 4096)])
def test_stored_many_strips_repeated(dims):
    """Several strips of systems per cluster, stored, twenty times from inputs that
    stay in the L2 cache (the smaller ones): the copy of a strip must not overtake
    the reads of the strip before it."""
    n = int(np.prod(dims))
    a, b, c, d = inputs.dominant_system((n,), seed=11, dtype=np.float32)
    ta, tb, tc, td = (torch.from_numpy(v).cuda() for v in (a, b, c, d))
    ref = torch.from_numpy(oracle.solve_mesh(a, b, c, d, dims, 1)).cuda()
    scale = ref.abs().max()
    x = torch.empty_like(td)
    for _ in range(20):
        trid.solve(ta, tb, tc, x.copy_(td), dims, 1)
        assert ((x - ref).abs().max() / scale).item() <= TOL


def test_weak_dominance():
    """Diagonal dominance margin 0.01 instead of 0.5..1.5: the responses to
    the outside unknowns decay slowly across a chunk, and the chunk-level
    system carries them over many chunks."""
    dims, k = (32, 1500), 1
    total = dims[0] * dims[1]
    rng = np.random.default_rng(9)
    a = rng.uniform(-1, -0.1, total)
    c = rng.uniform(-1, -0.1, total)
    b = np.abs(a) + np.abs(c) + 0.01
    d = rng.uniform(-1, 1, total)
    a, b, c, d = (v.astype(np.float32) for v in (a, b, c, d))
    ref = oracle.solve_mesh(a, b, c, d, dims, k)
    ta, tb, tc, td = (torch.from_numpy(v).cuda() for v in (a, b, c, d))
    trid.solve(ta, tb, tc, td, dims, k)
    torch.cuda.synchronize()
    # the condition number grows as the margin shrinks, so the well-
    # conditioned tolerance does not apply; per system, check the FP32
    # backward error (normwise residual) and the forward error against
    # kappa_inf(A) times that backward error bound, both computed here
    x = td.cpu().numpy().astype(np.float64)
    assert np.all(np.isfinite(x))
    eps = float(np.finfo(np.float32).eps)
    bwd_bound = 64 * eps
    n = dims[1]
    for s in range(dims[0]):
        idx = s + dims[0] * np.arange(n)
        A = np.diag(b[idx].astype(np.float64))
        A[np.arange(1, n), np.arange(n - 1)] = a[idx][1:]
        A[np.arange(n - 1), np.arange(1, n)] = c[idx][:-1]
        xs, rs, ds = x[idx], ref[idx], d[idx].astype(np.float64)
        anorm = np.max(np.sum(np.abs(A), axis=1))
        resid = np.max(np.abs(A @ xs - ds)) / (anorm * np.max(np.abs(xs)) + np.max(np.abs(ds)))
        assert resid <= bwd_bound, (s, resid)
        kappa = anorm * np.max(np.sum(np.abs(np.linalg.inv(A)), axis=1))
        fwd = np.max(np.abs(xs - rs)) / np.max(np.abs(rs))
        assert fwd <= kappa * bwd_bound, (s, fwd, kappa)
