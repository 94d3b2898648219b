"""Solves that add into u, by the paths that load u's rows together before they
store them: uneven batches, thread-block clusters, the passes for the longest
systems; u on a 16-byte boundary and (meshes) not.  Against the FP64 oracle.  GPU only."""
import numpy as np
import pytest

import oracle
from paper_2201_03950_gb300 import inputs, trid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {np.float32: 1e-5, np.float64: 1e-12}   # of the largest value, as everywhere


def dev(v, offset=0):
    t = torch.from_numpy(v)
    return torch.empty(v.size + offset, dtype=t.dtype, device="cuda")[offset:].copy_(t)


def check(got, u0, ref, dtype):
    x = got.cpu().numpy().astype(np.float64) - u0.astype(np.float64)
    # the sum is rounded once, at most half an ulp of |u| + |x| (inside TOL)
    assert np.max(np.abs(x - ref)) <= TOL[dtype] * max(np.max(np.abs(ref)), 1.0)


@pytest.mark.parametrize("dtype", [np.float32, np.float64], ids=["f32", "f64"])
def test_varlen(dtype):
    lengths = [1, 7, 8, 9, 31, 248, 249, 255, 511, 1016, 1017, 2047, 4088, 4089, 9001, 3, 16384, 0, 5]
    off = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    n = int(off[-1])
    a, b, c, d = inputs.dominant_system((n,), seed=7, dtype=dtype)
    u0 = inputs.random_rhs((n,), seed=8, dtype=dtype)
    u = dev(u0)
    trid.solve_varlen(dev(a), dev(b), dev(c), dev(d), torch.from_numpy(off).cuda(), max(lengths), u=u)
    check(u, u0, oracle.solve_varlen(a, b, c, d, off), dtype)


@pytest.mark.parametrize("dtype", [np.float32, np.float64], ids=["f32", "f64"])
@pytest.mark.parametrize("dims,k", [((36, 1025), 1), ((20, 4095), 1), ((20, 4096), 1), ((400, 1500), 1),
                                    ((9001, 5), 0), ((9004, 5), 0), ((5, 9001), 1)])
@pytest.mark.parametrize("offset", [0, 1])
def test_mesh(dtype, dims, k, offset):
    n = int(np.prod(dims))
    a, b, c, d = inputs.dominant_system((n,), seed=n, dtype=dtype)
    u0 = inputs.random_rhs((n,), seed=9, dtype=dtype)
    u = dev(u0, offset)
    trid.solve(dev(a), dev(b), dev(c), dev(d), dims, k, u=u)
    check(u, u0, oracle.solve_mesh(a, b, c, d, dims, k), dtype)


@pytest.mark.parametrize("dims", [(8192, 512), (3000, 1400), (4096, 2048)])
def test_clusters_many_strips(dims):
    """Several strips of systems per cluster, ten times: the copy of a strip must
    not overtake the reads of the strip before it."""
    n = int(np.prod(dims))
    a, b, c, d = inputs.dominant_system((n,), seed=11, dtype=np.float32)
    u0 = inputs.random_rhs((n,), seed=12, dtype=np.float32)
    ref = oracle.solve_mesh(a, b, c, d, dims, 1)
    ta, tb, tc, td = (dev(v) for v in (a, b, c, d))
    for _ in range(10):
        u = dev(u0)
        trid.solve(ta, tb, tc, td, dims, 1, u=u)
        check(u, u0, ref, np.float32)
