"""Systems of 257 to 4096 rows (FP32: 8192) in one pass (k_team), against the FP64
oracle: row counts around every number of tiles per warp and every number of
systems per block, contiguous in whole vectors and not, strided, system counts
that fill no block, weakly coupled and nearly singular systems, and the limits
beyond which the passes through scratch run.  GPU only."""
import numpy as np
import pytest

import oracle
from paper_2201_03950_gb300 import inputs, trid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def solve(dims, k, acc=False, offset=0, margin=None, dtype=np.float64, out_offset=None):
    n = int(np.prod(dims))
    a, b, c, d = inputs.dominant_system((n,), seed=n + k, dtype=dtype)
    if margin is not None:
        b = np.abs(a) + np.abs(c) + margin
    idx = np.moveaxis(np.arange(n).reshape(dims[::-1]), len(dims) - 1 - k, 0)
    ref = oracle.solve_mesh(a, b, c, d, dims, k)
    a[idx[0].reshape(-1)] = np.nan     # not part of the system, so never used
    c[idx[-1].reshape(-1)] = np.nan

    def dev(v, offset=offset):
        v = torch.from_numpy(v)
        return torch.empty(n + offset, dtype=v.dtype, device="cuda")[offset:].copy_(v)

    ta, tb, tc, td = (dev(v) for v in (a, b, c, d))
    u0 = inputs.random_rhs((n,), seed=5, dtype=dtype) if acc else np.zeros(n, dtype)
    tu = dev(u0, offset if out_offset is None else out_offset) if acc else None
    out = trid.solve(ta, tb, tc, td, dims, k, u=tu)
    if acc:
        assert np.array_equal(td.cpu().numpy(), d)
    return out.cpu().numpy() - u0, ref


def check(got, ref, tol=1e-12):
    assert np.all(np.isfinite(got))
    assert np.max(np.abs(got - ref)) <= tol * np.max(np.abs(ref))


ROWS = [257, 260, 271, 272, 273, 300, 511, 512, 513, 700, 1001, 1024, 1536, 2047, 3072, 3073, 4095,
        4096, 4097]


@pytest.mark.parametrize("n", ROWS)
@pytest.mark.parametrize("acc", [False, True], ids=["store", "acc"])
def test_rows(n, acc):
    check(*solve((n, 7), 0, acc))
    check(*solve((7, n), 1, acc))


@pytest.mark.parametrize("n", [300, 400, 512, 700, 1000])
def test_many_systems(n):
    check(*solve((n, 2503), 0))          # several systems per block, the last block not full
    check(*solve((2503, n), 1))
    check(*solve((13, n, 197), 1))       # neighbours across the rows of a plane


def test_unaligned_arrays():
    check(*solve((512, 40), 0, offset=1))
    check(*solve((40, 512), 1, offset=1))


@pytest.mark.parametrize("margin,tol", [(1e-3, 1e-10), (1e-6, 1e-7)])
def test_weak_dominance(margin, tol):
    """Couplings that stay above the stopping bound for every round; the
    condition number (at most 3 / margin) times 2^-53, a few hundred times over."""
    check(*solve((1500, 9), 0, margin=margin), tol=tol)
    check(*solve((9, 1500), 1, margin=margin), tol=tol)


@pytest.mark.parametrize("n", [513, 1023, 1025, 1537, 2049, 4095, 4097, 4100, 5000, 8176, 8191, 8192, 8193])
@pytest.mark.parametrize("acc", [False, True], ids=["store", "acc"])
def test_fp32(n, acc):
    """The oracle in FP64 from the same FP32 arrays; 1e-5 of the largest value is
    about 80 units of 2^-23, for a condition number of at most 3 and the sum."""
    f = np.float32
    check(*solve((n, 7), 0, acc, dtype=f), tol=1e-5)
    check(*solve((n, 611), 0, acc, offset=1, dtype=f), tol=1e-5)
    check(*solve((7, n), 1, acc, dtype=f), tol=1e-5)
    check(*solve((307, n), 1, acc, dtype=f), tol=1e-5)


def test_fp32_unaligned_out():
    """Beyond 4096 rows the same kernel, so the same bits, as into an aligned
    array; below, the aligned call runs another kernel and both are held to the
    bound of test_fp32."""
    f = np.float32
    check(*solve((600, 40), 0, True, offset=0, dtype=f, out_offset=1), tol=1e-5)
    got, ref = solve((5000, 40), 0, True, dtype=f, out_offset=1)
    check(got, ref, tol=1e-5)
    assert np.array_equal(got, solve((5000, 40), 0, True, dtype=f)[0])


@pytest.mark.parametrize("which", ["a", "b", "c"])
@pytest.mark.parametrize("dims,k,dtype", [((3000, 5), 0, np.float64), ((5, 3000), 1, np.float64),
                                          ((700, 9), 0, np.float64), ((5000, 3), 0, np.float32),
                                          ((1001, 5), 0, np.float32), ((41, 1500), 1, np.float32)])
def test_a_coefficient_that_is_no_number_spoils_its_whole_system(dims, k, dtype, which):
    """And no other one, as in the passes: no value of it is determined."""
    n = int(np.prod(dims))
    v = dict(zip("abcd", inputs.dominant_system((n,), seed=1, dtype=dtype)))
    idx = np.moveaxis(np.arange(n).reshape(dims[::-1]), len(dims) - 1 - k, 0)
    v[which][idx[dims[k] // 2, 2]] = np.nan
    t = [torch.from_numpy(x).cuda() for x in v.values()]
    x = trid.solve(*t, dims, k).cpu().numpy()[idx]
    assert np.all(np.isnan(x[:, 2]))
    assert np.all(np.isfinite(np.delete(x, 2, axis=1)))
