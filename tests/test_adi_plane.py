"""Batches of small 2D meshes whose steps all run on chip with two threads per
line (k_adi_plane), against the FP64 oracle: extents around the multiples of
32 that select the kernel, odd and even, the smallest and largest, elongated
ones, more meshes than blocks, operators from weak to strong coupling, and
values outside the field (corners, another mesh) that must not enter it.
GPU only."""
import numpy as np
import pytest

import oracle
from paper_2201_03950_gb300 import inputs, trid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {np.float32: 1e-5, np.float64: 1e-12}


def batch(dims, nb, seed, dtype):
    rng = np.random.default_rng(seed)
    n = int(np.prod(dims))
    return np.concatenate([inputs.sine_field(dims, inputs.sine_modes(dims, seed=seed + b))
                           + rng.uniform(-0.5, 0.5, n) for b in range(nb)]).astype(dtype)


def run(u0, nb, dims, lam, steps):
    tu = torch.from_numpy(u0.copy()).cuda()
    trid.adi_step_batched(tu, nb, dims, lam, steps)
    return tu.cpu().numpy()


def check(got, u0, nb, dims, lam, steps, dtype, meshes=None):
    n = int(np.prod(dims))
    for b in range(nb) if meshes is None else meshes:
        ref = oracle.adi(u0[b * n:(b + 1) * n], dims, lam, steps)
        g = got[b * n:(b + 1) * n].astype(np.float64)
        assert np.max(np.abs(g - ref)) <= TOL[dtype] * np.max(np.abs(ref)), b


DIMS = [(3, 3), (3, 40), (40, 3), (4, 4), (5, 6), (16, 17), (31, 32), (32, 33), (33, 31), (34, 64),
        (63, 66), (65, 64), (95, 97), (96, 96), (98, 35), (128, 100), (20, 127), (129, 20)]


@pytest.mark.parametrize("dtype", [np.float32, np.float64], ids=["f32", "f64"])
@pytest.mark.parametrize("dims", DIMS, ids=["x".join(map(str, d)) for d in DIMS])
def test_extents(dims, dtype):
    u0 = batch(dims, 3, sum(dims), dtype)
    check(run(u0, 3, dims, 0.15, 7), u0, 3, dims, 0.15, 7, dtype)


@pytest.mark.parametrize("dims", [(160, 160), (159, 130), (160, 24), (12, 160), (161, 40)])
def test_largest(dims):
    u0 = batch(dims, 2, sum(dims), np.float32)
    check(run(u0, 2, dims, 0.1, 5), u0, 2, dims, 0.1, 5, np.float32)


@pytest.mark.parametrize("lam", [1e-3, 0.5, 20.0])
@pytest.mark.parametrize("dtype", [np.float32, np.float64], ids=["f32", "f64"])
def test_coupling(lam, dtype):
    u0 = batch((45, 70), 2, 3, dtype)
    check(run(u0, 2, (45, 70), lam, 4), u0, 2, (45, 70), lam, 4, dtype)


@pytest.mark.parametrize("dims,nb", [((6, 5), 11000), ((64, 64), 1900), ((128, 36), 1300)])
def test_more_meshes_than_blocks(dims, nb):
    one = batch(dims, 7, 1, np.float32)
    n = int(np.prod(dims))
    u0 = np.tile(one, nb // 7 + 1)[:nb * n]
    got = run(u0, nb, dims, 0.1, 3)
    check(got, u0, nb, dims, 0.1, 3, np.float32, meshes=range(7))
    assert np.array_equal(got.reshape(nb, n)[7:], got.reshape(nb, n)[np.arange(7, nb) % 7])


def test_values_outside_the_field_do_not_enter():
    dims, nb = (37, 50), 5000
    n = dims[0] * dims[1]
    u0 = np.tile(batch(dims, 1, 9, np.float32), nb)
    clean = run(u0, nb, dims, 0.2, 6)
    u0 = u0.reshape(nb, dims[1], dims[0]).copy()
    u0[:, [0, 0, -1, -1], [0, -1, 0, -1]] = np.nan    # corners: in no stencil
    u0[::3] = np.inf                                  # other meshes
    got = run(u0.reshape(-1), nb, dims, 0.2, 6).reshape(nb, dims[1], dims[0])
    keep = np.arange(nb) % 3 != 0
    want = clean.reshape(nb, dims[1], dims[0])[keep].copy()
    want[:, [0, 0, -1, -1], [0, -1, 0, -1]] = np.nan
    assert np.array_equal(got[keep], want, equal_nan=True)
