"""3D ADI steps through the whole-plane kernels (k_adi_planes, k_adi_zlines)
against the FP64 oracle: extents around the sizes that select a kernel, odd and
even, the smallest and longest lines, batches stacked along z with all, some or
none of the scratch they ask for, unaligned arrays, poisoned scratch, values
that enter no stencil, and a captured graph.  GPU only."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2201_03950_gb300 import inputs, trid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {np.float32: 1e-5, np.float64: 1e-12}


def field(dims, nb, seed, dtype):
    rng = np.random.default_rng(seed)
    n = int(np.prod(dims))
    return np.concatenate([inputs.sine_field(dims, inputs.sine_modes(dims, seed=seed + b))
                           + rng.uniform(-0.5, 0.5, n) for b in range(nb)]).astype(dtype)


def check(got, u0, nb, dims, lam, steps, dtype):
    n = int(np.prod(dims))
    for b in range(nb):
        ref = oracle.adi(u0[b * n:(b + 1) * n], dims, lam, steps)
        g = got[b * n:(b + 1) * n].astype(np.float64)
        assert np.max(np.abs(g - ref)) <= TOL[dtype] * np.max(np.abs(ref)), b


def one(dims, lam, steps, dtype, offset=0):
    u0 = field(dims, 1, sum(dims), dtype)
    buf = torch.zeros(u0.size + offset, dtype=torch.float32 if dtype is np.float32
                      else torch.float64, device="cuda")[offset:]
    buf.copy_(torch.from_numpy(u0))
    ws = torch.full((trid.adi_workspace_bytes(dims, buf.dtype) // buf.element_size(),),
                    float("nan"), dtype=buf.dtype, device="cuda")   # scratch holds no numbers
    trid.adi_step(buf, dims, lam, steps, ws)
    check(buf.cpu().numpy(), u0, 1, dims, lam, steps, dtype)


DIMS = [(3, 3, 3), (4, 3, 5), (3, 20, 7), (33, 31, 32), (47, 50, 17), (48, 49, 34), (65, 63, 20),
        (80, 82, 9), (95, 40, 64), (97, 30, 65), (126, 128, 6), (129, 34, 8), (160, 20, 5),
        (20, 160, 5), (159, 100, 4), (17, 18, 129), (60, 60, 161), (50, 50, 256), (64, 48, 225),
        (161, 20, 6), (140, 150, 5)]


@pytest.mark.parametrize("dtype", [np.float32, np.float64], ids=["f32", "f64"])
@pytest.mark.parametrize("dims", DIMS, ids=["x".join(map(str, d)) for d in DIMS])
def test_extents(dims, dtype):
    one(dims, 0.25, 3, dtype)


@pytest.mark.parametrize("lam", [1e-3, 0.1, 1.0, 30.0])
@pytest.mark.parametrize("dtype", [np.float32, np.float64], ids=["f32", "f64"])
def test_coupling(lam, dtype):
    one((44, 37, 29), lam, 4, dtype)


def test_unaligned_field():
    one((40, 36, 20), 0.2, 3, np.float32, offset=1)
    one((41, 20, 22), 0.2, 3, np.float64, offset=1)


def stepped(u0, nb, dims, lam, steps, ws_bytes=None, shift=0):
    """adi_step_batched through the C entry point with scratch of a given size."""
    tu = torch.from_numpy(u0.copy()).cuda()
    dc, nd = trid._dims(dims)
    need = int(trid.load().adi_batched_workspace_bytes(nb, dc, nd, trid._dtype(tu)))
    size = need if ws_bytes is None else ws_bytes
    ws = torch.full((max(size + shift, 1),), 255, dtype=torch.uint8, device="cuda")  # NaN
    st = trid.load().adi_step_batched(
        trid._ptr(tu), nb, dc, nd, lam, steps, trid._dtype(tu),
        ctypes.c_void_p(ws.data_ptr() + shift) if size else None, size, trid._stream(None))
    torch.cuda.synchronize()
    return st, tu.cpu().numpy(), need


@pytest.mark.parametrize("dtype", [np.float32, np.float64], ids=["f32", "f64"])
@pytest.mark.parametrize("dims,nb", [((30, 21, 25), 7), ((48, 48, 48), 3), ((24, 24, 24), 5),
                                     ((40, 51, 16), 4), ((24, 32, 48), 3), ((32, 32, 32), 4)])
def test_batches(dims, nb, dtype):
    u0 = field(dims, nb, 11, dtype)
    st, got, _ = stepped(u0, nb, dims, 0.2, 3)
    assert st == 0
    check(got, u0, nb, dims, 0.2, 3, dtype)


@pytest.mark.parametrize("dims,nb,dtype", [((30, 31, 25), 7, np.float32), ((25, 28, 24), 5, np.float32),
                                           ((40, 33, 50), 4, np.float64)])
def test_less_scratch_than_asked_for(dims, nb, dtype):
    u0 = field(dims, nb, 4, dtype)
    mesh = int(np.prod(dims)) * np.dtype(dtype).itemsize
    full = stepped(u0, nb, dims, 0.3, 3)
    assert full[0] == 0 and full[2] >= nb * mesh
    dc, nd = trid._dims(dims)
    single = trid.adi_workspace_bytes(dims, "float32" if dtype is np.float32 else "float64")
    for size in (2 * mesh + 100, single):
        st, got, _ = stepped(u0, nb, dims, 0.3, 3, ws_bytes=size)
        assert st == 0
        assert np.array_equal(got, full[1])


def test_resident_meshes_need_no_scratch():
    dims, nb = (20, 18, 22), 4
    u0 = field(dims, nb, 6, np.float32)
    for size, shift in ((0, 0), (4096, 0), (1 << 20, 64)):   # none, too little, misaligned
        st, got, _ = stepped(u0, nb, dims, 0.2, 3, ws_bytes=size, shift=shift)
        assert st == 0
        check(got, u0, nb, dims, 0.2, 3, np.float32)


def test_too_little_scratch_is_refused():
    st, got, _ = stepped(field((50, 51, 40), 2, 6, np.float32), 2, (50, 51, 40), 0.2, 3, ws_bytes=512)
    assert st == 5   # TRID_ERR_ALLOC


def test_scratch_asked_for_is_bounded():
    dc, nd = trid._dims((100, 100, 100))
    one = trid.adi_workspace_bytes((100, 100, 100), "float32")
    for nb in (1, 60, 500, 600, 1000, 1 << 20):
        need = int(trid.load().adi_batched_workspace_bytes(nb, dc, nd, trid.TRID_F32))
        assert one <= need <= 2 << 30


@pytest.mark.parametrize("dims,dtype", [((30, 31, 170), np.float32), ((33, 29, 20), np.float64),
                                        ((25, 28, 24), np.float32)])
def test_place_and_scratch_do_not_change_the_bits(dims, dtype):
    """Five times the same mesh, with scratch for one to five of them."""
    nb = 5
    u0 = np.tile(field(dims, 1, 5, dtype), nb)
    mesh = int(np.prod(dims)) * np.dtype(dtype).itemsize
    least = trid.adi_workspace_bytes(dims, "float32" if dtype is np.float32 else "float64")
    first = None
    for size in (None, least, 2 * mesh, 3 * mesh, 4 * mesh):
        if size is not None and size < least:
            continue
        st, got, _ = stepped(u0, nb, dims, 0.25, 3, ws_bytes=size)
        assert st == 0
        first = got[:got.size // nb] if first is None else first
        assert np.array_equal(got, np.tile(first, nb))


def test_less_than_one_meshs_scratch_is_refused():
    dims = (50, 51, 40)     # too large to be resident on chip
    u0 = field(dims, 2, 5, np.float32)
    least = trid.adi_workspace_bytes(dims, "float32")
    for size in (u0.nbytes // 2, least - 256):
        st, got, _ = stepped(u0, 2, dims, 0.25, 3, ws_bytes=size)
        assert st == 5 and np.array_equal(got, u0)   # TRID_ERR_ALLOC


def test_box_edges_do_not_enter():
    dims = (34, 29, 31)
    u0 = field(dims, 1, 8, np.float32).reshape(dims[::-1])
    edge = np.zeros(u0.shape, dtype=int)
    for ax in range(3):
        edge[tuple(slice(None) if a != ax else [0, -1] for a in range(3))] += 1
    poisoned = u0.copy()
    poisoned[edge >= 2] = np.nan          # the box's edges: in no stencil
    out = []
    for v in (u0, poisoned):
        tu = torch.from_numpy(v.reshape(-1).copy()).cuda()
        ws = torch.empty(trid.adi_workspace_bytes(dims, tu.dtype), dtype=torch.uint8, device="cuda")
        trid.adi_step(tu, dims, 0.2, 4, ws)
        out.append(tu.cpu().numpy().reshape(u0.shape))
    out[0][edge >= 2] = np.nan
    assert np.array_equal(out[0], out[1], equal_nan=True)


def test_captured():
    dims = (52, 45, 40)
    u0 = field(dims, 1, 3, np.float32)
    tu = torch.from_numpy(u0).cuda()
    ws = torch.empty(trid.adi_workspace_bytes(dims, tu.dtype), dtype=torch.uint8, device="cuda")
    trid.adi_step(tu, dims, 0.3, 2, ws)
    direct = tu.clone()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        trid.adi_step(tu, dims, 0.3, 2, ws)
    tu.copy_(torch.from_numpy(u0))
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(tu, direct)
