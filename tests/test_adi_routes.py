"""Which kernels step a mesh or a batch of meshes, read from a captured graph, at
the sizes where a faster schedule must not be passed over; and the step there
against the FP64 oracle.  GPU only."""
import numpy as np
import pytest

import oracle
from graphs import graph_text
from paper_2201_03950_gb300 import inputs, trid

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore:DEBUG")]

TOL = {np.float32: 1e-5, np.float64: 1e-12}


def step(u, dims, nb, lam, steps, ws):
    if nb is None:
        trid.adi_step(u, dims, lam, steps, ws)
    else:
        trid.adi_step_batched(u, nb, dims, lam, steps, workspace=ws)


def scratch(dims, nb, dtype):
    dc, nd = trid._dims(dims)
    need = (trid.adi_workspace_bytes(dims, dtype) if nb is None else
            int(trid.load().adi_batched_workspace_bytes(nb, dc, nd, trid._code(dtype))))
    return torch.empty(need, dtype=torch.uint8, device="cuda") if need else None


SINGLE, F4, F8 = None, np.float32, np.float64
CASES = [((24, 32, 192), SINGLE, 0.1, F4, "k_adi_xyw"), ((32, 32, 256), SINGLE, 0.1, F4, "k_adi_xyw"),
         ((16, 32, 176), SINGLE, 0.1, F4, "k_adi_xyw"), ((32, 32, 192), 1, 0.1, F4, "k_adi_xyw"),
         ((32, 32, 128), 20, 0.1, F4, "k_adi_xyw"), ((32, 32, 48), 60, 0.1, F4, "k_adi_xyw"),
         ((32, 32, 32), SINGLE, 0.1, F4, "k_adi_planes"), ((32, 32, 32), 72, 0.1, F4, "k_adi_planes"),
         ((16, 32, 160), SINGLE, 0.1, F4, "k_adi_planes"),
         ((32, 32, 128), SINGLE, 0.3, F4, "k_adi_planes"),      # not windowed: slow decay
         # extents that are no multiples of 16, stacked: windowed too
         ((40, 64, 64), 1, 0.1, F4, "k_adi_xyw"), ((120, 96, 96), 3, 0.1, F4, "k_adi_xyw"),
         ((104, 128, 16), 5, 0.1, F4, "k_adi_xyw"), ((40, 64, 64), 3, 0.3, F4, "k_adi_planes"),
         ((40, 32, 16), 3, 0.1, F4, "k_adi_planes"),
         # long rows, short columns: whole planes for few meshes only
         ((160, 8, 8), 8, 0.2, F4, "k_adi_planes"), ((160, 8, 8), 72, 0.2, F4, "k_adi_fused"),
         ((64, 8, 8), 150, 0.2, F4, "k_adi_fused"), ((64, 16, 16), 72, 0.2, F4, "k_adi_planes"),
         # 2D in double precision: not where most of the rows issued would be padding
         ((3, 3), 100, 0.2, F8, "k_adi_fused"), ((40, 3), 3000, 0.2, F8, "k_adi_fused"),
         ((20, 20), 1000, 0.2, F8, "k_adi_fused"), ((20, 20), 100, 0.2, F8, "k_adi_plane"),
         ((18, 18), 1000, 0.2, F8, "k_adi_plane"), ((3, 3), 100, 0.2, F4, "k_adi_plane")]


@pytest.mark.parametrize("dims,nb,lam,dtype,kernel", CASES,
                         ids=[f"{'x'.join(map(str, c[0]))}-{c[1]}-{c[2]}-{c[3].__name__}" for c in CASES])
def test_route(dims, nb, lam, dtype, kernel, tmp_path):
    n = int(np.prod(dims))
    rng = np.random.default_rng(n)
    u0 = np.concatenate([inputs.sine_field(dims, inputs.sine_modes(dims, seed=b))
                         + rng.uniform(-0.5, 0.5, n) for b in range(nb or 1)]).astype(dtype)
    u = torch.from_numpy(u0).cuda()
    ws = scratch(dims, nb, u.dtype)
    # (the route of FP64 meshes on chip depends on there being 8 steps)
    steps = 8 if len(dims) == 2 else 2
    v = u.clone()
    assert kernel in graph_text(lambda: step(v, dims, nb, lam, steps, ws), tmp_path / "graph.dot")
    step(u, dims, nb, lam, 2, ws)
    got = u.cpu().numpy()
    for b in {0, (nb or 1) - 1}:
        ref = oracle.adi(u0[b * n:(b + 1) * n], dims, lam, 2)
        assert np.max(np.abs(got[b * n:(b + 1) * n] - ref)) <= TOL[dtype] * np.max(np.abs(ref))
