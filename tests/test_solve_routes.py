"""Which kernel solves a mesh's systems, read from a captured graph, at the sizes
where a slower one must not be chosen; and the solution there against the FP64
oracle.  GPU only."""
import numpy as np
import pytest

import oracle
from graphs import graph_text
from paper_2201_03950_gb300 import inputs, trid

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore:DEBUG")]

TOL = {np.float32: 1e-5, np.float64: 1e-12}


def check(dims, k, dtype, acc, kernel, path, offset=0):
    n = int(np.prod(dims))
    host = inputs.dominant_system((n,), seed=n, dtype=dtype)
    dev = [torch.empty(n + offset, dtype=torch.from_numpy(v).dtype, device="cuda")[offset:]
           .copy_(torch.from_numpy(v)) for v in host]
    u = torch.zeros_like(dev[3]) if acc else None
    x = dev[3].clone()
    got = trid.solve(*dev[:3], x, dims, k, u=u).cpu().numpy()
    ref = oracle.solve_mesh(*host, dims, k)
    assert np.max(np.abs(got - ref)) <= TOL[dtype] * np.max(np.abs(ref))
    text = graph_text(lambda: trid.solve(*dev[:3], x, dims, k, u=u), path / "graph.dot")
    assert kernel in text
    return text


@pytest.mark.parametrize("n", [64, 128, 256])
@pytest.mark.parametrize("acc", [False, True], ids=["store", "acc"])
def test_fp64_short_strided(n, acc, tmp_path):
    """Two threads per system from the second round of the tiled kernel on."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    check((32 * sms, n), 1, np.float64, acc, "k_strided", tmp_path)
    check((32 * sms + 4, n), 1, np.float64, acc, "k_twist", tmp_path)


@pytest.mark.parametrize("n", [8, 192])
def test_fp64_short_strided_early(n, tmp_path):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    check((30 * sms, n), 1, np.float64, False, "k_strided", tmp_path)
    check((30 * sms + 4, n), 1, np.float64, False, "k_twist", tmp_path)


@pytest.mark.parametrize("acc", [False, True], ids=["store", "acc"])
def test_fp32_contiguous_257_to_512(acc, tmp_path):
    check((400, 1000), 0, np.float32, acc, "k_lines_chained", tmp_path)


@pytest.mark.parametrize("dims,k", [((260, 1), 0), ((400, 64), 0), ((512, 1000), 0), ((64, 64, 64), 1),
                                    ((64, 64, 64), 2), ((128, 128, 128), 1), ((1000, 256, 25), 1),
                                    ((304, 200, 90), 1)], ids=str)
def test_chained_calls_see_each_other(dims, k):
    """Ten calls in a row, each on what the one before has written, as with a
    synchronisation in between."""
    n = int(np.prod(dims))
    t = [torch.from_numpy(v).cuda() for v in inputs.dominant_system((n,), seed=n, dtype=np.float32)]
    out = []
    for wait in (False, True):
        x, b, u = t[3].clone(), t[1].clone(), torch.zeros_like(t[3])
        for _ in range(10):
            trid.solve(t[0], b, t[2], x, dims, k)
            if wait:
                torch.cuda.synchronize()
            trid.solve(t[0], b, t[2], x, dims, k, u=u)
            if wait:
                torch.cuda.synchronize()
            torch.add(t[1], u.abs(), out=b)     # the next call's coefficients
        out.append((x, u))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


@pytest.mark.parametrize("n,dtype,acc,offset,kernel", [
    (3, np.float32, False, 0, "k_lines"), (13, np.float32, False, 0, "k_lines"),
    (8, np.float32, False, 1, "k_lines_staged"), (16, np.float32, False, 1, "k_lines_staged"),
    (3, np.float32, True, 0, "k_lines_staged"), (3, np.float64, False, 0, "k_lines_staged"),
    (201, np.float32, False, 0, "k_lines_staged")])
def test_contiguous_no_whole_vectors(n, dtype, acc, offset, kernel, tmp_path):
    text = check((n, 5000), 0, dtype, acc, kernel, tmp_path, offset)
    assert ("staged" in kernel) == ("staged" in text)
