"""What no path may take is refused before anything is launched: more tiles than
the passes can count, whether or not scratch is given.  GPU only (it holds two
arrays of 67 GB and 52 GB of scratch, and reads none of them)."""
import pytest

from paper_2201_03950_gb300 import trid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_tiles_beyond_32_bits():
    n, nsys = 257, (1 << 31) // 33 + 1       # 33 tiles of 8 rows, no whole vectors
    dims = (n, nsys)
    need = trid.solve_workspace_bytes(dims, 0, torch.float32)
    free, _ = torch.cuda.mem_get_info()
    if free < need + 8 * n * nsys + (1 << 30):
        pytest.skip("not enough free memory")
    co, d = (torch.empty(n * nsys, device="cuda") for _ in range(2))
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    try:
        for workspace in (ws, ws[:256]):
            with pytest.raises(trid.TridError) as e:
                trid.solve(co, co, co, d, dims, 0, workspace=workspace)
            assert e.value.status == (2 if workspace is ws else 5)   # UNSUPPORTED, ALLOC
    finally:
        del co, d, ws
        torch.cuda.empty_cache()
