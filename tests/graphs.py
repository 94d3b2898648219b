"""The kernels of a call, read from a captured graph."""
import torch


def graph_text(call, path):
    """``call()`` once (the library's per-device set-up is not capturable), then
    captured; the graph as text, in which the kernels appear by name."""
    call()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    g.enable_debug_mode()
    with torch.cuda.graph(g):
        call()
    g.debug_dump(str(path))
    return path.read_text()
