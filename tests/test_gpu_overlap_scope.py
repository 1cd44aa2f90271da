"""Which launches overlap, read from the edges of a captured graph: those of a
clustering call of up to 2^21 points, and none of a component entry point,
whatever the thread called before."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2103_05162_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu

PROGRAMMATIC = 1  # cudaGraphDependencyTypeProgrammatic


class EdgeData(ctypes.Structure):
    _fields_ = [("from_port", ctypes.c_ubyte), ("to_port", ctypes.c_ubyte), ("type", ctypes.c_ubyte),
                ("reserved", ctypes.c_ubyte * 5)]


def edge_types(fn):
    """The types of the edges of the graph that fn's launches make."""
    rt = ctypes.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")
    s = torch.cuda.Stream()
    vp = ctypes.c_void_p
    with torch.cuda.stream(s):
        fn()  # workspaces and tuning before the capture
        s.synchronize()
        graph, n = vp(), ctypes.c_size_t()
        assert rt.cudaStreamBeginCapture(vp(s.cuda_stream), 2) == 0  # relaxed: the outputs' allocations may go on
        try:
            fn()
        finally:
            assert rt.cudaStreamEndCapture(vp(s.cuda_stream), ctypes.byref(graph)) == 0
    get = rt.cudaGraphGetEdges if torch.version.cuda.startswith("13") else rt.cudaGraphGetEdges_v2
    assert get(graph, None, None, None, ctypes.byref(n)) == 0
    a, b, data = (vp * n.value)(), (vp * n.value)(), (EdgeData * n.value)()
    assert get(graph, a, b, data, ctypes.byref(n)) == 0
    assert rt.cudaGraphDestroy(graph) == 0
    return [d.type for d in data]


def test_only_clustering_calls_overlap():
    pts = torch.rand(3000, 3, device="cuda")
    big = torch.rand((1 << 21) + 1, 3, device="cuda")
    lo, hi = np.zeros(3, np.float32), np.ones(3, np.float32)

    def codes():
        gb.morton_codes(pts, lo, hi, 16)
        gb.morton_codes(pts, lo, hi, 16)

    try:
        gb.set_tuning(128, 1.0)
        assert edge_types(codes) == [0]
        assert PROGRAMMATIC in edge_types(lambda: gb.dbscan_run(pts, 0.01, 5))
        assert edge_types(codes) == [0]
        assert PROGRAMMATIC not in edge_types(lambda: gb.dbscan_run(big, 0.002, 5))
    finally:
        gb.set_tuning(0, 0.0)
