"""A context does its work on its own stream alone: creating one must not touch
the legacy default stream, which orders itself with every blocking stream of
the process and may not be used while one of them is being captured."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu

RELAXED = 2   # cudaStreamCaptureModeRelaxed


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nvdim", [1, 3])
def test_create_beside_a_capture(nvdim, precision):
    import torch
    assert torch.cuda.is_available()
    torch.cuda.current_stream().synchronize()
    from paper_1804_03901_gb300 import avl as A
    rt = ctypes.CDLL("libcudart.so.13")
    stream, graph = ctypes.c_void_p(), ctypes.c_void_p()
    prec = A.AVL_FP32 if precision == "fp32" else A.AVL_FP64
    dom = A.make_domain(nvdim, 16, 4.0, 0.05, precision=prec)
    species = [A.make_species(-1.0, 1.0, (8,) * nvdim, (-3.0,) * nvdim, (3.0,) * nvdim)]
    A.Simulation(dom, species).close()   # modules loaded
    assert rt.cudaStreamCreate(ctypes.byref(stream)) == 0
    assert rt.cudaStreamBeginCapture(stream, RELAXED) == 0
    try:
        sim = A.Simulation(dom, species)
    finally:
        ended = rt.cudaStreamEndCapture(stream, ctypes.byref(graph))
        rt.cudaStreamDestroy(stream)
    assert ended == 0
    sim.close()
