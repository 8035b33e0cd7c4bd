"""Which kernels a call launches (the nodes of a graph captured from it), so that
a test of two routes to the same bits knows that both were taken."""
import ctypes
import os
import tempfile


def kernels_of(call):
    """Run call(stream) once, then capture it: text that names its kernels."""
    import torch
    call(torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call(torch.cuda.current_stream().cuda_stream)
    with tempfile.TemporaryDirectory() as d:
        path = os.path.join(d, "graph.dot")
        rc = ctypes.CDLL("libcuda.so.1").cuGraphDebugDotPrint(ctypes.c_void_p(graph.raw_cuda_graph()), path.encode(), 1)
        assert rc == 0
        with open(path) as f:
            return f.read()
