"""The kernels that a call queues, by their (mangled) names: the kernel nodes of its captured
graph, as the driver prints them."""
import ctypes
import re


def kernel_names(call, path, pattern):
    """Names of the kernels of `call` that contain a match of `pattern`, in the driver's order."""
    import torch
    call()                                       # first-use work happens outside the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    driver = ctypes.CDLL("libcuda.so.1")
    assert driver.cuGraphDebugDotPrint(ctypes.c_void_p(graph.raw_cuda_graph()),
                                       str(path).encode(), ctypes.c_uint(0)) == 0
    return re.findall(rf"\w*(?:{pattern})\w*", open(path).read())
