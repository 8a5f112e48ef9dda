"""Launch shapes of the library's kernels, read from a captured graph (nothing is executed)."""
import ctypes


def launches(stream, call):
    """[(grid, block)] of the kernels that call() launches on `stream` (a torch stream)."""
    cu = ctypes.CDLL("libcuda.so.1")
    s, graph, count = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    assert cu.cuStreamBeginCapture_v2(s, 1) == 0  # CU_STREAM_CAPTURE_MODE_THREAD_LOCAL
    call()
    assert cu.cuStreamEndCapture(s, ctypes.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(count)) == 0
    nodes = (ctypes.c_void_p * count.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(count)) == 0
    out = []
    for n in nodes:
        p = (ctypes.c_uint32 * 64)()  # CUDA_KERNEL_NODE_PARAMS: function, gridDimX, .. Z, blockDimX, .. Z
        assert cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(n), p) == 0
        out.append((tuple(p[2:5]), tuple(p[5:8])))
    assert cu.cuGraphDestroy(graph) == 0
    return out
