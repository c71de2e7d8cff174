"""Stream capture through the driver, for what PyTorch's CUDAGraph does not offer: captures that are
meant to fail, and the attributes of the captured kernels. Handles are those of the runtime."""
import ctypes as C

THREAD_LOCAL = 1            # CU_STREAM_CAPTURE_MODE_THREAD_LOCAL
_KERNEL_NODE, _PRIORITY = 0, 8   # CU_GRAPH_NODE_TYPE_KERNEL, CU_LAUNCH_ATTRIBUTE_PRIORITY


def _driver():
    return C.CDLL("libcuda.so.1")


def begin(stream: int):
    assert _driver().cuStreamBeginCapture_v2(C.c_void_p(stream), THREAD_LOCAL) == 0


def end(stream: int):
    """the captured graph, None if the capture was spoilt"""
    graph = C.c_void_p()
    status = _driver().cuStreamEndCapture(C.c_void_p(stream), C.byref(graph))
    return graph if status == 0 else None


def destroy(graph):
    assert _driver().cuGraphDestroy(graph) == 0


def kernel_priorities(graph):
    """launch priority of every kernel of the graph"""
    lib, n = _driver(), C.c_size_t(0)
    assert lib.cuGraphGetNodes(graph, None, C.byref(n)) == 0
    nodes = (C.c_void_p * n.value)()
    assert lib.cuGraphGetNodes(graph, nodes, C.byref(n)) == 0
    out = []
    for node in nodes:
        kind = C.c_int()
        assert lib.cuGraphNodeGetType(C.c_void_p(node), C.byref(kind)) == 0
        if kind.value == _KERNEL_NODE:
            value = (C.c_char * 64)()          # CUlaunchAttributeValue
            assert lib.cuGraphKernelNodeGetAttribute(C.c_void_p(node), _PRIORITY, value) == 0
            out.append(C.c_int.from_buffer(value).value)
    return out
