"""The kernel launches that a call enqueues, read back from a stream capture."""
import ctypes


class _KernelParams(ctypes.Structure):  # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", ctypes.c_void_p)] + [(f"{k}{a}", ctypes.c_uint) for k in ("grid", "block") for a in "xyz"] + [
        ("shared", ctypes.c_uint), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
        ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


CARVEOUT = 14  # CU_LAUNCH_ATTRIBUTE_PREFERRED_SHARED_MEMORY_CARVEOUT


def captured_kernels(stream, enqueue, attribute=None):
    """[(CTAs, threads of a CTA)] of the kernels that enqueue() launches on `stream` (an
    address; not the default stream), in the order of the graph's nodes; with an
    attribute (of integer value) its values instead.  Nothing runs."""
    cu = ctypes.CDLL("libcuda.so.1")

    def check(status):
        assert status == 0, f"CUresult {status}"

    st, graph, n = ctypes.c_void_p(stream), ctypes.c_void_p(), ctypes.c_size_t()
    check(cu.cuStreamBeginCapture_v2(st, 2))  # relaxed
    try:
        enqueue()
    finally:
        check(cu.cuStreamEndCapture(st, ctypes.byref(graph)))
    check(cu.cuGraphGetNodes(graph, None, ctypes.byref(n)))
    nodes = (ctypes.c_void_p * n.value)()
    check(cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)))
    out = []
    for node in nodes:
        kind = ctypes.c_int()
        check(cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)))
        if kind.value != 0:  # CU_GRAPH_NODE_TYPE_KERNEL
            continue
        if attribute is not None:
            value = (ctypes.c_int * 16)()  # CUlaunchAttributeValue
            check(cu.cuGraphKernelNodeGetAttribute(ctypes.c_void_p(node), attribute, ctypes.byref(value)))
            out.append(value[0])
            continue
        p = _KernelParams()
        check(cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(p)))
        out.append((p.gridx * p.gridy * p.gridz, p.blockx * p.blocky * p.blockz))
    check(cu.cuGraphDestroy(graph))
    return out
