"""The library kernels a call launches, by name and in order: the call is
recorded on a capturing stream, nothing runs, and the driver names the nodes of
the graph.  For tests of which kernel a launch is routed to, where every route
gives the same result."""
import ctypes
import re

KERNEL_NODE = 0


def _check(code, what):
    assert code == 0, f"{what}: CUDA error {code}"


def kernels_of(call):
    """Names of the kernels that ``call(stream)`` enqueues on the torch stream
    it is given."""
    import torch
    cu = ctypes.CDLL("libcuda.so.1")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    handle, graph = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    _check(cu.cuStreamBeginCapture_v2(handle, 2), "begin capture")  # relaxed
    try:
        call(stream)
    finally:
        end = cu.cuStreamEndCapture(handle, ctypes.byref(graph))
    _check(end, "end capture")
    try:
        n = ctypes.c_size_t()
        _check(cu.cuGraphGetNodes(graph, None, ctypes.byref(n)), "nodes")
        nodes = (ctypes.c_void_p * max(n.value, 1))()
        _check(cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)), "nodes")
        out = []
        for k in range(n.value):
            kind = ctypes.c_int()
            node = ctypes.c_void_p(nodes[k])
            _check(cu.cuGraphNodeGetType(node, ctypes.byref(kind)), "node type")
            if kind.value == KERNEL_NODE:
                out.append(_name(cu, node))
        return out
    finally:
        cu.cuGraphDestroy(graph)


def _name(cu, node):
    # CUDA_KERNEL_NODE_PARAMS_v2: func, 7 x uint32 (grid, block, shared bytes),
    # kernelParams, extra, kern, ctx
    words = (ctypes.c_uint64 * 16)()
    _check(cu.cuGraphKernelNodeGetParams_v2(node, words), "kernel node")
    text = ctypes.c_char_p()
    if words[0]:
        _check(cu.cuFuncGetName(ctypes.byref(text), ctypes.c_void_p(words[0])), "function name")
    else:
        _check(cu.cuKernelGetName(ctypes.byref(text), ctypes.c_void_p(words[7])), "kernel name")
    mangled = text.value.decode()
    # the name in lower case, up to the template's or the signature's letter
    m = re.search(r"\dk_[a-z0-9_]+", mangled)
    return m.group(0)[1:] if m else mangled
