"""Which of the library's kernels a call launches: tests that are about one form of a kernel make sure that it is the one that ran."""
import collections
import ctypes as C
import re

import torch

Launch = collections.namedtuple("Launch", "kernel blocks shared")  # name with template arguments; blocks; dynamic shared memory of each


class _KernelNode(C.Structure):  # CUDA_KERNEL_NODE_PARAMS
    _fields_ = [("func", C.c_void_p), ("grid", C.c_uint * 3), ("block", C.c_uint * 3), ("shared", C.c_uint),
                ("params", C.c_void_p), ("extra", C.c_void_p), ("kern", C.c_void_p), ("ctx", C.c_void_p)]


def _name(mangled):
    """'cowa_x_kernel<64,true,2>' of the mangled name of an instance; None for other kernels."""
    m = re.search(r"\d(cowa_\w+?_kernel)(?:I((?:L[ib]\d+E)+)E)?", mangled)
    if not m:
        return None
    args = [v if t == "i" else "true" if v == "1" else "false" for t, v in re.findall(r"L([ib])(\d+)E", m.group(2) or "")]
    return m.group(1) + (f"<{','.join(args)}>" if args else "")


def launched(call):
    """The kernels of this library that call() launches, in their order.  Runs it, and once more into a graph, whose nodes tell."""
    call()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    driver = C.CDLL("libcuda.so.1")

    def check(status):
        assert status == 0, f"CUDA driver error {status}"

    handle, n = C.c_void_p(graph.raw_cuda_graph()), C.c_size_t(0)
    check(driver.cuGraphGetNodes(handle, None, C.byref(n)))
    nodes = (C.c_void_p * n.value)()
    check(driver.cuGraphGetNodes(handle, nodes, C.byref(n)))
    out = []
    for node in nodes:
        kind, p, name = C.c_int(-1), _KernelNode(), C.c_char_p()
        check(driver.cuGraphNodeGetType(C.c_void_p(node), C.byref(kind)))
        if kind.value != 0:  # a kernel
            continue
        check(driver.cuGraphKernelNodeGetParams_v2(C.c_void_p(node), C.byref(p)))
        if p.func:
            check(driver.cuFuncGetName(C.byref(name), C.c_void_p(p.func)))
        else:
            check(driver.cuKernelGetName(C.byref(name), C.c_void_p(p.kern)))
        kernel = _name(name.value.decode())
        if kernel:
            out.append(Launch(kernel, p.grid[0] * p.grid[1] * p.grid[2], p.shared))
    return out
