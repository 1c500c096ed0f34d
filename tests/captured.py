"""What a call enqueues, seen in a capture of it: the kernel launches' grids and
how they depend on one another (read through the driver; the graph is not run)."""
import ctypes

_HANDLES = 512


class _KernelParams(ctypes.Structure):
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3),
                ("smem", ctypes.c_uint), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


class Captured:
    """kernels: the grid size of every kernel node; functions: their kernels; depth: kernels on
    the longest chain."""

    def __init__(self, call):
        import torch
        cu = ctypes.CDLL("libcuda.so.1")

        def check(rc):
            assert rc == 0, f"CUDA driver error {rc}"

        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        check(cu.cuStreamBeginCapture_v2(ctypes.c_void_p(stream.cuda_stream), 2))  # relaxed
        graph = ctypes.c_void_p()
        try:
            call(stream)
        finally:
            rc = cu.cuStreamEndCapture(ctypes.c_void_p(stream.cuda_stream), ctypes.byref(graph))
        check(rc)
        nodes, n = (ctypes.c_void_p * _HANDLES)(), ctypes.c_size_t(_HANDLES)
        check(cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)))
        grids, self.functions = {}, []
        for i in range(n.value):
            kind = ctypes.c_int()
            check(cu.cuGraphNodeGetType(ctypes.c_void_p(nodes[i]), ctypes.byref(kind)))
            if kind.value == 0:
                kp = _KernelParams()
                check(cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(nodes[i]), ctypes.byref(kp)))
                grids[nodes[i]] = kp.grid[0]
                self.functions.append((kp.func, kp.kern))
        src, dst, data = (ctypes.c_void_p * _HANDLES)(), (ctypes.c_void_p * _HANDLES)(), (ctypes.c_uint64 * _HANDLES)()
        e = ctypes.c_size_t(_HANDLES)
        check(cu.cuGraphGetEdges_v2(graph, src, dst, data, ctypes.byref(e)))
        after = {}
        for i in range(e.value):
            after.setdefault(dst[i], []).append(src[i])
        length = {}

        def chain(node):
            if node not in length:
                length[node] = (node in grids) + max((chain(p) for p in after.get(node, [])), default=0)
            return length[node]

        self.kernels = list(grids.values())
        self.depth = max(chain(nodes[i]) for i in range(n.value))
        check(cu.cuGraphDestroy(graph))
