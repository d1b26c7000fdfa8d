"""What a call of the library would launch, read from a recorded CUDA graph (nothing runs): which kernels, with what grids, in what
order."""
import ctypes as C
import re

import workloads as wl
from parity_util import make_session


def _ok(r):
    assert int(r[0]) == 0, r[0]
    return r[1] if len(r) == 2 else r[1:]


class Recorded:
    """The graph that `call` puts on a session's stream, without a launch: name and grid of the kernels by node, and every node's
    edges from nodes before it."""

    def __init__(self, s, call):
        import torch
        from cuda.bindings import driver as cu
        from cuda.bindings import runtime as rt
        torch.cuda.synchronize()
        st = rt.cudaStream_t(s.stream)
        _ok(rt.cudaStreamBeginCapture(st, rt.cudaStreamCaptureMode.cudaStreamCaptureModeThreadLocal) + (None,))
        try:
            call()
        finally:
            graph = cu.CUgraph(int(_ok(rt.cudaStreamEndCapture(st))))
        try:
            nodes, n = _ok(cu.cuGraphGetNodes(graph, 1 << 14))
            nodes = nodes[:n]
            self.name, self.grid, self.edges = {}, {}, {int(x): [] for x in nodes}
            for x in nodes:
                if int(_ok(cu.cuGraphNodeGetType(x))) == int(cu.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL):
                    k = _ok(cu.cuGraphKernelNodeGetParams(x))
                    self.name[int(x)], self.grid[int(x)] = _ok(cu.cuFuncGetName(k.func)).decode(), (k.gridDimX, k.gridDimY, k.gridDimZ)
            # (through ctypes: edge data are from port, to port, type, five bytes reserved)
            n, most = C.c_size_t(1 << 16), 1 << 16
            a, b, data = (C.c_void_p * most)(), (C.c_void_p * most)(), ((C.c_ubyte * 8) * most)()
            assert C.CDLL("libcuda.so.1").cuGraphGetEdges_v2(C.c_void_p(int(graph)), a, b, data, C.byref(n)) == 0
            for i in range(n.value):
                self.edges[b[i]].append((a[i], data[i][2] != 0))      # (node, whether it may still be running)
        finally:
            cu.cuGraphDestroy(graph)
        self._before, self._complete = {}, {}

    def before(self, x):
        """Every node on a path to x."""
        if x not in self._before:
            self._before[x] = set().union(*({y} | self.before(y) for y, _ in self.edges[x]))
        return self._before[x]

    def complete(self, x):
        """The nodes that have finished when x starts.  One whose launch does not wait for the end of the node before it starts
        no earlier than that one; no kernel ends before those in front of it have."""
        if x not in self._complete:
            self._complete[x] = set().union(*(self.complete(y) if early else {y} | self.before(y) for y, early in self.edges[x]))
        return self._complete[x]

    def find(self, pattern):
        return [x for x, n in self.name.items() if re.search(pattern, n)]

    def grids(self, pattern):
        return [self.grid[x] for x in self.find(pattern)]


def recorded_prefill(pair, lens, W=None, **session):
    """The graph of kvp_prefill_predict for prompts of these lengths."""
    import torch

    import paper_2410_08391_b200 as kvp
    pr = wl.custom_prompts(pair.base.vocab, lens, seed=2)
    s = make_session(pair, W or wl.make_weights(pair, seed=2), pr, **session)
    try:
        tokens = torch.from_numpy(pr.tokens).to(s.device)
        return Recorded(s, lambda: kvp.kvp_prefill_predict(s.h, tokens, lens, s.cache, s.workspace, s.logits, s.first, s.stream))
    finally:
        s.close()
