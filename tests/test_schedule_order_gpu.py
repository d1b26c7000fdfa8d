"""Order of the kernels that a call of up to 4096 prompt tokens puts on three streams, read from the recorded graph (nothing is
launched): the predictor of an auxiliary layer runs beside the layer's attention and FFN and reads buffers that the next layer's
projection overwrites; the base step's layers run beside the auxiliary layers after them and read what the predictor wrote."""
import ctypes as C
import re

import pytest

import workloads as wl
from parity_util import make_session

pytestmark = pytest.mark.gpu

# kernels that write an auxiliary layer's keys and values, and predictor kernels, which read them: on the tensor cores, or not
PROJECTION = re.compile(r"gemm_tc_kernelILi3E|rope_split_kernel")
PREDICTOR = re.compile(r"gemm_tc_kernelILi4E|gemm_simt_kernelI\w+?Li2ELi")


def _ok(r):
    assert int(r[0]) == 0, r[0]
    return r[1] if len(r) == 2 else r[1:]


class Recorded:
    """The graph of one kvp_prefill_predict call: kernel names by node, and every node's edges from nodes before it."""

    def __init__(self, s, tokens, lens):
        import torch
        from cuda.bindings import driver as cu
        from cuda.bindings import runtime as rt
        torch.cuda.synchronize()
        st = rt.cudaStream_t(s.stream)
        _ok(rt.cudaStreamBeginCapture(st, rt.cudaStreamCaptureMode.cudaStreamCaptureModeThreadLocal) + (None,))
        try:
            import paper_2410_08391_b200 as kvp
            kvp.kvp_prefill_predict(s.h, tokens, lens, s.cache, s.workspace, s.logits, s.first, s.stream)
        finally:
            graph = cu.CUgraph(int(_ok(rt.cudaStreamEndCapture(st))))
        try:
            nodes, n = _ok(cu.cuGraphGetNodes(graph, 1 << 14))
            nodes = nodes[:n]
            self.name, self.edges = {}, {int(x): [] for x in nodes}
            for x in nodes:
                if int(_ok(cu.cuGraphNodeGetType(x))) == int(cu.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL):
                    self.name[int(x)] = _ok(cu.cuFuncGetName(_ok(cu.cuGraphKernelNodeGetParams(x)).func)).decode()
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
        return [x for x, n in self.name.items() if pattern.search(n)]


def _recorded(pair, lens):
    import torch
    pr = wl.custom_prompts(pair.base.vocab, lens, seed=2)
    s = make_session(pair, wl.make_weights(pair, seed=2), pr)
    try:
        return Recorded(s, torch.from_numpy(pr.tokens).to(s.device), lens)
    finally:
        s.close()


def _narrow():
    """bf16, heads too narrow for the tensor-core kernels"""
    return wl.PairCfg("narrow", wl.uniform_model(4, 64, 2, 1, 32, 96, 97), wl.uniform_model(4, 64, 2, 1, 32, 96, 97), (0, 1, 2, 3))


@pytest.mark.parametrize("name,lens", [("t_small", [70, 63]), ("t_small", [9] * 6), ("t_small", [4096]), ("t_small_gap", [40, 9]),
                                       ("t_small_f32", [70]), ("t_hd128_qkn", [130]), ("narrow", [30, 7])], ids=str)
def test_predictor_is_ordered_against_every_projection(name, lens):
    pair = _narrow() if name == "narrow" else wl.pair(name)
    g = _recorded(pair, lens)
    projections, predictors = g.find(PROJECTION), g.find(PREDICTOR)
    assert len(projections) == max(pair.layer_map) + 1
    assert len(predictors) == 2 * len(set(pair.layer_map))
    for r in predictors:
        for w in projections:
            assert r in g.before(w) or w in g.before(r), "a projection may overwrite keys and values that a predictor kernel still reads"


@pytest.mark.parametrize("name,lens", [("t_small", [9] * 6), ("t_small_gap", [40, 9, 130, 17, 64, 65]), ("t_hd128_qkn", [70] * 9), ("t_small", [600] * 6)], ids=str)
def test_pages_are_complete_when_the_steps_attention_starts(name, lens):
    """It asks for cache pages (and reads lengths) before it waits for the kernel in front of it."""
    pair = wl.pair(name)
    g = _recorded(pair, lens)
    attention, predictors, lengths = g.find(re.compile("step_attn_mma_kernel")), g.find(PREDICTOR), g.find(re.compile("build_index_kernel"))
    assert len(attention) == pair.base.n_layers and len(predictors) == 2 * len(set(pair.layer_map)) and len(lengths) == 1
    first = min(len(set(predictors) & g.before(x)) for x in attention)
    assert first == 2      # its first layers do run beside the auxiliary layers
    for x in attention:
        assert set(lengths + predictors) & g.before(x) <= g.complete(x), "a page may be read while a predictor kernel writes it"


@pytest.mark.parametrize("name,lens", [("t_small_f32", [70, 63]), ("t_small_f32", [9] * 6), ("narrow", [30, 7])], ids=str)
def test_kernels_of_the_cuda_core_path_are_ordinary_launches(name, lens):
    """Recorded as dependent launches they made first calls and, while they waited, other kernels slower."""
    g = _recorded(_narrow() if name == "narrow" else wl.pair(name), lens)
    nodes = g.find(re.compile("gemm_simt_kernel|attn_prefill_simt_kernel|rope_split_kernel|swiglu_kernel"))
    assert len(nodes) >= 7
    assert not any(early for x in nodes for _, early in g.edges[x])
