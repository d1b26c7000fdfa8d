"""Order of the kernels that a call of up to 4096 prompt tokens puts on three streams, read from the recorded graph (nothing is
launched): the predictor of an auxiliary layer runs beside the layer's attention and FFN and reads buffers that the next layer's
projection overwrites; the base step's layers run beside the auxiliary layers after them and read what the predictor wrote."""
import re

import pytest

import workloads as wl
from recorded_graph import recorded_prefill

pytestmark = pytest.mark.gpu

# kernels that write an auxiliary layer's keys and values, and predictor kernels, which read them: on the tensor cores, or not
PROJECTION = re.compile(r"gemm_tc_kernelILi3E|rope_split_kernel")
PREDICTOR = re.compile(r"gemm_tc_kernelILi4E|gemm_simt_kernelI\w+?Li2ELi")


def _narrow():
    """bf16, heads too narrow for the tensor-core kernels"""
    return wl.PairCfg("narrow", wl.uniform_model(4, 64, 2, 1, 32, 96, 97), wl.uniform_model(4, 64, 2, 1, 32, 96, 97), (0, 1, 2, 3))


@pytest.mark.parametrize("name,lens", [("t_small", [70, 63]), ("t_small", [9] * 6), ("t_small", [4096]), ("t_small_gap", [40, 9]),
                                       ("t_small_f32", [70]), ("t_hd128_qkn", [130]), ("narrow", [30, 7])], ids=str)
def test_predictor_is_ordered_against_every_projection(name, lens):
    pair = _narrow() if name == "narrow" else wl.pair(name)
    g = recorded_prefill(pair, lens)
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
    g = recorded_prefill(pair, lens)
    attention, predictors, lengths = g.find(re.compile("step_attn_mma_kernel")), g.find(PREDICTOR), g.find(re.compile("build_index_kernel"))
    assert len(attention) == pair.base.n_layers and len(predictors) == 2 * len(set(pair.layer_map)) and len(lengths) == 1
    first = min(len(set(predictors) & g.before(x)) for x in attention)
    assert first == 2      # its first layers do run beside the auxiliary layers
    for x in attention:
        assert set(lengths + predictors) & g.before(x) <= g.complete(x), "a page may be read while a predictor kernel writes it"


@pytest.mark.parametrize("name,lens", [("t_small_f32", [70, 63]), ("t_small_f32", [9] * 6), ("narrow", [30, 7])], ids=str)
def test_kernels_of_the_cuda_core_path_are_ordinary_launches(name, lens):
    """Recorded as dependent launches they made first calls and, while they waited, other kernels slower."""
    g = recorded_prefill(_narrow() if name == "narrow" else wl.pair(name), lens)
    nodes = g.find(re.compile("gemm_simt_kernel|attn_prefill_simt_kernel|rope_split_kernel|swiglu_kernel"))
    assert len(nodes) >= 7
    assert not any(early for x in nodes for _, early in g.edges[x])
