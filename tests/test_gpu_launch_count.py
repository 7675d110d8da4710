"""launches_per_step against the kernel nodes of the same calls captured into a CUDA graph, and that graph's replay against
the calls themselves (GPU)."""
import ctypes

import numpy as np
import pytest

import workloads as W
from tests.cases import make_case, gpu_console

pytestmark = pytest.mark.gpu


def kernel_nodes(graph) -> int:
    cu = ctypes.CDLL("libcuda.so.1")
    g, n = ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t(0)
    assert cu.cuGraphGetNodes(g, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(g, nodes, ctypes.byref(n)) == 0
    kind, kernels = ctypes.c_int(), 0
    for v in nodes:
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(v), ctypes.byref(kind)) == 0
        kernels += kind.value == 0
    return kernels


@pytest.mark.parametrize("types", ["ecnsgdr", "eg"])
def test_launches_per_step_counts_the_kernels(types):
    import torch
    case = make_case([W.SongLayout(3, 1, [0, 0, -1], 20011)], types=types, seed=27, n_fft=(512, 2048))
    con = gpu_console(case)
    con.set_params(case.params)
    con.train_step()
    con.reset_optimizer()
    con.set_params(case.params)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        losses = con.forward_loss()
        con.backward()
        con.adam_step()
    assert kernel_nodes(g) == con.get_info()["launches_per_step"]
    g.replay()
    torch.cuda.synchronize()
    got = [losses.cpu().numpy(), con.get_params().cpu().numpy()]
    con.reset_optimizer()
    con.set_params(case.params)
    want = [con.forward_loss().cpu().numpy()]
    con.backward()
    con.adam_step()
    want.append(con.get_params().cpu().numpy())
    for a, b in zip(got, want):
        assert np.array_equal(a, b)
