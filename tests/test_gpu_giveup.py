"""A stateless solve whose exchange wait gave up: nobody reads its error word,
so the outputs say so."""
import ctypes

import numpy as np
import pytest

import paper_1804_02883_gb300 as P
from paper_1804_02883_gb300 import workloads as W

pytestmark = pytest.mark.gpu


class MemsetParams(ctypes.Structure):  # CUDA_MEMSET_NODE_PARAMS
    _fields_ = [("dst", ctypes.c_uint64), ("pitch", ctypes.c_size_t), ("value", ctypes.c_uint), ("element", ctypes.c_uint),
                ("width", ctypes.c_size_t), ("height", ctypes.c_size_t)]


def _preset_error_word(graph, word_ptr):
    """Let the captured call start with the give-up bit set (its clearing of the
    error word writes 4 per byte instead of 0): what the chain kernel leaves
    after a wait that ran out, without one running out."""
    cu = ctypes.CDLL("libcuda.so.1")
    n = ctypes.c_size_t()
    assert cu.cuGraphGetNodes(ctypes.c_void_p(graph), None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(ctypes.c_void_p(graph), nodes, ctypes.byref(n)) == 0
    done = 0
    for node in nodes:
        t = ctypes.c_int()
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(t)) == 0
        if t.value != 2:  # CU_GRAPH_NODE_TYPE_MEMSET
            continue
        p = MemsetParams()
        assert cu.cuGraphMemsetNodeGetParams(ctypes.c_void_p(node), ctypes.byref(p)) == 0
        if p.dst == word_ptr and p.width * p.element * p.height == 4:
            p.value = 4 if p.element == 1 else 0x04040404
            assert cu.cuGraphMemsetNodeSetParams(ctypes.c_void_p(node), ctypes.byref(p)) == 0
            done += 1
    assert done == 1


def test_outputs_of_a_solve_that_gave_up_are_nan():
    import torch

    run = W.with_(W.plain_small(), nx=64, ny=64, ns=8, precision=P.MIXED_FP32)
    om = torch.from_numpy(W.random_omega(64, 64, 3)).cuda()
    nb = P.epd_prop_solve_workspace_bytes(run)
    ws = torch.empty(nb + 256, dtype=torch.uint8, device="cuda")
    wptr = (ws.data_ptr() + 255) & ~255  # the error word is the workspace's first
    phi, q = torch.empty_like(om), torch.empty(2, dtype=torch.float64, device="cuda")

    def solve():
        P.epd_prop_solve(run, om.data_ptr(), phi.data_ptr(), q.data_ptr(), wptr, nb, torch.cuda.current_stream().cuda_stream)

    def outputs():
        torch.cuda.synchronize()
        return phi.cpu().numpy().copy(), q.cpu().numpy().copy()

    solve()
    want = outputs()
    assert np.isfinite(want[0]).all() and (want[1] > 0).all()
    graphs = []
    for preset in (False, True):
        g = torch.cuda.CUDAGraph(keep_graph=True)
        with torch.cuda.graph(g):
            solve()
        if preset:
            _preset_error_word(g.raw_cuda_graph(), wptr)
        g.instantiate()
        g.replay()
        got = outputs()
        if preset:
            assert np.isnan(got[0]).all() and np.isnan(got[1]).all()
        else:
            assert all(np.array_equal(a, b) for a, b in zip(got, want))
        graphs.append(g)
    solve()  # and the next call is a good one
    assert all(np.array_equal(a, b) for a, b in zip(outputs(), want))
