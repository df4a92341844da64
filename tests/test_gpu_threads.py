"""Stateless solves from two host threads, each on its own stream, workspace
and outputs."""
import threading

import numpy as np
import pytest

import paper_1804_02883_gb300 as P
from paper_1804_02883_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_boxes_of_two_threads_do_not_disturb_each_other():
    # row tiles of 58 and 52 KB of one kernel, whose shared-memory limit both
    # threads' launches set
    import ctypes

    import torch

    def job(nz, ny, nx, seed):
        run = W.with_(W.plain_small(), nx=nx, ny=ny, ns=8)
        nb = P.epd_prop_solve3d_workspace_bytes(run, nz)
        gen = torch.Generator(device="cuda").manual_seed(seed)
        om = 0.1 * torch.rand((3, nz, ny, nx), generator=gen, dtype=torch.float64, device="cuda")
        ws = torch.empty(nb + 256, dtype=torch.uint8, device="cuda")
        phi = [torch.empty_like(om) for _ in range(2)]
        q = torch.empty(2, dtype=torch.float64, device="cuda")
        st = torch.cuda.Stream()
        st.wait_stream(torch.cuda.current_stream())

        def solve(out):
            return P.lib().epd_prop_solve3d(ctypes.byref(run.c()), nz, om.data_ptr(), phi[out].data_ptr(), q.data_ptr(),
                                            (ws.data_ptr() + 255) & ~255, nb, st.cuda_stream)

        return solve, phi

    jobs = [job(160, 256, 100, 1), job(256, 320, 50, 2)]
    for solve, _ in jobs:  # each alone
        assert solve(0) == 0
    torch.cuda.synchronize()
    codes = [[], []]
    start = threading.Barrier(2)

    def work(t):
        start.wait()
        for _ in range(12):
            codes[t].append(jobs[t][0](1))

    threads = [threading.Thread(target=work, args=(t,)) for t in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert codes == [[0] * 12] * 2
    for _, phi in jobs:
        assert np.array_equal(phi[0].cpu().numpy(), phi[1].cpu().numpy())
