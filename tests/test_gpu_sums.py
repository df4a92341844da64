"""The contour sums of MIXED_FP32 against sums in FP64 of the same chain."""
import numpy as np
import pytest

import paper_1804_02883_gb300 as P
from paper_1804_02883_gb300 import workloads as W
from helpers import rel_err

pytestmark = pytest.mark.gpu


def stateless(run, om, nbytes=None):
    import torch

    od = torch.from_numpy(om).cuda()
    pd, qd = torch.empty_like(od), torch.empty(2, dtype=torch.float64, device="cuda")
    nb = nbytes or P.epd_prop_solve_workspace_bytes(run)
    ws = torch.empty(nb + 256, dtype=torch.uint8, device="cuda")
    P.epd_prop_solve(run, od.data_ptr(), pd.data_ptr(), qd.data_ptr(), (ws.data_ptr() + 255) & ~255, nb,
                     torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return pd.cpu().numpy(), qd.cpu().numpy()


@pytest.mark.parametrize("jr", [0, 1])
@pytest.mark.parametrize("ny,nx,ns,f_a", [(150, 150, 17, 0.882), (96, 90, 32, 0.5), (32, 64, 64, 0.3), (12, 1458, 5, 0.0), (16, 10, 512, 1.0)])
def test_handle_sums_equal_fp64_sums(ny, nx, ns, f_a, jr):
    # grids of the general passes: a handle sums its full history in pairs of
    # FP32 values, a stateless solve of the same chain in FP64.  Per term a pair
    # rounds to 2^-47 of the sum: below 513 x 2^-47 = 4e-12
    run = W.with_(W.plain_small(), nx=nx, ny=ny, ns=ns, f_a=f_a, precision=P.MIXED_FP32, junction_rule=jr)
    om = W.random_omega(ny, nx, 5)
    phi, q = stateless(run, om)
    h = P.EpdLb([run])
    ph, qh = h.solve(0, om)
    h.close()
    assert np.array_equal(qh, q)
    for s in range(2):
        assert rel_err(ph[s], phi[s]) < 4e-12
    assert rel_err(ph[2], phi[2]) < 1e-15
