"""The in-place transforms of the streaming passes on every kind of plan: two
to four radices, every first, inner and last radix, lines fewer than a tile,
columns that do not fill their last tile.  Single-chain solves against the
FP64 oracle: 1e-12 in FP64; FP32 2e-6 (transforms of O(1) fields over two
chains of N_s steps round to about 1e-7 of the largest value per step)."""
import numpy as np
import pytest

import oracle as O
import paper_1804_02883_gb300 as P
from paper_1804_02883_gb300 import workloads as W
from helpers import oracle_params, rel_err

GRIDS = [(8, 486), (162, 10), (250, 18), (54, 32), (2048, 8), (12, 1458), (1250, 12), (96, 90), (60, 108), (40, 270), (16, 1536), (200, 24)]


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [P.PLAIN_FP64, P.MIXED_FP32])
@pytest.mark.parametrize("ny,nx", GRIDS)
def test_solve_on_every_plan(ny, nx, precision):
    import torch

    run = P.RunParams(nx=nx, ny=ny, ns=4, precision=precision, f_a=0.25)
    om = W.random_omega(ny, nx, 11)
    od = torch.from_numpy(om).cuda()
    pd = torch.empty_like(od)
    qd = torch.empty(2, dtype=torch.float64, device="cuda")
    nb = P.epd_prop_solve_workspace_bytes(run)
    ws = torch.empty(nb + 256, dtype=torch.uint8, device="cuda")
    P.epd_prop_solve(run, od.data_ptr(), pd.data_ptr(), qd.data_ptr(), (ws.data_ptr() + 255) & ~255, nb,
                     torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    phi, q = O.solve(oracle_params(run), om)
    tol = 1e-12 if precision == P.PLAIN_FP64 else 2e-6
    assert rel_err(pd.cpu().numpy(), phi) < tol
    assert rel_err(qd.cpu().numpy(), q) < tol
    # a handle of one run: the full history and its own contour pass in MIXED_FP32
    h = P.EpdLb([run])
    ph, qh = h.solve(0, om)
    h.close()
    assert rel_err(ph, phi) < tol and rel_err(qh, q) < tol


@pytest.mark.gpu
@pytest.mark.parametrize("ny,nx,ns", [(64, 64, 8), (128, 128, 6), (64, 512, 4), (512, 256, 6), (512, 512, 4), (64, 2048, 4)])
def test_stateless_solve_takes_either_workspace(ny, nx, ns):
    """MIXED_FP32 on powers of two: the cluster-resident solve with the queried
    workspace, the streaming passes with one that only holds half the history
    (the size documented for the allocation-free call); grids without a
    cluster shape stream with both."""
    import torch

    run = P.RunParams(nx=nx, ny=ny, ns=ns, precision=P.MIXED_FP32, f_a=0.5)
    om = W.random_omega(ny, nx, 12)
    phi, q = O.solve(oracle_params(run), om)
    od = torch.from_numpy(om).cuda()
    nb = P.epd_prop_solve_workspace_bytes(run)
    for size in (nb, min(nb, ny * nx * (16 + (ns // 2 + 3) * 8) + 192 * 1024)):
        pd = torch.empty_like(od)
        qd = torch.empty(2, dtype=torch.float64, device="cuda")
        ws = torch.empty(size + 256, dtype=torch.uint8, device="cuda")
        P.epd_prop_solve(run, od.data_ptr(), pd.data_ptr(), qd.data_ptr(), (ws.data_ptr() + 255) & ~255, size,
                         torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        assert rel_err(pd.cpu().numpy(), phi) < 2e-6 and rel_err(qd.cpu().numpy(), q) < 2e-6


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [P.PLAIN_FP64, P.MIXED_FP32])
@pytest.mark.parametrize("nz,ny,nx", [(128, 144, 200), (160, 256, 100)])
def test_box_with_more_rows_than_partials(nz, ny, nx, precision):
    """Boxes of many x rows take more rows per tile to fit the Q partials, in
    more shared memory than a kernel has by default.  Fields constant along z
    give the 2D solve's densities in every plane (the same bounds as above)."""
    run = P.RunParams(nx=nx, ny=ny, ns=2, precision=precision)
    om = W.random_omega(ny, nx, 13)
    phi, q = P.prop_solve3d(run, np.repeat(om[:, None], nz, axis=1))
    h = P.EpdLb([run])
    ph, qh = h.solve(0, om)
    h.close()
    tol = 1e-12 if precision == P.PLAIN_FP64 else 4e-6  # FP32: both sides round
    assert rel_err(phi, np.repeat(ph[:, None], nz, axis=1)) < tol
    assert rel_err(q, qh) < tol
