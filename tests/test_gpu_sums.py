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


# RMS error of Phi_A and Phi_B over their largest value, per grid, of the
# stateless MIXED_FP32 solves with radix-2 transforms and read twiddles (smooth
# fields of RMS 0.05 and noise, mean of three seeds): what any later solve keeps
RADIX2_RMS = {
    (64, 64, 32): 2.5387e-7, (64, 128, 64): 4.2111e-7, (128, 64, 24): 1.2415e-7, (128, 128, 64): 3.9270e-7,
    (128, 256, 40): 2.1481e-7, (256, 128, 64): 3.3935e-7, (256, 256, 32): 1.5922e-7, (128, 512, 64): 3.1791e-7,
    (512, 128, 48): 2.5676e-7, (256, 512, 64): 2.8740e-7, (512, 256, 96): 3.7735e-7, (512, 512, 32): 1.4365e-7,
    (64, 1024, 48): 2.2394e-7, (2048, 64, 32): 1.4473e-7, (1024, 512, 24): 9.3447e-8, (256, 2048, 16): 6.7729e-8,
    (64, 256, 64): 3.8114e-7,
}


def smooth_omega(ny, nx, seed):
    rng = np.random.default_rng(seed)
    k = np.sqrt(np.fft.fftfreq(ny)[:, None] ** 2 + np.fft.rfftfreq(nx)[None, :] ** 2)
    f = np.fft.irfft2(np.fft.rfft2(rng.standard_normal((3, ny, nx))) * np.exp(-(k * 2 * np.pi * 1.5) ** 2), s=(ny, nx))
    f -= f.mean(axis=(1, 2), keepdims=True)
    return 0.05 * f / f.std(axis=(1, 2), keepdims=True) + 1e-3 * (2 * rng.random((3, ny, nx)) - 1)


def rms_error(ny, nx, ns, nbytes=None):
    out = []
    for seed in (1, 2, 3):
        run = W.with_(W.plain_small(), nx=nx, ny=ny, ns=ns, precision=P.MIXED_FP32)
        om = smooth_omega(ny, nx, seed)
        phi, _ = stateless(run, om, nbytes)
        ref, _ = stateless(W.with_(run, precision=P.PLAIN_FP64), om)
        out.append(np.sqrt(((phi - ref)[:2] ** 2).mean()) / np.abs(ref[:2]).max())
    return float(np.mean(out))


@pytest.mark.parametrize("ny,nx,ns", list(RADIX2_RMS))
def test_stateless_solves_are_as_accurate_as_radix_2(ny, nx, ns):
    # with the queried workspace, and the streaming passes with a small one
    for nbytes in (None, ny * nx * (16 + (ns // 2 + 3) * 8) + 192 * 1024):
        assert rms_error(ny, nx, ns, nbytes) <= RADIX2_RMS[ny, nx, ns]


@pytest.mark.parametrize("jr", [0, 1])
@pytest.mark.parametrize("ny,nx,ns,f_a", [(64, 64, 32, 0.5), (128, 128, 64, 0.3), (128, 512, 10, 0.882), (512, 256, 12, 0.0), (256, 512, 8, 1.0)])
def test_resident_stateless_sums_equal_fp64_sums(ny, nx, ns, f_a, jr):
    # the states a_m = E_dep(m) g_m that the cluster kernel leaves in the
    # workspace (error word and partials, factors (E_A, E_B), three factor planes, the
    # states of both chains in pairs of rows), summed here in FP64
    import torch

    run = W.with_(W.plain_small(), nx=nx, ny=ny, ns=ns, f_a=f_a, precision=P.MIXED_FP32, junction_rule=jr)
    om = torch.from_numpy(W.random_omega(ny, nx, 7)).cuda()
    pd, qd = torch.empty_like(om), torch.empty(2, dtype=torch.float64, device="cuda")
    nb = P.epd_prop_solve_workspace_bytes(run)
    ws = torch.zeros(nb + 256, dtype=torch.uint8, device="cuda")
    off = -ws.data_ptr() % 256
    P.epd_prop_solve(run, om.data_ptr(), pd.data_ptr(), qd.data_ptr(), ws.data_ptr() + off, nb, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    phi, q = pd.cpu().numpy(), qd.cpu().numpy()
    raw, n = ws[off:].cpu().numpy(), ny * nx
    o = 256 + 4096 * 8
    e = raw[o:o + 8 * n].view(np.float32).reshape(ny, nx, 2).astype(np.float64)
    o += 8 * n + 12 * n
    a = raw[o:o + 8 * (ns + 1) * n].view(np.float32).reshape(2, ns + 1, ny // 2, nx, 2)
    a = a.transpose(0, 1, 2, 4, 3).reshape(2, ns + 1, ny, nx).astype(np.float64)
    na = int(np.round(f_a * ns))

    def block(chain, m):  # of the departing half-step
        if jr == 0:
            return int((m if chain == 0 else ns - m) >= na)
        j = m - 1 if m == ns else m
        return int((j if chain == 0 else ns - 1 - j) >= na)

    want = np.zeros((2, ny, nx))
    for m in range(ns + 1):
        t = (a[0, m] / e[..., block(0, m)]) * (a[1, ns - m] / e[..., block(1, ns - m)])
        if na and m <= na:
            want[0] += t * (0.5 if m in (0, na) else 1.0)
        if na < ns and m >= na:
            want[1] += t * (0.5 if m in (na, ns) else 1.0)
    qp = (a[0, ns] / e[..., block(0, ns)]).mean()
    assert abs(q[0] / qp - 1) < 1e-12
    want *= run.phi_p / ns / qp
    for s in range(2):
        assert rel_err(phi[s], want[s]) < 4e-12


# the same of the passes of radices 2 to 5 on grids that are not powers of two
RADIX5_RMS = {
    (150, 150, 17): 6.0607e-8, (270, 384, 24): 1.0300e-7, (96, 90, 32): 1.6063e-7, (32, 64, 32): 2.5659e-7,
    (128, 432, 24): 1.0157e-7, (320, 480, 24): 9.2380e-8, (200, 240, 33): 1.2030e-7, (54, 162, 48): 3.3837e-7,
    (486, 30, 40): 2.3627e-7, (36, 250, 48): 2.9919e-7, (1458, 40, 16): 5.9600e-8, (48, 96, 48): 3.5349e-7,
    (90, 1024, 24): 9.0197e-8, (180, 300, 32): 1.1285e-7,
}


def test_general_grids_are_as_accurate_as_small_radices():
    # on one grid a few per cent either way are chance; over these the errors
    # are no larger
    ratio = [rms_error(*g) / e for g, e in RADIX5_RMS.items()]
    assert np.exp(np.mean(np.log(ratio))) <= 1.0, ratio
