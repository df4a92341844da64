"""The network on the smallest grid: alone, and in batches of more samples than
a grid dimension of 65535 holds planes of."""
import numpy as np
import pytest

import paper_1804_02883_gb300 as P
from paper_1804_02883_gb300 import surrogate as S
from test_gpu_surrogate import rand_params, test_tangent_matches_oracle as _tangent

pytestmark = pytest.mark.gpu


def test_tangent_on_the_smallest_grid():
    # its sums of the fields lie in the output's buffer, 8 KB a sample here
    import torch

    _tangent(torch, 16, 16)


@pytest.mark.parametrize("batch", [16384, 20000])
def test_samples_of_a_large_batch_equal_single_ones(batch):
    import torch

    run = P.RunParams(nx=16, ny=16, ns=8, precision=P.MIXED_FP32, phi_p=0.2, f_a=0.5)
    p = rand_params(3)
    gen = torch.Generator(device="cuda").manual_seed(5)
    om0 = 0.01 * torch.randn((batch, 3, 16, 16), generator=gen, dtype=torch.float64, device="cuda")
    om = om0 + 1e-5 * torch.randn((batch, 3, 16, 16), generator=gen, dtype=torch.float64, device="cuda")
    sur = S.Surrogate(run, batch, params=p, s_in=100.0, s_out=1e-3)
    one = S.Surrogate(run, 1, params=p, s_in=100.0, s_out=1e-3)
    phi = sur.forward(om0).cpu().numpy()
    phi0, phi1 = (t.cpu().numpy() for t in sur.tangent(om0, om))
    for b in (0, batch // 2, batch - 1):
        assert np.array_equal(one.forward(om0[b:b + 1]).cpu().numpy()[0], phi[b])
        a, c = (t.cpu().numpy()[0] for t in one.tangent(om0[b:b + 1], om[b:b + 1]))
        assert np.array_equal(a, phi0[b]) and np.array_equal(c, phi1[b])
