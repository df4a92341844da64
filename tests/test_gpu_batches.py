"""Batches past the sizes where the streaming passes change their tiles."""
import numpy as np
import pytest

import paper_1804_02883_gb300 as P
from paper_1804_02883_gb300 import workloads as W
from helpers import rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny,nx,runs", [(2048, 128, 38), (2048, 1024, 5), (512, 512, 19)])
def test_wide_batches_of_long_columns_step(ny, nx, runs):
    # the batches whose default column tile was refused, against their last
    # run stepped alone (FP32 densities of two steps: 1e-5)
    rs = [W.with_(W.plain_small(), nx=nx, ny=ny, ns=4, precision=P.MIXED_FP32, f0=0.0, seed=s + 1) for s in range(runs)]
    hb = P.EpdLb(rs)
    assert hb.tiles(0)["path"] == 1
    hb.step(2)
    hb.sync()
    hs = P.EpdLb(rs[-1:])
    hs.step(2)
    hs.sync()
    assert rel_err(hb.densities(runs - 1)[0], hs.densities(0)[0]) < 1e-5
    hb.close()
    hs.close()


def test_forms_of_the_chain_kernel_give_the_same_bits():
    # a run stepped alone (whole register file, cached factors), in a batch
    # that takes turns or shares SMs, and beside groups that fill the chip
    r = W.with_(W.plain_small(), nx=512, ny=256, ns=16, precision=P.MIXED_FP32, f0=1e-6, seed=9)
    others = [W.with_(r, seed=20 + s) for s in range(7)]
    crowd = [W.with_(r, ns=n, seed=n) for n in (8, 10, 12, 14)]
    ref = None
    for runs in ([r], [r] + others[:3], [r] + others, [r] + crowd):
        h = P.EpdLb(runs)
        h.step(2)
        h.sync()
        got = (*h.densities(0), h.velocity(0), h.get_state(0)[0])
        h.close()
        ref = ref or got
        for a, b in zip(got, ref):
            assert np.array_equal(a, b)
