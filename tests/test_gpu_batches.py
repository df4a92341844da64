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


@pytest.mark.parametrize("precision,ny,nx,runs", [(P.PLAIN_FP64, 64, 64, 33), (P.MIXED_FP32, 150, 150, 17), (P.PLAIN_FP64, 90, 96, 24),
                                                  (P.MIXED_FP32, 64, 1024, 11), (P.MIXED_FP32, 512, 512, 9), (P.MIXED_FP32, 256, 2048, 3)])
def test_a_batch_equals_its_runs_stepped_alone(precision, ny, nx, runs):
    # batches past the sizes where the row passes take more rows per tile
    rs = [W.with_(W.plain_small(), nx=nx, ny=ny, ns=6, precision=precision, f0=0.0, seed=s + 1) for s in range(runs)]
    hb = P.EpdLb(rs)
    hb.step(2)
    hb.sync()
    for k in (0, runs - 1):
        hs = P.EpdLb([rs[k]])
        hs.step(2)
        hs.sync()
        for a, b in zip((*hb.densities(k), hb.velocity(k), hb.get_state(k)[0]), (*hs.densities(0), hs.velocity(0), hs.get_state(0)[0])):
            assert np.array_equal(a, b)
        hs.close()
    hb.close()
