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
