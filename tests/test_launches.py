"""Launches of the library's host side, checked without a GPU (fake_runtime)."""
import pytest

import paper_1804_02883_gb300 as P
from paper_1804_02883_gb300 import workloads as W
from fake_runtime import FakeRuntime


@pytest.fixture(scope="module")
def rt(tmp_path_factory):
    return FakeRuntime(str(tmp_path_factory.mktemp("fake")))


@pytest.mark.parametrize("ny", [64, 128, 256, 512, 1024, 2048])
def test_default_column_tiles_launch_for_every_batch(rt, ny):
    """epd_lb_init solves Phi(0) before it times the column widths: the default
    width has to launch whatever the batch."""
    for nx in (64, 128, 256, 512, 1024, 2048):
        for runs in (1, 2, 3, 5, 10, 19, 38, 64):
            r = W.with_(W.plain_small(), nx=nx, ny=ny, ns=2, precision=P.MIXED_FP32, f0=0.0)
            rc, _ = rt.init([W.with_(r, seed=s) for s in range(runs)])
            assert rc == 0, (nx, runs)


def test_shared_memory_limits_never_fall(rt):
    """The limit is the function's, shared by every host thread: a launch that
    lowered it would fail another thread's launch of a wider tile.  Boxes whose
    row tiles (58 and 52 KB) are one kernel's, the wider one first and last."""
    boxes = [(160, 256, 100), (256, 320, 50), (160, 256, 100)]
    for precision in (P.PLAIN_FP64, P.MIXED_FP32):
        for nz, ny, nx in boxes:
            assert rt.solve3d(W.with_(W.plain_small(), nx=nx, ny=ny, ns=2, precision=precision), nz) == 0
            assert rt.L.fake_lowered() == 0


CLUSTER_GRIDS = [(64, 64), (64, 128), (128, 64), (128, 128), (128, 256), (256, 128), (256, 256), (128, 512), (512, 128), (256, 512), (512, 256)]


def test_kernel_attributes_are_set_on_every_device(rt):
    """Shared-memory limits and cluster sizes belong to a device: a process that
    used one device solves, steps and runs the network on the next."""
    for dev in (0, 1):
        rt.L.fake_device(dev)
        try:
            for ny, nx in CLUSTER_GRIDS:
                r = W.with_(W.plain_small(), nx=nx, ny=ny, ns=2, precision=P.MIXED_FP32, f0=0.0)
                assert rt.solve(r) == 0
                assert any("prop_chain" in l[0] for l in rt.launches())
                rc, out = rt.init([r])
                assert rc == 0 and any("epd_row8" in l[0] for l in out)
            assert rt.sur_forward(W.with_(W.plain_small(), nx=64, ny=64), 2) == 0
            assert sum("conv3x3_tc" in l[0] for l in rt.launches()) == 4
        finally:
            rt.L.fake_device(0)


def _chains(out):
    """Template arguments of the chain launches: log2 nx and ny, CTAs, threads, CTAs per SM
    the registers are sized for, differential, cached, every twiddle read."""
    return [l[1] for l in out if "prop_chain" in l[0]]


def test_chains_share_an_sm_only_where_the_groups_fill_the_chip(rt):
    """Groups stepped side by side take the half-register form once their
    clusters are more than the SMs; two small ones, and the benchmark batch
    beside a small run, keep the whole register file, the batch its turns."""
    def run(ny, nx, n, ns=16):
        r = W.with_(W.plain_small(), nx=nx, ny=ny, ns=ns, precision=P.MIXED_FP32, f0=0.0)
        return [W.with_(r, seed=s) for s in range(n)]

    rc, out = rt.init(run(128, 128, 1) + run(128, 256, 1))
    assert rc == 0 and _chains(out) and all(a[6] == 1 for a in _chains(out))
    rc, out = rt.init(run(256, 512, 4) + run(128, 128, 1))
    wide = [a for a in _chains(out) if a[:2] == (9, 8)]
    # Phi(0), then two solves a step in two graphs, 8 launches each
    assert rc == 0 and len(wide) == 5 * 8 and all(a[4] == 1 for a in wide)
    rc, out = rt.init(W.ensemble_32())
    step = _chains(out)[len({(r.ny, r.nx, r.ns) for r in W.ensemble_32()}):]  # after the solves of Phi(0)
    assert rc == 0 and step and all(a[4] == 2 and a[6] == 0 for a in step if a[2] >= 4)


def test_groups_of_an_exact_step_run_alone(rt):
    """The exact step takes its groups one after the other."""
    rc, out = rt.step_exact(W.ensemble_32(), 2)
    assert rc == 0 and _chains(out) and all(a[6] == 1 for a in _chains(out) if a[2] < 16)


@pytest.mark.parametrize("precision,ny,nx", [(P.PLAIN_FP64, 64, 64), (P.MIXED_FP32, 150, 150), (P.MIXED_FP32, 64, 1024), (P.MIXED_FP32, 1024, 512)])
def test_q_is_summed_over_the_same_tiles_in_every_batch(rt, precision, ny, nx):
    """The last row pass of a solve leaves the Q partials: its tile, and so the
    order of the sum, is that of one run whatever the batch."""
    tiles = set()
    for n in (1, 2, 10, 16, 32, 64):
        r = W.with_(W.plain_small(), nx=nx, ny=ny, ns=4, precision=precision, f0=0.0)
        rc, out = rt.init([W.with_(r, seed=s) for s in range(n)])
        assert rc == 0
        for a, b in zip(out, out[1:]):
            if "prop_finalize" in b[0] or "prop_contour_stream" in b[0]:
                tiles.add((a[1], a[2][0], a[3]))
    assert len({t[1:] for t in tiles}) == 1, tiles


def _dw_split(tiles):
    """CTAs of the weight-gradient kernel, and tiles per CTA and per accumulator (restated)."""
    per512 = -(-tiles // 512)
    cap = min(512, tiles) if per512 == 1 else 304
    per = -(-tiles // cap)
    return -(-tiles // per), per, max(1, per512 - 1)


def test_weight_gradient_values_pass_few_roundings():
    """8 chunks of 16 pixels a tile in turn, then the accumulators added: no more
    roundings than the chunks of one in 512 of the tiles, whose partials (the CTAs')
    are added in FP64."""
    for tiles in range(1, 70000):
        _, per, seg = _dw_split(tiles)
        assert 8 * min(seg, per) + -(-per // seg) - 1 <= 8 * -(-tiles // 512), tiles


@pytest.mark.parametrize("batch,ny,nx", [(4, 256, 512), (1, 256, 256), (8, 512, 512), (1, 16, 16), (3, 48, 80), (2, 240, 160)])
def test_weight_gradient_ctas(rt, batch, ny, nx):
    assert rt.sur_gradients(W.with_(W.plain_small(), nx=nx, ny=ny), batch) == 0
    dw = [l for l in rt.launches() if "conv3x3_dw" in l[0]]
    assert len(dw) == 4 and all(l[2][0] == _dw_split(batch * ny * nx // 128)[0] for l in dw)


@pytest.mark.parametrize("batch", [1, 16000, 16384, 21845, 30000])
def test_network_takes_large_batches_of_small_grids(rt, batch):
    """The planes of a batch are a grid dimension: 65535 in y, 2^31 - 1 in x."""
    assert rt.sur_forward(W.with_(W.plain_small(), nx=16, ny=16), batch) == 0
