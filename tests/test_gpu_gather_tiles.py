"""The gather vote's tiles (needs a GPU): grids narrower than a tile's window, windows that wrap around phi,
detectors of up to 16 layers, the tile as a grid's default chooses it and given, alone and in a batch, each
cell against the FP64 oracle; grids with more rows than the rank form of the vote takes."""
import numpy as np
import pytest

import oracle
from paper_1310_7556_gb300 import eventgen as eg

from parity import assert_accumulator_parity
from test_gpu_parity import check_event

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1310_7556_gb300 import binding as b
    b.load()
    return b


def _event(n_layers=10):
    geo = eg.Geometry(radii_cm=tuple(float(x) for x in np.linspace(4.0, 110.0, n_layers)))
    return geo, eg.simulate_event(geo, 60, (0.6, 50.0), 200, seed=17 + n_layers)


@pytest.mark.parametrize("n_phi", [64, 128, 192, 256, 704, 1024])
@pytest.mark.parametrize("n_layers", [3, 8, 10, 11, 16])
def test_default_tile_of_a_grid(binding, n_phi, n_layers):
    geo, ev = _event(n_layers)
    bn = eg.Binning(n_qpt=37, qpt_min=-2.0, qpt_max=2.0, n_phi=n_phi, threshold=max(2, n_layers - 3))
    check_event(binding, geo, bn, ev)


@pytest.mark.parametrize("rows, cols, threads", [(1, 64, 256), (3, 128, 256), (7, 1024, 512), (32, 2048, 1024),
                                                 (5, 512, 256)])
def test_given_tile(binding, rows, cols, threads):
    geo, ev = _event()
    bn = eg.Binning(n_qpt=70, qpt_min=-2.0, qpt_max=2.0, n_phi=2048, threshold=7)
    check_event(binding, geo, bn, ev, tiling=dict(gather_rows=rows, gather_cols=cols, gather_threads=threads))


@pytest.mark.parametrize("n_qpt", [1, 2, 4095, 4096, 4097])
def test_rows_at_the_limit_of_the_ranks(binding, n_qpt):
    geo, ev = _event()
    bn = eg.Binning(n_qpt=n_qpt, qpt_min=-2.0, qpt_max=2.0, n_phi=128, threshold=8)
    check_event(binding, geo, bn, ev.subset(np.arange(0, ev.n_hits, 3)))


def test_change_of_mode_between_events(binding):
    """The bucket profile is left empty for the next event whichever kernel read it last."""
    w = eg.WORKLOADS["single_50trk"]
    evs = [w.event(k) for k in range(4)]
    want = [oracle.run(w.geometry, w.binning, e) for e in evs]
    with binding.HoughContext(w.geometry, w.binning, max_hits=max(e.n_hits for e in evs)) as ctx:
        for ev, ref, mode in zip(evs, want, (0, 1, 0, 0)):
            ctx.set_tiling(vote_mode=mode)
            ctx.vote_event(ev)
            ctx.peaks()
            ctx.stage2()
            assert_accumulator_parity(ctx.accumulator(), ref["M"], ref["vote_flags"])


def test_batch_tile(binding):
    geo, ev = _event()
    bn = eg.Binning(n_qpt=37, qpt_min=-2.0, qpt_max=2.0, n_phi=512, threshold=7)
    other = eg.simulate_event(geo, 20, (0.6, 50.0), 300, seed=3)
    with binding.HoughBatch(geo, bn, max_events=3, max_hits=2 * ev.n_hits + other.n_hits) as b:
        b.run_events([ev, other, ev])
        for e, x in enumerate((ev, other, ev)):
            ref = oracle.run(geo, bn, x)
            assert_accumulator_parity(b.accumulator(e), ref["M"], ref["vote_flags"])
