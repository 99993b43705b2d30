"""The gather vote's tiles at widths that are not whole strips of 256 columns (needs a GPU): every column of
every tile against the FP64 oracle, with the tile given and as a grid's default chooses it."""
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


@pytest.mark.parametrize("n_phi", [64, 192, 320, 384, 448, 704, 768, 960, 1344])
@pytest.mark.parametrize("n_layers", [3, 10, 13])
def test_default_tile_of_a_grid(binding, n_phi, n_layers):
    geo, ev = _event(n_layers)
    bn = eg.Binning(n_qpt=37, qpt_min=-2.0, qpt_max=2.0, n_phi=n_phi, threshold=max(2, n_layers - 3))
    check_event(binding, geo, bn, ev)


@pytest.mark.parametrize("rows, cols, threads", [(1, 64, 256), (3, 320, 256), (7, 640, 512), (32, 1920, 1024), (5, 960, 256)])
def test_given_tile(binding, rows, cols, threads):
    geo, ev = _event()
    bn = eg.Binning(n_qpt=70, qpt_min=-2.0, qpt_max=2.0, n_phi=1920, threshold=7)
    check_event(binding, geo, bn, ev, tiling=dict(gather_rows=rows, gather_cols=cols, gather_threads=threads))


def test_batch_tile(binding):
    geo, ev = _event()
    bn = eg.Binning(n_qpt=37, qpt_min=-2.0, qpt_max=2.0, n_phi=448, threshold=7)
    other = eg.simulate_event(geo, 20, (0.6, 50.0), 300, seed=3)
    with binding.HoughBatch(geo, bn, max_events=3, max_hits=2 * ev.n_hits + other.n_hits) as b:
        b.run_events([ev, other, ev])
        for e, x in enumerate((ev, other, ev)):
            ref = oracle.run(geo, bn, x)
            assert_accumulator_parity(b.accumulator(e), ref["M"], ref["vote_flags"])
