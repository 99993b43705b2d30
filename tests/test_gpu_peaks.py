"""The peak search of layer masks (needs a GPU) at the edges of what a warp and a band take: grids of less
than, exactly and more than a segment of 256 columns, plateaus across the seam of phi, bands taller than
the grid, every band height -- the candidates against the FP64 oracle."""
import numpy as np
import pytest

from paper_1310_7556_gb300 import eventgen as eg

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


@pytest.mark.parametrize("band_rows", [1, 2, 3, 8, 16])
@pytest.mark.parametrize("n_qpt, n_phi, threshold", [(1, 64, 1), (17, 64, 3), (40, 256, 5), (33, 704, 4), (9, 4096, 2)])
def test_bands(binding, band_rows, n_qpt, n_phi, threshold):
    geo = eg.Geometry()
    bn = eg.Binning(n_qpt=n_qpt, qpt_min=-1.0, qpt_max=1.0, n_phi=n_phi, threshold=threshold)
    ev = eg.simulate_event(geo, 40, (0.8, 50.0), 300, seed=n_qpt + n_phi)
    check_event(binding, geo, bn, ev, tiling=dict(band_rows=band_rows))


@pytest.mark.parametrize("n_layers", [1, 16])
def test_saturated_grid(binding, n_layers):
    """Nearly every cell at the same count: long plateaus, also across phi = +-pi."""
    geo = eg.Geometry(radii_cm=tuple(float(x) for x in np.linspace(4.0, 60.0, n_layers)))
    bn = eg.Binning(n_qpt=24, qpt_min=-1.0, qpt_max=1.0, n_phi=320 if n_layers == 1 else 256, threshold=n_layers)
    if n_layers == 1:
        bn = eg.Binning(n_qpt=24, qpt_min=-1.0, qpt_max=1.0, n_phi=512, threshold=1)
    ev = eg.simulate_event(geo, 0, (1.0, 50.0), 1500 * n_layers, seed=5)
    check_event(binding, geo, bn, ev)


@pytest.mark.parametrize("band_rows", [1, 2, 5, 16])
@pytest.mark.parametrize("n_qpt, n_phi, n_d0, threshold", [(1, 64, 1, 2), (7, 128, 3, 4), (18, 704, 2, 5), (5, 512, 9, 3)])
def test_bands_of_a_d0_grid(binding, band_rows, n_qpt, n_phi, n_d0, threshold):
    geo = eg.Geometry()
    bn = eg.Binning(n_qpt=n_qpt, qpt_min=-0.8, qpt_max=0.8, n_phi=n_phi, threshold=threshold, n_d0=n_d0, d0_min=-1.5,
                    d0_max=1.5)
    ev = eg.simulate_event(geo, 40, (1.5, 50.0), 300, seed=n_qpt + n_phi, d0_range=(-1.5, 1.5))
    check_event(binding, geo, bn, ev, tiling=dict(band_rows=band_rows))
