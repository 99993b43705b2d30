"""The vote of layers whose hits lie at several radii (needs a GPU): radii close together (the cubic of the
arcsine, and its form near |x| = 1 on the outer rows), far apart (an arcsine per vote), one layer of several
radii among uniform ones, windows as wide as the axis, tiles cut by the grid's edges, masks and counts,
alone and in a batch -- each cell against the FP64 oracle."""
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


def _event(jitter, seed, n=60, noise=400):
    return eg.simulate_event(eg.Geometry(), n, (0.5, 50.0), noise, seed=seed, radius_jitter_cm=jitter)


@pytest.mark.parametrize("jitter", [0.01, 0.5, 2.0, 3.9])
@pytest.mark.parametrize("n_qpt, n_phi, qpt", [(64, 64, 2.0), (33, 320, 1.0), (200, 2048, 2.0), (96, 4096, 1.6), (1, 128, 0.1)])
@pytest.mark.parametrize("acc", [eg.ACC_LAYERS, eg.ACC_COUNTS])
def test_radii_match_oracle(binding, jitter, n_qpt, n_phi, qpt, acc):
    bn = eg.Binning(n_qpt=n_qpt, qpt_min=-qpt, qpt_max=qpt, n_phi=n_phi, threshold=6, accumulator=acc)
    if acc == eg.ACC_LAYERS and n_phi == 320:
        bn = eg.Binning(n_qpt=n_qpt, qpt_min=-qpt, qpt_max=qpt, n_phi=512, threshold=6)
    check_event(binding, eg.Geometry(), bn, _event(jitter, seed=3))


def test_one_layer_of_several_radii(binding):
    ev = _event(0.0, seed=9)
    r = ev.r.copy()
    outer = np.flatnonzero(ev.layer == 9)
    r[outer] += np.linspace(-0.8, 0.8, outer.size).astype(np.float32)
    ev.r[:] = r
    bn = eg.Binning(n_qpt=128, qpt_min=-2.0, qpt_max=2.0, n_phi=1024, threshold=7)
    res = check_event(binding, eg.Geometry(), bn, ev)
    assert res["got"]["stats"].uniform_layers == (1 << 9) - 1


def test_batch(binding):
    bn = eg.Binning(n_qpt=70, qpt_min=-2.0, qpt_max=2.0, n_phi=512, threshold=7)
    events = [_event(0.5, seed=k, n=20 * k + 5) for k in range(5)]
    with binding.HoughBatch(eg.Geometry(), bn, max_events=5, max_hits=sum(e.n_hits for e in events)) as b:
        b.run_events(events)
        for e, ev in enumerate(events):
            ref = oracle.run(eg.Geometry(), bn, ev)
            assert_accumulator_parity(b.accumulator(e), ref["M"], ref["vote_flags"])
            assert int(b.stats(e).votes) == int(ref["votes_by_layer"].sum())
