"""Confirmation of the candidates (needs a GPU) where its grouping changes: candidates taken three or
two to a warp (detectors of up to 10, up to 16 layers), one warp or one CTA each; members past what a
warp lists at a time; buckets that wrap around phi; stage-2 grids other than 64 x 64.  Events alone are
compared with the FP64 oracle, batches with each event alone, record for record."""
import numpy as np
import pytest

from paper_1310_7556_gb300 import eventgen as eg

from test_gpu_parity import check_event, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1310_7556_gb300 import binding as b
    b.load()
    return b


def _geometry(n_layers):
    return eg.Geometry(radii_cm=tuple(float(x) for x in np.linspace(4.0, 110.0, n_layers)))


@pytest.mark.parametrize("n_layers, tracks, noise, n_qpt, n_phi, kw", [
    (10, 1, 0, 32, 64, {}),                                   # a handful of candidates
    (10, 40, 300, 65, 192, {}),                               # a CTA each
    (10, 400, 0, 1024, 2048, {"threshold": 5}),               # a warp for several
    (11, 60, 300, 65, 192, {}),
    (16, 400, 0, 512, 2048, {"threshold": 8}),
    (3, 200, 100, 64, 256, {"threshold": 2}),
    (10, 60, 200, 64, 256, {"n_cot": 33, "n_z0": 50}),        # runs that end on odd rows, a grid of partial words
    (12, 60, 200, 64, 256, {"n_cot": 256, "n_z0": 3}),
    (10, 60, 200, 64, 256, {"n_cot": 1, "n_z0": 256}),
])
@pytest.mark.parametrize("accumulator", [eg.ACC_LAYERS, eg.ACC_COUNTS])
def test_groups_match_oracle(binding, n_layers, tracks, noise, n_qpt, n_phi, kw, accumulator):
    geo = _geometry(n_layers)
    bn = eg.Binning(**{**dict(n_qpt=n_qpt, qpt_min=-1.0, qpt_max=1.0, n_phi=n_phi, threshold=max(2, n_layers - 3),
                              accumulator=accumulator), **kw})
    ev = eg.simulate_event(geo, tracks, (1.0, 50.0), noise, seed=31 + n_layers + tracks)
    check_event(binding, geo, bn, ev)


@pytest.mark.parametrize("jitter", [0.0, 0.3])
@pytest.mark.parametrize("hits", [95, 97, 400, 3000])
def test_crowded_cells_match_oracle(binding, hits, jitter):
    """Hits within a few azimuth bins around the seam at phi = +-pi: candidates with more members than
    a warp lists at a time, whose two buckets wrap around the axis; layers of one and of several radii."""
    geo = _geometry(10)
    rng = np.random.default_rng(hits)
    layer = rng.integers(0, 10, hits)
    phi = np.pi - 0.02 + rng.uniform(0.0, 0.04, hits)
    r = np.asarray(geo.radii_cm)[layer] + rng.uniform(-jitter, jitter, hits)
    ev = eg.Event(r.astype(np.float32), np.where(phi > np.pi, phi - 2 * np.pi, phi).astype(np.float32),
                  rng.uniform(-40.0, 40.0, hits).astype(np.float32), layer.astype(np.uint8), np.full(hits, -1, np.int32))
    bn = eg.Binning(n_qpt=16, qpt_min=-0.5, qpt_max=0.5, n_phi=128, threshold=6)
    check_event(binding, geo, bn, ev)


@pytest.mark.parametrize("n_layers", [10, 12])
def test_batch_groups_straddle_events(binding, n_layers):
    """Events of 0 to a few candidates among larger ones: groups that hold candidates of two events."""
    geo = _geometry(n_layers)
    bn = eg.Binning(n_qpt=64, qpt_min=-1.0, qpt_max=1.0, n_phi=256, threshold=n_layers - 2)
    events = [eg.simulate_event(geo, t, (1.0, 50.0), t, seed=7 * t + n_layers) for t in (30, 1, 0, 2, 80, 1, 1, 3, 50)]
    with binding.HoughBatch(geo, bn, max_events=len(events), max_hits=sum(e.n_hits for e in events)) as b:
        b.run_events(events)
        cands, offs = b.candidates()
        stats = [b.stats(e) for e in range(len(events))]
    for e, ev in enumerate(events):
        alone = run_gpu(binding, geo, bn, ev)
        assert np.array_equal(cands[offs[e]:offs[e + 1]], alone["candidates"]), f"event {e}"
        for k in ("n_members", "stage2_votes", "n_candidates"):
            assert getattr(stats[e], k) == getattr(alone["stats"], k), (e, k)


def test_list_read_before_and_between_stage2(binding):
    """The candidates read before stage 2 (cells and masks), and stage 2 run a second time, by the list
    or from the bands, give the records of one run."""
    w = eg.WORKLOADS["single_50trk"]
    ev = w.event(3)
    want = run_gpu(binding, w.geometry, w.binning, ev)["candidates"]
    for read_first in (False, True):
        with binding.HoughContext(w.geometry, w.binning, max_hits=ev.n_hits) as ctx:
            ctx.vote_event(ev)
            ctx.peaks()
            if read_first:
                early = ctx.candidates()
                for k in ("iq", "jphi", "mask"):
                    assert np.array_equal(early[k], want[k])
                assert not early["n_members"].any() and not early["mask2"].any()
            ctx.stage2()
            assert np.array_equal(ctx.candidates(), want)
            ctx.stage2()
            assert np.array_equal(ctx.candidates(), want)
