"""The trees by cells and by bands where they are smallest, against the FP64 oracle (GPU).

Rays walk one tree per selected cone of a band with up to three of them, one tree per
band beyond; a class of one primitive is a tree of one node.  Small fields over few
cells reach every shape of root, and masks of each kind choose between the trees.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2602_05081_gb300 import api as _api
    return _api


@pytest.fixture(scope="module")
def ctx(api):
    c = api.Context(0)
    yield c
    c.close()


def _field(n, bands, seed):
    p = synth.absorption_field(n, seed=seed)
    rng = np.random.default_rng(seed)
    p["log_scale"] = (p["log_scale"] + 0.9).astype(np.float32)  # most rays cross most kernels
    p["band"] = np.asarray(bands, np.uint8)[rng.integers(0, len(bands), n)]
    return p


# (freq, max_band, cone, delta): every cone; a cutoff; cones below a threshold (three or
# fewer per band at 0.3, more at 0.9)
MASKS = [("all", 7, "all", 0.5), ("cutoff", 1, "all", 0.5), ("all", 7, "thresh", 0.3),
         ("all", 7, "thresh", 0.9)]
FREQ = {"all": 0, "cutoff": 1}
CONE = {"all": 0, "thresh": 3}


@pytest.mark.parametrize("n,bands", [(1, (0,)), (1, (7,)), (2, (0, 1)), (2, (3,)), (3, (0, 1, 7)),
                                     (5, (2,)), (9, (0, 1, 2)), (33, (0, 5)), (70, (0, 1, 2, 3, 4, 5, 6, 7)),
                                     (400, (1, 2))])
def test_optical_depth_on_small_trees(api, ctx, n, bands):
    """tau per ray within 1e-5 max(1, |tau|) of the oracle (the bound of the deterministic
    transmittance), by quadrature and in closed form."""
    p = _field(n, bands, seed=n)
    f, orc = api.Field(ctx, p), oracle.Field(p)
    o, d, tr = synth.random_rays(200, seed=3)
    od, dd, trd = (torch.from_numpy(a).cuda() for a in (o, d, tr))
    for freq, mb, cone, delta in MASKS:
        f.set_lod(api.lod(freq, mb, cone, 0.0, delta))
        lo = oracle.Lod(FREQ[freq], mb, CONE[cone], 0.0, delta)
        for mode in ("det", "closed"):
            _, tau = f.transmittance(od, dd, trd, mode=mode)
            f.sync()
            _, ref = orc.transmittance(o, d, tr, mode="det", lod=lo)
            err = np.abs(tau.cpu().numpy() - ref)
            assert np.all(err <= 1e-5 * np.maximum(1.0, np.abs(ref))), (n, bands, mode, freq, cone, err.max())


@pytest.mark.parametrize("n,bands", [(1, (0,)), (2, (0, 2)), (5, (1,)), (40, (0, 1, 2)), (300, (0, 3))])
def test_images_on_small_trees(api, ctx, n, bands):
    """Single and double scattering against the oracle under shared streams: pixels agree
    to FP32 rounding of a path (1e-4 of the largest pixel), except where a decision lands
    on the other side in FP32 (at most 1 % of the pixels)."""
    p = _field(n, bands, seed=n)
    f, orc = api.Field(ctx, p), oracle.Field(p)
    c = synth.DEFAULT_CAMERA
    cg = api.camera(c["eye"], c["look_at"], c["up"], 40.0, 16, 12)
    co = oracle.camera(c["eye"], c["look_at"], c["up"], 40.0, 16, 12)
    for freq, mb, cone, delta in MASKS:
        f.set_lod(api.lod(freq, mb, cone, 0.0, delta))
        lo = oracle.Lod(FREQ[freq], mb, CONE[cone], 0.0, delta)
        img = f.render(cg, api.render_opts("scatter", 2, 2), seed=6)
        f.sync()
        ref = orc.render(co, oracle.render_opts("scatter", 2, 2), seed=6, lod=lo, lod_nee=lo)
        a = img.cpu().numpy().astype(np.float64)
        off = np.abs(a - ref) > 1e-4 * max(ref.max(), 1e-6)
        assert off.mean() <= 0.01, (n, bands, freq, cone, off.sum())
