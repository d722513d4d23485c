"""Adjoints and analytic flights where their per-warp buffers overflow, against the FP64
oracle (GPU).

A warp holds up to 4,096 chords and 64 tentative points of a ray's window, 64 (then
128) chords covering a point, 1,024 chords of a tomography ray, 4,096 chords of an
analytic flight.  Each field here passes one of these limits, on few pixels.
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


def _field(n, tau, seed):
    """n absorption kernels scaled to a mean majorant depth of about tau: a kernel of
    scales s and weight w adds (2 pi)^1.5 s^3 w per unit area, s^3 2.05e-4 and w 1.25
    on average."""
    p = synth.absorption_field(n, seed=seed)
    p["weight"] = (p["weight"] * (tau / (15.75 * 2.05e-4 * 1.25 * n))).astype(np.float32)
    return p


def _check(g, g_ref, n, what):
    # both sides evaluate the same estimator on the same streams: they differ by FP32
    # arithmetic, relative ~1e-6 per term; each parameter block is held to 1e-3 of the
    # element plus 1e-4 of the block's largest element
    for name, lo, hi in (("mu", 0, 3), ("quat", 3, 7), ("log_scale", 7, 10), ("omega", 10, 13),
                         ("phase", 13, 14), ("weight", 14, 15)):
        a, b = g[lo * n:hi * n], g_ref[lo * n:hi * n]
        scale = np.abs(b).max()
        assert scale > 0, (what, name)
        worst = (np.abs(a - b) / (1e-3 * np.abs(b) + 1e-4 * scale)).max()
        print("%s %-9s worst |d| / lim %.2f" % (what, name, worst))
        assert worst <= 1.0, (what, name, worst)


@pytest.mark.parametrize("n,tau,res,bounces", [
    (6_000, 5.0, 6, 1),      # about 140 chords cover a point: more than 64
    (6_000, 5.0, 6, 2),
    (14_000, 5.0, 5, 1),     # about 320: more than 128
    (3_000, 300.0, 5, 1),    # more than 64 tentative points on a ray
    (3_000, 300.0, 5, 3),
    # about 18,000 chords on a ray, 5,000 covering a point: no window holds them
    (220_000, 80.0, 3, 2),
])
def test_radiance_adjoint_beyond_the_buffers(api, ctx, n, tau, res, bounces):
    p = _field(n, tau, seed=31)
    f = api.Field(ctx, p)
    c = synth.DEFAULT_CAMERA
    cg = api.camera(c["eye"], c["look_at"], c["up"], 30.0, res, res)
    co = oracle.camera(c["eye"], c["look_at"], c["up"], 30.0, res, res)
    dL = np.random.default_rng(7).standard_normal((res, res)).astype(np.float32)
    g = f.render_backward(cg, api.render_opts("scatter", 1, bounces), 5, torch.from_numpy(dL).cuda())
    f.sync()
    _, ref = oracle.Field(p).radiance_grad(co, oracle.render_opts("scatter", 1, bounces), 5, dLdI=dL)
    _check(g.cpu().numpy().astype(np.float64), ref, n, "n=%d" % n)


def test_tomography_adjoint_beyond_the_buffers(api, ctx):
    """About 1,400 chords on a ray: more than 1,024."""
    n, res = 14_000, 5
    p = _field(n, 2.0, seed=32)
    f = api.Field(ctx, p)
    c = synth.DEFAULT_CAMERA
    cg = api.camera(c["eye"], c["look_at"], c["up"], 30.0, res, res)
    co = oracle.camera(c["eye"], c["look_at"], c["up"], 30.0, res, res)
    orc = oracle.Field(p)
    target = np.zeros((res, res), np.float32)
    img = orc.tomo_image(co, 1, 5)
    dL = (2.0 * (img - target)).astype(np.float32)
    g = f.render_backward(cg, api.render_opts("tomo", 1), 5, torch.from_numpy(dL).cuda())
    f.sync()
    _, ref = orc.tomo_loss_grad(co, 1, 5, target)
    _check(g.cpu().numpy().astype(np.float64), ref, n, "tomography")


@pytest.mark.parametrize("flight", ["cdf", "segment"])
def test_analytic_flight_beyond_the_list(api, ctx, flight):
    """About 5,000 chords on a ray (Gaussians, so that the density is positive): every
    depth traverses the tree.  The radiance is smooth in the collision point, whose FP32
    depth is within 1e-5 of the target: 1e-3 of a pixel and 1e-4 of the largest."""
    n, res = 60_000, 4
    p = synth.octave_field(n, 1, seed=33)
    f = api.Field(ctx, p)
    c = synth.DEFAULT_CAMERA
    cg = api.camera(c["eye"], c["look_at"], c["up"], 30.0, res, res)
    co = oracle.camera(c["eye"], c["look_at"], c["up"], 30.0, res, res)
    img = f.render(cg, api.render_opts("scatter", 1, 2, free_flight=flight), seed=3)
    f.sync()
    ref = oracle.Field(p, omega_frame="local").render(
        co, oracle.render_opts("scatter", 1, 2, free_flight=flight), seed=3)
    a = img.cpu().numpy().astype(np.float64)
    assert ref.max() > 0
    assert np.all(np.abs(a - ref) <= 1e-3 * np.abs(ref) + 1e-4 * ref.max())
