"""Ratio tracking where many kernels cover a point (GPU).

A window's buffer holds 170 chords (256 in a small batch's form); beyond, the window is
traversed twice and its chords are added a buffer at a time.  The estimates' mean at the
buffer's edges, in a small batch and in a large one, and the number of tree nodes that a
dense ray visits.
"""
import numpy as np
import pytest

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


def _blob(n, depth, seed):
    """n kernels that all cover the centre; a ray through it has about `depth` points."""
    p = synth.absorption_field(n, seed=seed)
    rng = np.random.default_rng(seed)
    p["mu"] = (0.5 + 0.02 * rng.standard_normal((n, 3))).astype(np.float32)
    p["log_scale"] = np.log(rng.uniform(0.1, 0.14, (n, 3))).astype(np.float32)
    p["omega"] = rng.uniform(-6.0, 6.0, (n, 3)).astype(np.float32)
    # the integral of an envelope of scale 0.12 along a line is 0.3
    p["weight"] = (rng.uniform(0.5, 1.5, n) * depth / (0.3 * n)).astype(np.float32)
    return p


def _rays(n, seed):
    rng = np.random.default_rng(seed)
    u = rng.standard_normal((n, 3))
    o = 0.5 + 1.5 * u / np.linalg.norm(u, axis=1, keepdims=True)
    d = 0.5 + 0.1 * rng.standard_normal((n, 3)) - o
    tr = np.tile(np.array([0.0, 4.0], np.float32), (n, 1))
    return o.astype(np.float32), d.astype(np.float32), tr


@pytest.mark.parametrize("n,depth", [(120, 4), (169, 4), (170, 4), (171, 4), (256, 4), (257, 4), (340, 4),
                                     (700, 4), (700, 150)])
def test_dense_rays_are_unbiased(api, ctx, n, depth):
    """The mean of the estimates is exp(-tau) (quadrature), in a small batch and in a large
    one: within five standard errors of the rays' mean and 1e-4."""
    f = api.Field(ctx, _blob(n, depth, seed=n))
    o, d, tr = _rays(12_000, seed=2)
    for m, spp in ((500, 512), (o.shape[0], 32)):
        od, dd, trd = (torch.from_numpy(np.ascontiguousarray(a[:m])).cuda() for a in (o, d, tr))
        T, _ = f.transmittance(od, dd, trd, mode="rt", spp=spp, seed=7)
        Td, tau = f.transmittance(od, dd, trd, mode="det")
        f.sync()
        z = (T - Td).double()
        assert float(tau.abs().mean()) > 0.02  # the rays cross the field
        assert abs(float(z.mean())) <= 5 * float(z.std()) / m ** 0.5 + 1e-4, (m, float(z.mean()), float(z.std()))
    f.free()


@pytest.mark.parametrize("rays", [200, 12_000])
def test_dense_rays_are_traversed_twice(api, ctx, rays):
    """700 chords a ray and about ten points: one traversal for the points, one for the sums."""
    p = _blob(700, 10, seed=3)
    f = api.Field(ctx, p)
    od, dd, trd = (torch.from_numpy(a).cuda() for a in _rays(rays, seed=5))
    nodes = {}
    for mode in ("det", "rt"):
        f.stats(True)
        f.transmittance(od, dd, trd, mode=mode, spp=1, seed=7)
        f.sync()
        nodes[mode] = f.stats(True)["nodes"]
    assert nodes["rt"] <= 2 * nodes["det"], nodes
    f.free()
