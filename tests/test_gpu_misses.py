"""Rays that miss the scene, in batches and images (GPU).

A warp takes up to 32 rays of a batch and works only through those that meet the scene's
bounds; the others are answered by one lane each.  Of an image the warps take the pixels
around the projected bounds, and the background is filled.  Results, counters and
gradients must not depend on how rays that hit and rays that miss lie side by side.
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


def _rays(n, share, seed):
    """n rays of which about `share` aim at the unit cube, the others away from it."""
    rng = np.random.default_rng(seed)
    u = rng.standard_normal((n, 3))
    o = 0.5 + 1.5 * u / np.linalg.norm(u, axis=1, keepdims=True)
    d = rng.random((n, 3)) - o
    d[rng.random(n) >= share] *= -1.0
    return tuple(torch.from_numpy(a.astype(np.float32)).cuda() for a in (o, d))


@pytest.mark.parametrize("mode", ["det", "closed", "rt"])
@pytest.mark.parametrize("n,share", [(12_161, 0.5), (100_003, 0.0), (100_003, 0.03), (100_003, 0.9), (400_001, 0.3)])
def test_batches_with_misses(api, ctx, mode, n, share):
    """A batch equals the same rays with the misses taken out, and T = 1, tau = 0 where rays
    miss.  Rays keep their numbers only without the misses before them, so ratio tracking is
    compared on a batch whose rays that hit come first."""
    f = api.Field(ctx, synth.absorption_field(60, seed=1))
    o, d = _rays(n, share, seed=n)
    lo = torch.tensor([0.0, 6.0], device="cuda").expand(n, 2).contiguous()
    _, tau = f.transmittance(o, d, lo, mode="det")
    hit = tau != 0.0
    order = torch.argsort(~hit, stable=True)
    o, d, k = o[order].contiguous(), d[order].contiguous(), int(hit.sum())
    f.stats(True)
    T, tau = f.transmittance(o, d, lo, mode=mode, seed=3)
    f.sync()
    assert f.stats(True)["rays"] == n
    assert bool((T[k:] == 1.0).all()) and (tau is None or bool((tau[k:] == 0.0).all()))
    # the same rays again among others of their kind, and mixed up
    if mode != "rt":
        mix = torch.randperm(n, device="cuda")
        Tm, taum = f.transmittance(o[mix].contiguous(), d[mix].contiguous(), lo, mode=mode)
        assert torch.equal(Tm, T[mix]) and torch.equal(taum, tau[mix])
    elif k > 10_000:  # (a small batch takes another form of the terms)
        Tk, _ = f.transmittance(o[:k].contiguous(), d[:k].contiguous(), lo[:k].contiguous(), mode=mode, seed=3)
        assert torch.equal(Tk, T[:k])
    f.sync()
    f.free()


@pytest.mark.parametrize("w,h,vfov", [(37, 21, 150.0), (640, 400, 150.0), (640, 400, 20.0)])
def test_images_with_background(api, ctx, w, h, vfov):
    """Background pixels of tomography and flight images, and gradients that the background
    does not touch: the same from an image gradient that is zero there."""
    f = api.Field(ctx, synth.absorption_field(40, seed=2))
    c = synth.DEFAULT_CAMERA
    cam = api.camera(c["eye"], c["look_at"], c["up"], vfov, w, h)
    tomo = api.render_opts("tomo", 2)
    f.stats(True)
    img = f.render(cam, tomo, 5)
    f.sync()
    assert f.stats(True)["rays"] == 2 * w * h
    back = img == 1.0
    assert not bool(back.all()) and (bool(back.any()) or vfov < 90.0)
    for ff in ("cdf", "segment"):
        fl = f.render(cam, api.render_opts("scatter", 2, 1, free_flight=ff), 5)
        assert bool((fl[back] == 0.0).all()) and (float(fl.max()) > 0.0 or w < 100)
    dL = torch.rand(h, w, device="cuda")
    part = torch.where(back, torch.zeros_like(dL), dL)
    for o in (tomo, api.render_opts("scatter", 2, 1), api.render_opts("scatter", 2, 2)):
        a, b = f.render_backward(cam, o, 5, dL), f.render_backward(cam, o, 5, part)
        f.sync()
        # FP32 atomics of the same terms in another order, at most 6 w h of them per entry
        lim = 2.0 * 6 * w * h * 2.0 ** -24
        assert float((a - b).abs().max()) <= lim * float(a.abs().max()) and (float(a.abs().max()) > 0.0 or w < 100)
    f.sync()
    f.free()


def test_images_from_all_sides(api, ctx):
    """Tomography images against the FP64 oracle for cameras around, beside and inside the
    scene, near and far, wide and narrow: no pixel that a kernel reaches is taken for
    background.  A ray's place in FP32 is off by up to 4 * 2^-24 of its distance; across a ray
    an optical depth changes by at most 0.5 * 0.6 / 0.02 = 15 per unit and kernel, ten of
    them: 150 * 4 * 2^-24 = 3.6e-5 times the distance."""
    p = synth.absorption_field(30, seed=8)
    p["weight"] = np.abs(p["weight"]).astype(np.float32)
    p["omega"] = np.zeros_like(p["omega"])
    p["phase"] = np.zeros_like(p["phase"])
    f, orc = api.Field(ctx, p), oracle.Field(p)
    rng = np.random.default_rng(4)
    seen = 0
    for k in range(24):
        u = rng.standard_normal(3)
        eye = 0.5 + (0.2, 0.9, 1.4, 4.0, 60.0)[k % 5] * u / np.linalg.norm(u)
        at = 0.5 + (0.0, 0.4, 2.0)[k % 3] * rng.standard_normal(3)
        vfov = float(np.clip((20.0, 70.0, 140.0)[k % 3] / (1.0 if k % 5 < 3 else 8.0), 0.5, 170.0))
        w, h = ((31, 18), (17, 40), (64, 64))[k % 3]
        a = [float(x) for x in eye], [float(x) for x in at], (0.0, 1.0, 0.0), vfov, w, h
        img = f.render(api.camera(*a), api.render_opts("tomo", 2), 5)
        f.sync()
        ref = orc.render(oracle.camera(*a), oracle.render_opts("tomo", 2), 5)
        err = np.abs(img.cpu().numpy() - ref)
        assert err.max() <= 3.6e-5 * (1.0 + float(np.linalg.norm(eye - 0.5))), (k, err.max())
        seen += int((ref < 0.999).any())
    assert seen >= 8
    f.free()


@pytest.mark.parametrize("mode", ["det", "rt"])
def test_misses_cost_little(api, ctx, mode):
    """2,000,000 rays that miss: 64 MB of rays and results, at 100 GB/s at least."""
    f = api.Field(ctx, synth.absorption_field(256, seed=1))
    o, d = _rays(2_000_000, 0.0, seed=1)
    T, times = None, []
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        T, _ = f.transmittance(o, d, mode=mode, out_T=T)
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    assert bool((T == 1.0).all())
    assert sorted(times)[2] <= 0.64, times
    f.free()
