"""Large batches and images through a few kernels, a ray per lane (GPU).

Up to 24 kernels (48 in closed form, 128 for images), and a 2,500th of the rays or pixels, a
ray goes to one lane instead of a warp.  At the lines, against the FP64 oracle, against small
batches, and the time that made the difference.
"""
import ctypes

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


def _field(n, seed):
    p = synth.absorption_field(n, seed=seed)
    rng = np.random.default_rng(seed)
    p["log_scale"] = (p["log_scale"] + 0.5).astype(np.float32)
    p["band"] = rng.integers(0, 4, n).astype(np.uint8)
    return p


@pytest.mark.parametrize("precision", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("n", [1, 2, 24, 25, 48, 49])
def test_batches_of_a_ray_per_lane(api, ctx, n, precision):
    """tau of a large batch equals that of the same rays in a small one within 2e-6 max(1,
    |tau|) (compensated sums of the same terms in another order), and the oracle's within the
    bound of the deterministic transmittance; ratio tracking has the mean exp(-tau)."""
    p = _field(n, seed=n)
    f = api.Field(ctx, p, precision=precision)
    o, d, tr = synth.random_rays(130_001, seed=3)
    od, dd, trd = (torch.from_numpy(a).cuda() for a in (o, d, tr))
    few = 300
    for lod in (api.lod(), api.lod("cutoff", 1), api.lod("all", 7, "thresh", 0.0, 0.4)):
        f.set_lod(lod)
        f.stats(True)
        for mode in ("det", "closed"):
            T, tau = f.transmittance(od, dd, trd, mode=mode)
            Ts, taus = f.transmittance(od[:few], dd[:few], trd[:few], mode=mode)
            f.sync()
            a, b = tau[:few].cpu().numpy(), taus.cpu().numpy()
            assert np.all(np.abs(a - b) <= 2e-6 * np.maximum(1.0, np.abs(a))), (mode, np.abs(a - b).max())
            assert torch.equal(T, torch.exp(-tau)) or float((T - torch.exp(-tau)).abs().max()) <= 1e-6 * float(T.max())
        assert f.stats(True)["rays"] == 2 * (130_001 + few)
    if precision == "fp32":
        f.set_lod(api.lod())
        _, ref = oracle.Field(p).transmittance(o[:few], d[:few], tr[:few], mode="det")
        _, tau = f.transmittance(od, dd, trd, mode="det")
        f.sync()
        err = np.abs(tau[:few].cpu().numpy() - ref)
        assert np.all(err <= 1e-5 * np.maximum(1.0, np.abs(ref))), err.max()
        T, _ = f.transmittance(od, dd, trd, mode="rt", spp=8, seed=2)
        f.sync()
        z = (T - torch.exp(-tau)).double()
        assert abs(float(z.mean())) <= 5 * float(z.std()) / 130_001 ** 0.5 + 1e-4
    f.free()


@pytest.mark.parametrize("n", [1, 40, 104, 105, 128, 129])
def test_images_of_a_ray_per_lane(api, ctx, n):
    """An image large enough for lanes holds the pixels that its samples' warps gave: the
    mean over samples in two halves equals the whole, and small renders by warps of the same
    camera agree where their pixels' streams do (the first rows)."""
    f = api.Field(ctx, _field(n, seed=n))
    c = synth.DEFAULT_CAMERA
    big = api.camera(c["eye"], c["look_at"], c["up"], 60.0, 640, 512)
    img = f.render(big, api.render_opts("tomo", 4), 7)
    a = f.render(big, api.render_opts("tomo", 2), 7)
    b = f.render(big, api.render_opts("tomo", 2, first_sample=2), 7)
    f.sync()
    assert float((img - 0.5 * (a + b)).abs().max()) <= 4 * 2.0 ** -24 * float(img.max())
    orc = oracle.Field(_field(n, seed=n))
    small = oracle.camera(c["eye"], c["look_at"], c["up"], 60.0, 640, 512)
    # the oracle's rays of some pixels
    pix = np.random.default_rng(1).integers(0, 640 * 512, 400)
    T = np.zeros(400)
    for s in range(4):
        ov = [oracle.camera_ray(small, 7, int(p % 640), int(p // 640), s) for p in pix]
        o = np.array([x[0] for x in ov], np.float32)
        v = np.array([x[1] for x in ov], np.float32)
        T += orc.transmittance(o, v, np.tile(np.array([0.0, 8.0], np.float32), (400, 1)), mode="det")[0] / 4
    err = np.abs(img.cpu().numpy().reshape(-1)[pix] - T)
    assert np.all(err <= 2e-5 * np.maximum(1.0, T)), err.max()
    f.free()


@pytest.mark.parametrize("ff", ["cdf", "segment"])
@pytest.mark.parametrize("n,w,h", [(1, 100, 80), (4, 200, 160), (5, 200, 160), (16, 400, 320), (17, 400, 320)])
def test_flight_images_of_a_ray_per_lane(api, ctx, ff, n, w, h):
    """Up to 16 kernels and a 7,500th of the pixels a flight image goes to lanes.  Against the
    oracle under shared streams (a non-negative mixture): pixels within 1e-4 of the largest,
    but for those where a decision lands on the other side in FP32 (1 %)."""
    p = _field(n, seed=n)
    p["omega"] = np.zeros_like(p["omega"])
    p["phase"] = np.zeros_like(p["phase"])
    f = api.Field(ctx, p)
    c = synth.DEFAULT_CAMERA
    cam = api.camera(c["eye"], c["look_at"], c["up"], 50.0, w, h)
    cor = oracle.camera(c["eye"], c["look_at"], c["up"], 50.0, w, h)
    img = f.render(cam, api.render_opts("scatter", 2, 3, free_flight=ff), seed=6)
    f.sync()
    ref = oracle.Field(p).render(cor, oracle.render_opts("scatter", 2, 3, free_flight=ff), seed=6)
    off = np.abs(img.cpu().numpy() - ref) > 1e-4 * ref.max()
    assert ref.max() > 0.0 and off.mean() <= 0.01, off.mean()
    f.free()


def test_a_smaller_stack_limit_takes_warps(api, ctx):
    """Another component may lower the context's stack limit (a limit of this process).  A
    lane's list then does not fit (1,824 bytes), and a pixel goes to a warp as in fields of
    more kernels: same image to rounding."""
    cu = ctypes.CDLL("libcuda.so.1")
    size = ctypes.c_size_t()
    torch.zeros(1, device="cuda")
    assert cu.cuCtxGetLimit(ctypes.byref(size), 0) == 0
    f = api.Field(ctx, _field(3, seed=3))
    c = synth.DEFAULT_CAMERA
    cam = api.camera(c["eye"], c["look_at"], c["up"], 50.0, 320, 240)
    o = api.render_opts("scatter", 1, 1, free_flight="cdf")
    lanes = f.render(cam, o, 3).clone()
    f.sync()
    try:
        assert cu.cuCtxSetLimit(0, ctypes.c_size_t(1024)) == 0
        warps = f.render(cam, o, 3).clone()
        f.sync()
    finally:
        assert cu.cuCtxSetLimit(0, size) == 0
    off = (lanes - warps).abs() > 1e-4 * lanes.max()
    assert float(lanes.max()) > 0.0 and float(off.float().mean()) <= 0.01
    f.free()


@pytest.mark.parametrize("ff,limit", [("cdf", 0.8), ("segment", 0.6)])
def test_few_kernel_flights_take_little_time(api, ctx, ff, limit):
    """A 1024x1024 flight image through 8 kernels: four times what it takes (ms)."""
    f = api.Field(ctx, synth.absorption_field(8, seed=1))
    c = synth.DEFAULT_CAMERA
    cam = api.camera(c["eye"], c["look_at"], c["up"], 45.0, 1024, 1024)
    o, img, times = api.render_opts("scatter", 1, 1, free_flight=ff), None, []
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        img = f.render(cam, o, 3, out=img)
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    assert sorted(times)[2] <= limit, times
    f.free()


@pytest.mark.parametrize("mode,limit", [("det", 1.2), ("closed", 1.0), ("rt", 1.4)])
def test_few_kernels_take_little_time(api, ctx, mode, limit):
    """2,000,000 rays through 8 kernels: three times what a ray per lane takes (ms)."""
    f = api.Field(ctx, synth.absorption_field(8, seed=1))
    o, d, _ = synth.random_rays(2_000_000, seed=3)
    od, dd = torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda()
    T, times = None, []
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        T, _ = f.transmittance(od, dd, mode=mode, out_T=T)
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    assert sorted(times)[2] <= limit, times
    f.free()


def test_work_counters_add_up(api, ctx):
    """The counters of a call, summed over its warps: a batch in two halves counts what the
    whole does, and chord counts are those of the chord lists."""
    f = api.Field(ctx, _field(60, seed=6))
    o, d, tr = synth.random_rays(6_000, seed=3)
    od, dd, trd = (torch.from_numpy(a).cuda() for a in (o, d, tr))
    for mode in ("det", "closed"):
        f.stats(True)
        f.transmittance(od, dd, trd, mode=mode)
        f.sync()
        whole = f.stats(True)
        for s in (slice(0, 2_500), slice(2_500, 6_000)):
            f.transmittance(od[s].contiguous(), dd[s].contiguous(), trd[s].contiguous(), mode=mode)
        f.sync()
        parts = f.stats(True)
        assert all(whole[k] == parts[k] for k in ("rays", "chords", "evals", "nodes", "windows", "leaves"))
        counts, _, _, _ = f.chords(o, d, tr, cap=64)
        assert whole["rays"] == 6_000 and whole["chords"] == int(counts.sum())
    f.free()
