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


@pytest.mark.parametrize("case", ["plain", "normalised", "clamped", "camera", "foveated"])
def test_lanes_and_warps_agree_in_every_form(api, ctx, case):
    """The same calls by lanes and, under a stack limit that only the warps' kernels fit, by
    warps: ranges and none, host and device buffers, unnormalised directions, sample ranges,
    stochastic masks, and the fields and cameras of `case`.  Optical depths within 2e-6 max(1,
    |tau|) (the same terms in another order); flights up to 1 % of the pixels."""
    n = 12
    p = _field(n, seed=20)
    kw = {}
    if case == "normalised":
        s3 = np.exp(np.asarray(p["log_scale"], np.float64)).prod(1)
        p["weight"] = (p["weight"] * (2 * np.pi) ** 1.5 * s3).astype(np.float32)
        kw["weight_mode"] = "normalized"
    if case == "clamped":
        kw["clamp_eps"] = 0.05
    f = api.Field(ctx, p, **kw)
    c = synth.DEFAULT_CAMERA
    cam = api.camera(c["eye"], c["look_at"], c["up"], 55.0, 401, 307)
    if case == "camera":
        f.set_lod_camera(api.camera(c["eye"], c["look_at"], c["up"], 55.0, 40, 8))
    fov = {"gaze": (200.0, 150.0), "f0": 60.0, "slope": 300.0, "smooth": 0.3} if case == "foveated" else None
    o, d, tr = synth.random_rays(50_001, seed=8)
    d = (d * np.random.default_rng(1).uniform(0.1, 30.0, (len(d), 1))).astype(np.float32)
    od, dd, trd = (torch.from_numpy(a).cuda() for a in (o, d, tr))

    def results():
        out = {}
        for name, lod, spp in (("all", api.lod(), 1), ("stochastic", api.lod("unif_cv", 7, "is"), 3)):
            f.set_lod(lod)
            for mode in ("det", "closed"):
                _, tau = f.transmittance(od, dd, trd, mode=mode, spp=spp, seed=4)
                out["tau", name, mode] = tau.cpu()
                _, tau = f.transmittance(od, dd, None, mode=mode, spp=spp, seed=4)
                out["tau", name, mode, "no range"] = tau.cpu()
                T, tau = np.empty(len(o), np.float32), np.empty(len(o), np.float32)
                f.transmittance(o, d, tr, mode=mode, spp=spp, seed=4, out_T=T, out_tau=tau)
                out["tau", name, mode, "host"] = torch.from_numpy(tau)
            out["tau", name, "image"] = f.render(cam, api.render_opts("tomo", 2, first_sample=3, foveation=fov), 5).cpu()
            for ff in ("cdf", "segment"):
                ro = api.render_opts("scatter", 2, 2, free_flight=ff, first_sample=1, foveation=fov)
                out["flight", name, ff] = f.render(cam, ro, 5).cpu()
        f.sync()
        return out

    cu = ctypes.CDLL("libcuda.so.1")
    size = ctypes.c_size_t()
    lanes = results()
    assert cu.cuCtxGetLimit(ctypes.byref(size), 0) == 0
    try:
        assert cu.cuCtxSetLimit(0, ctypes.c_size_t(512)) == 0
        low = ctypes.c_size_t()
        assert cu.cuCtxGetLimit(ctypes.byref(low), 0) == 0 and low.value < 576  # the lanes' frames
        warps = results()
    finally:
        assert cu.cuCtxSetLimit(0, size) == 0
    for k, a in lanes.items():
        d = (a - warps[k]).abs()
        if k[0] == "tau":
            assert bool((d <= 2e-6 * a.abs().clamp(min=1.0)).all()), (k, float(d.max()))
            assert float(a.abs().max()) > 0.01
        else:
            assert float((d > 1e-4 * a.max()).float().mean()) <= 0.01, k
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
