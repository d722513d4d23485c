"""gf_reserve under an allocator that refuses large blocks (GPU).

Later calls within the reserved sizes ask the allocator for nothing, whatever it refused,
and so run under stream capture; a further gf_reserve asks again.
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


class _Limited:
    """A context whose allocator refuses blocks above `limit` bytes and counts its calls."""

    def __init__(self, api, limit):
        from paper_2602_05081_gb300 import _abi
        self.limit, self.asked, self.refused = limit, 0, 0
        al = api.TorchAllocator(0)
        inner = al._on_alloc

        def on_alloc(user, nbytes, stream):
            self.asked += 1
            if nbytes > self.limit:
                self.refused += 1
                return None
            return inner(user, nbytes, stream)

        al._alloc = _abi.ALLOC_FN(on_alloc)
        al.c = _abi.gf_allocator(al._alloc, al._free, None)
        self.ctx = api.Context(0, allocator=al)
        self.freed = lambda: al.calls_free


def test_calls_after_a_refused_reserve_allocate_nothing(api):
    L = _Limited(api, 48 << 20)
    c = synth.DEFAULT_CAMERA
    cam = api.camera(c["eye"], c["look_at"], c["up"], c["vfov_deg"], 48, 40)
    f = api.Field(L.ctx, synth.octave_field(2000, 4, seed=4))
    f.reserve(max_pixels=48 * 40, render=True, adjoint=True)
    assert L.refused > 0
    asked, freed = L.asked, L.freed()
    dL = torch.ones(40, 48, device="cuda")
    out = torch.empty(40, 48, device="cuda")
    opts = {"single": api.render_opts("scatter", 2, 1), "path": api.render_opts("scatter", 1, 3),
            "tomo": api.render_opts("tomo", 2)}
    images = {}
    for k, o in opts.items():
        images[k] = f.render(cam, o, 3, out=out).clone()
        f.render_backward(cam, o, 4, dL)
    f.sync()
    assert (L.asked, L.freed()) == (asked, freed)
    # captured, and the same image
    g = torch.cuda.CUDAGraph()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(g, stream=s):
        f.render(cam, opts["path"], 3, out=out, stream=s.cuda_stream)
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, images["path"])
    assert (L.asked, L.freed()) == (asked, freed)
    # asked again, more is had, and the captured render still has its memory
    L.limit = 1 << 40
    f.reserve(max_pixels=48 * 40, render=True, adjoint=True)
    assert L.asked > asked
    asked, freed = L.asked, L.freed()
    for k, o in opts.items():
        assert torch.equal(images[k], f.render(cam, o, 3, out=out)), k
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, images["path"])
    assert (L.asked, L.freed()) == (asked, freed)
    del g
    f.free()
    L.ctx.close()


@pytest.mark.parametrize("ff", ["cdf", "segment"])
def test_flights_take_what_is_held(api, ff):
    """The chord lists of an analytic flight: within the reserved store, by the launch's own
    grid, and with the same image from fewer blocks or without lists."""
    c = synth.DEFAULT_CAMERA
    cam = api.camera(c["eye"], c["look_at"], c["up"], c["vfov_deg"], 120, 80)
    o = api.render_opts("scatter", 1, 2, free_flight=ff)
    p = synth.octave_field(2000, 4, seed=4)
    images = []
    for limit in (1 << 40, 200 << 20, 8 << 20):  # lists for every block, for a quarter, for none
        L = _Limited(api, limit)
        f = api.Field(L.ctx, p)
        if limit == 200 << 20:
            f.reserve(max_pixels=120 * 80, render=True)
        asked, freed = L.asked, L.freed()
        images.append(f.render(cam, o, 3).clone())
        f.sync()
        if limit == 200 << 20:
            assert (L.asked, L.freed()) == (asked, freed)
        f.free()
        L.ctx.close()
    assert torch.equal(images[0], images[1]) and torch.equal(images[0], images[2])
    # a small image needs few lists, and a captured flight keeps them when the field's
    # store grows
    L = _Limited(api, 1 << 40)
    f = api.Field(L.ctx, p)
    small = api.camera(c["eye"], c["look_at"], c["up"], c["vfov_deg"], 16, 8)
    out = torch.empty(8, 16, device="cuda")
    live = L.ctx.allocator.live_bytes
    want = f.render(small, o, 3, out=out).clone()
    assert L.ctx.allocator.live_bytes - live <= 64 << 20
    g = torch.cuda.CUDAGraph()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(g, stream=s):
        f.render(small, o, 3, out=out, stream=s.cuda_stream)
    f.render(cam, api.render_opts("scatter", 1, 2), 3)
    f.render(cam, o, 3)
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    del g
    f.free()
    L.ctx.close()


def test_tomography_adjoint_without_scratch(api):
    """Refused its arrays, or captured before they exist, the tomography adjoint runs without
    them.  Gradients are FP32 atomics of the same terms in another order: at most 48 * 40 *
    2 = 3,840 per entry, each rounding to 2^-24 of a partial sum of at most twice the largest
    entry: 2 * 3,840 * 2^-24 = 4.6e-4 of it."""
    c = synth.DEFAULT_CAMERA
    cam = api.camera(c["eye"], c["look_at"], c["up"], c["vfov_deg"], 48, 40)
    o = api.render_opts("tomo", 2)
    dL = torch.ones(40, 48, device="cuda")
    n = 2000
    for mode in ("peak", "normalized"):
        for frame in ("local", "world"):
            p = {**synth.octave_field(n, 4, seed=4), "weight_mode": mode, "omega_frame": frame}
            if mode == "normalized":  # the weights that give the same amplitudes
                s3 = np.exp(np.asarray(p["log_scale"], np.float64)).prod(1)
                p["weight"] = (p["weight"] * (2 * np.pi) ** 1.5 * s3).astype(np.float32)
            L = _Limited(api, 1 << 40)
            f = api.Field(L.ctx, p)
            # staging reserved by another call, nothing of the adjoint's
            f.reserve(max_pixels=48 * 40 + 16 * n)
            asked = L.asked
            grad = torch.full((15 * n,), 7.0, device="cuda")
            L.limit = 0
            f.render_backward(cam, o, 4, dL, grad=grad)
            f.sync()
            bare = grad.clone()
            L.limit = 1 << 40
            refused = L.asked
            g = torch.cuda.CUDAGraph()
            s = torch.cuda.Stream()
            s.wait_stream(torch.cuda.current_stream())
            with torch.cuda.graph(g, stream=s):
                f.render_backward(cam, o, 4, dL, grad=grad, stream=s.cuda_stream)
            assert L.asked == refused > asked
            grad.fill_(7.0)
            g.replay()
            torch.cuda.synchronize()
            captured = grad.clone()
            full = f.render_backward(cam, o, 4, dL)
            f.sync()
            assert L.asked > refused and float(full.abs().max()) > 0.0
            for k, v in api.split_grad(full, n).items():
                for other in (bare, captured):
                    d = (v - api.split_grad(other, n)[k]).abs().max() / v.abs().max()
                    assert float(d) <= 4.6e-4, (mode, frame, k, float(d))
            del g
            f.free()
            L.ctx.close()


def test_outgrown_scratch_is_given_back(api):
    """A store that a larger one replaces goes back to the allocator, but for one that a
    captured graph uses, which stays until the field is freed."""
    p = synth.octave_field(2000, 4, seed=4)
    c = synth.DEFAULT_CAMERA
    cam = api.camera(c["eye"], c["look_at"], c["up"], c["vfov_deg"], 24, 16)
    flight, delta = api.render_opts("scatter", 1, 1, free_flight="cdf"), api.render_opts("scatter", 1, 1)
    sizes = {}
    for captured in (False, True):
        L = _Limited(api, 1 << 40)
        al = L.ctx.allocator
        f = api.Field(L.ctx, p)
        out = torch.empty(16, 24, device="cuda")
        f.render(cam, flight, 3, out=out)
        f.sync()
        held = al.live_bytes
        g = torch.cuda.CUDAGraph()
        if captured:
            s = torch.cuda.Stream()
            s.wait_stream(torch.cuda.current_stream())
            with torch.cuda.graph(g, stream=s):
                f.render(cam, flight, 3, out=out, stream=s.cuda_stream)
        before = al.calls_free
        f.render(cam, delta, 3)
        f.sync()
        assert al.calls_free - before == (0 if captured else 1)
        sizes[captured] = al.live_bytes - held
        if captured:
            out.zero_()
            g.replay()
            torch.cuda.synchronize()
            assert float(out.max()) > 0.0
        del g
        f.free()
        L.ctx.close()
    assert sizes[True] > sizes[False]


def test_tomography_adjoint_with_few_lists_takes_the_whole_grid(api):
    """With lists for a small part of the grid's blocks the tomography adjoint goes without them
    on every block: a ray is traversed twice."""
    c = synth.DEFAULT_CAMERA
    cam = api.camera(c["eye"], c["look_at"], c["up"], c["vfov_deg"], 48, 40)
    o, dL, n = api.render_opts("tomo", 2), torch.ones(40, 48, device="cuda"), 2000
    nodes = {}
    for limit in (1 << 40, 1 << 20):  # 1 MiB: the arrays per kernel and ten blocks' lists
        L = _Limited(api, 1 << 40)
        f = api.Field(L.ctx, synth.octave_field(n, 4, seed=4))
        f.reserve(max_pixels=48 * 40 + 16 * n)
        L.limit = limit
        f.stats(True)
        f.render_backward(cam, o, 4, dL)
        f.sync()
        nodes[limit] = f.stats(True)["nodes"]
        f.free()
        L.ctx.close()
    assert nodes[1 << 20] == 2 * nodes[1 << 40]
