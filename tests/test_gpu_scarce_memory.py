"""Renders and adjoints whose scratch is refused at full size (GPU).

The kernels are persistent, so a grid of fewer blocks needs less scratch and gives the
same results: an allocator that refuses large blocks makes the library ask for half as
much, and so on.  Images are sums of integers and stay bit-equal; gradients are FP32
atomics, whose order changes.  An entry receives at most 48 * 40 * 6 = 11,520 of them (three
segments and three NEE rays per path); each rounds to 2^-24 of a partial sum of at most
twice the largest entry: 2 * 11,520 * 2^-24 = 1.4e-3 of it.
"""
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


def _results(api, limit):
    ctx = api.Context(0)
    al = ctx.allocator
    inner, largest = al._on_alloc, [0]

    def on_alloc(user, nbytes, stream):
        if nbytes > limit:
            return None
        largest[0] = max(largest[0], nbytes)
        return inner(user, nbytes, stream)

    from paper_2602_05081_gb300 import _abi
    al._alloc = _abi.ALLOC_FN(on_alloc)
    al.c = _abi.gf_allocator(al._alloc, al._free, None)
    ctx.close()
    ctx = api.Context(0, allocator=al)
    c = synth.DEFAULT_CAMERA
    cam = api.camera(c["eye"], c["look_at"], c["up"], c["vfov_deg"], 48, 40)
    f = api.Field(ctx, synth.octave_field(2000, 4, seed=4))
    dL = torch.ones(40, 48, device="cuda")
    opts = {"single": api.render_opts("scatter", 2, 1), "path": api.render_opts("scatter", 1, 3),
            "tomo": api.render_opts("tomo", 2)}
    out = {}
    for k, o in opts.items():
        out["image " + k] = f.render(cam, o, 3).clone()
        out["grad " + k] = f.render_backward(cam, o, 4, dL).clone()
    srv = api.Server(ctx, [f], mem_budget=1 << 20)
    ticket, img = srv.submit(0, cam, opts["single"], seed=3)
    srv.wait(ticket)
    out["image server"] = torch.as_tensor(img).clone()
    torch.cuda.synchronize()
    srv.close()
    f.free()
    ctx.close()
    return out, largest[0]


def test_smaller_grids_when_scratch_is_refused(api):
    full, asked = _results(api, 1 << 40)
    small, got = _results(api, 48 << 20)
    assert asked > 1 << 30 and got <= 48 << 20
    for k, a in full.items():
        if k.startswith("image"):
            assert torch.equal(a.cpu(), small[k].cpu()), k
        else:
            d = (a - small[k]).abs().max() / a.abs().max()
            assert float(d) <= 1.4e-3, (k, float(d))
