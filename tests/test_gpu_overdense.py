"""Renders of fields that more kernels cover than a window can hold (GPU).

A window stores 448 chords.  Where 600 kernels cover every point of a region no window
can be halved far enough: such a render reports GF_EOVERFLOW after the halvings of each
ray (under a hundred windows, tests/test_windows.py), and a field beside it on the same
server or context is rendered as ever.
"""
import time

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


def _blob(n, seed):
    p = synth.absorption_field(n, seed=seed)
    rng = np.random.default_rng(seed)
    p["mu"] = (0.5 + 0.02 * rng.standard_normal((n, 3))).astype(np.float32)
    p["log_scale"] = np.log(rng.uniform(0.1, 0.12, (n, 3))).astype(np.float32)
    p["weight"] = (0.01 * p["weight"]).astype(np.float32)
    return p


def test_overdense_field_reports_overflow_at_once(api):
    from paper_2602_05081_gb300 import _abi
    ctx = api.Context(0)
    c = synth.DEFAULT_CAMERA
    cam = api.camera(c["eye"], c["look_at"], c["up"], c["vfov_deg"], 24, 16)
    plain = api.Field(ctx, synth.octave_field(2000, 4, seed=4))
    opts = api.render_opts("scatter", 2, 2)
    want = plain.render(cam, opts, 3).clone()
    plain.sync()
    dense = api.Field(ctx, _blob(600, 5))
    t0 = time.time()
    dense.render(cam, opts, 3)
    with pytest.raises(_abi.GfError) as e:
        dense.sync()
    assert e.value.status == _abi.GF_EOVERFLOW
    assert time.time() - t0 < 10.0
    again = plain.render(cam, opts, 3)
    plain.sync()
    assert torch.equal(want, again)
    dense.free()
    plain.free()
    ctx.close()
