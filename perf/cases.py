"""The work that users of the renderer have it do, as timed cases.

Each case is a plain dict; ``prepare`` makes the inputs and whatever a program
keeps between calls (a built field, a render server), ``run`` makes one pass
through the public API, ``work`` gives the bytes and operations of a pass and
``exact`` its outputs in 64-bit arithmetic where plain torch gives them in
reasonable time.

Kinds:
  trans    transmittance of a batch of rays through a resident field
  render   one image of a resident field (scattering, or tomography)
  step     one optimisation step: pack the parameters, render, loss, gradients
  serve    a burst of render requests to a render server over resident fields

Fields follow the recipes of the package's synthetic workloads: "absorb" is a
set of Gabor kernels in the unit cube with carriers of 0 to 8 cycles per unit,
"octave" a pyramid whose octaves quadruple the kernels and halve the scales.
"""
import math

import torch

from paper_2602_05081_gb300 import api

TWO_PI = 2.0 * math.pi
EYE, LOOK_AT, UP, VFOV = (0.5, 0.5, -1.0), (0.5, 0.5, 0.5), (0.0, 1.0, 0.0), 45.0
KEYS = ("mu", "quat", "log_scale", "omega", "phase", "weight")
S_LO, S_HI = 0.02, 0.1  # scales of the absorption field and of octave 0
MEAN_S = (S_HI - S_LO) / math.log(S_HI / S_LO)
MEAN_S2 = (S_HI ** 2 - S_LO ** 2) / (2.0 * math.log(S_HI / S_LO))
K_SIGMA = 3.0

_ctx = None


def _context():
    global _ctx
    if _ctx is None:
        _ctx = api.Context(0)
    return _ctx


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def _trans(name, field, n, octaves, rays, mode, precision="fp32", **kw):
    return dict(name=name, kind="trans", field=field, n=n, octaves=octaves, rays=rays, mode=mode,
                precision=precision, freq="all", max_band=7, **kw)


def _render(name, n, octaves, width, height, spp, bounces, freq="all", max_band=7, cone="all",
            precision="fp32", flight="delta", integrator="scatter", beta=0.0, delta=0.5):
    return dict(name=name, kind="render", n=n, octaves=octaves, width=width, height=height, spp=spp,
                bounces=bounces, freq=freq, max_band=max_band, cone=cone, precision=precision,
                flight=flight, integrator=integrator, beta=beta, delta=delta)


def _step(name, n, octaves, width, height, spp, bounces, integrator):
    return dict(name=name, kind="step", n=n, octaves=octaves, width=width, height=height, spp=spp,
                bounces=bounces, integrator=integrator)


def listed():
    return [
        # absorption tomography of a small asset: the smallest call, one 64x64 detector of
        # parallel rays, by quadrature and by one-sample ratio tracking (launch and latency)
        _trans("absorb_det_4096", "absorb", 256, 1, 4096, "det"),
        _trans("absorb_ratio_4096", "absorb", 256, 1, 4096, "rt"),
        # optical depths of a large ragged batch of free rays through a production-sized field
        _trans("rays_det_130k", "octave", 100_000, 4, 130_001, "det"),
        # interactive preview while a camera moves: few pixels, one sample, a coarse level of detail
        _render("preview_120x67", 50_000, 4, 120, 67, 1, 1, "cutoff", 1),
        # the single-scattering benchmark at full detail
        _render("single_512_16spp", 100_000, 4, 512, 512, 16, 1),
        # the multiple-scattering benchmark: per-bounce stochastic masks, one 8-sample launch
        _render("multi_1024_8spp", 1_000_000, 6, 1024, 1024, 8, 8, "unif_cv", 7, "is"),
        # half-precision records, ragged image, the power-law and threshold mask strategies
        _render("multi_fp16_333x217", 200_000, 5, 333, 217, 4, 3, "pow_cv_acc", 7, "thresh_uniform",
                "fp16", beta=0.2, delta=0.4),
        # single scattering with analytic free flight (inversion of the optical-depth CDF)
        _render("cdf_160x120", 50_000, 4, 160, 120, 2, 1, flight="cdf"),
        # tomography reconstruction step at the differentiable benchmark's size
        _step("step_tomo_256_8spp", 200_000, 4, 256, 256, 8, 0, "tomo"),
        # appearance optimisation: single scattering, then three-bounce paths
        _step("step_single_128_2spp", 200_000, 4, 128, 128, 2, 1, "scatter"),
        _step("step_path_96x64_1spp", 200_000, 4, 96, 64, 1, 3, "scatter"),
        # a burst of mixed requests on two resident assets of a render server
        dict(name="serve_burst_12", kind="serve", n=50_000, n2=200_000, octaves=4, requests=12,
             res_lo=64, res_hi=256, spp_hi=16, bounces=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("trans", "trans", "render", "render", "render", "step", "step", "serve"))
    if kind == "trans":
        mode = rng.choice(("det", "det", "rt", "closed"))
        if rng.random() < 0.4:
            c = _trans("", "absorb", _log_int(rng, 64, 1024), 1, _log_int(rng, 512, 40_000), mode)
        else:
            c = _trans("", "octave", _log_int(rng, 2_000, 100_000), rng.choice((3, 4)),
                       _log_int(rng, 1_000, 130_000), mode)
            if rng.random() < 0.3:
                c["freq"], c["max_band"] = "cutoff", rng.randrange(0, 3)
        c["precision"] = rng.choice(("fp32", "fp32", "fp16", "bf16"))
    elif kind == "render":
        style = rng.choice(("single", "single", "multi", "multi", "tomo", "cdf"))
        n, octaves = _log_int(rng, 10_000, 400_000), rng.choice((4, 5, 6))
        if style == "cdf":
            c = _render("", min(n, 60_000), 4, _log_int(rng, 40, 170), _log_int(rng, 30, 125), 1, 1,
                        flight=style)
        else:
            w = _log_int(rng, 48, 512)
            c = _render("", n, octaves, w, max(16, int(w * rng.uniform(0.5, 1.0))),
                        rng.choice((1, 2, 4, 8)), rng.choice((2, 3, 5, 8)) if style == "multi" else 1,
                        integrator="tomo" if style == "tomo" else "scatter")
            if style == "multi":
                c["freq"] = rng.choice(("unif_cv", "uniform", "pow_cv", "pow_cv_acc"))
                c["cone"] = rng.choice(("all", "is", "uniform", "thresh_uniform"))
                c["beta"] = round(rng.uniform(0.0, 0.4), 3)
            elif rng.random() < 0.5:
                c["freq"], c["max_band"] = "cutoff", rng.randrange(0, octaves)
            c["precision"] = rng.choice(("fp32", "fp32", "fp16", "bf16"))
    elif kind == "step":
        style = rng.choice(("tomo", "single", "path"))
        n = _log_int(rng, 20_000, 200_000)
        if style == "tomo":
            w = _log_int(rng, 32, 250)
            c = _step("", n, 4, w, max(16, int(w * rng.uniform(0.5, 1.0))), rng.choice((1, 2, 4)), 0, "tomo")
        elif style == "single":
            w = _log_int(rng, 32, 128)
            c = _step("", n, 4, w, max(16, int(w * rng.uniform(0.5, 1.0))), rng.choice((1, 2)), 1, "scatter")
        else:
            w = _log_int(rng, 24, 90)
            c = _step("", n, 4, w, max(16, int(w * rng.uniform(0.5, 1.0))), 1, rng.choice((2, 3)), "scatter")
    else:
        c = dict(kind="serve", n=_log_int(rng, 20_000, 100_000), n2=_log_int(rng, 50_000, 300_000),
                 octaves=4, requests=rng.randrange(3, 16), res_lo=64, res_hi=rng.choice((150, 256)),
                 spp_hi=rng.choice((4, 16)), bounces=rng.choice((1, 2)))
    c.pop("name", None)
    return c


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uniform(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device="cuda")


def _unit(g, n, k):
    v = torch.randn(n, k, generator=g, device="cuda")
    return v / v.norm(dim=1, keepdim=True)


def _octave_counts(n, octaves):
    total = sum(4 ** o for o in range(octaves))
    counts = [n // total * 4 ** o for o in range(octaves)]
    counts[-1] += n - sum(counts)
    return counts


def _absorb_params(n, g):
    f = torch.pow(9.0, torch.rand(n, generator=g, device="cuda")) - 1.0
    return {"mu": _uniform(g, 0.0, 1.0, n, 3), "quat": _unit(g, n, 4),
            "log_scale": _uniform(g, math.log(S_LO), math.log(S_HI), n, 3),
            "omega": _unit(g, n, 3) * (TWO_PI * f)[:, None], "phase": _uniform(g, 0.0, TWO_PI, n),
            "weight": _uniform(g, 0.5, 2.0, n), "band": None, "omega_frame": "world",
            "weight_mode": "peak"}


def _octave_params(n, octaves, g):
    counts = _octave_counts(n, octaves)
    band = torch.cat([torch.full((c,), o, dtype=torch.uint8, device="cuda")
                      for o, c in enumerate(counts)])
    b = band.float()
    # the Gaussian band has a mean optical depth of 4 per unit path
    c_rho = 4.0 / (counts[0] * 1.25 * TWO_PI ** 1.5 * MEAN_S ** 3)
    w = _uniform(g, 0.7, 1.5, n) * (band > 0)
    return {"mu": _uniform(g, 0.0, 1.0, n, 3), "quat": _unit(g, n, 4),
            "log_scale": _uniform(g, math.log(S_LO), math.log(S_HI), n, 3) - math.log(2.0) * b[:, None],
            "omega": w[:, None].expand(n, 3).contiguous(),
            "phase": _uniform(g, 0.0, TWO_PI, n) * (band > 0), "weight": c_rho * _uniform(g, 0.5, 2.0, n),
            "band": band, "omega_frame": "local", "weight_mode": "peak"}


def _params(case, g, n=None):
    if case.get("field") == "absorb":
        return _absorb_params(case["n"], g)
    return _octave_params(n or case["n"], case["octaves"], g)


def _rays(case, g):
    n = case["rays"]
    if case["field"] == "absorb":
        # a parallel detector: rays along +z through a grid over the unit square
        side = math.ceil(math.sqrt(n))
        i = (torch.arange(side, device="cuda") + 0.5) / side
        y, x = torch.meshgrid(i, i, indexing="ij")
        o = torch.stack([x.reshape(-1)[:n], y.reshape(-1)[:n], torch.full((n,), -0.5, device="cuda")], 1)
        d = torch.tensor([0.0, 0.0, 1.0], device="cuda").expand(n, 3).contiguous()
        far = 2.0
    else:
        # from a sphere around the cube, aimed at random points inside it
        o = 0.5 + 1.5 * _unit(g, n, 3)
        d = _uniform(g, 0.0, 1.0, n, 3) - o
        far = 3.0
    return o.contiguous(), d.contiguous(), torch.tensor([0.0, far], device="cuda").expand(n, 2).contiguous()


def _lod(case):
    return api.lod(case["freq"], case["max_band"], case.get("cone", "all"),
                   case.get("beta", 0.0), case.get("delta", 0.5))


def _camera(w, h, eye=EYE):
    return api.camera(eye, LOOK_AT, UP, VFOV, w, h)


def prepare(case, seed):
    ctx, g = _context(), _gen(seed)
    kind = case["kind"]
    if kind == "step":
        p = _params(case, g)
        w, h = case["width"], case["height"]
        scale = 1.0 if case["integrator"] == "tomo" else 0.1
        return {"kind": kind, "case": case, "ctx": ctx, "seed": seed, "cam": _camera(w, h),
                "leaves": [p[k].requires_grad_(True) for k in KEYS],
                "target": _uniform(g, 0.0, scale, h, w)}
    if kind == "serve":
        fields = [api.Field(ctx, _params(case, g, case[k])) for k in ("n", "n2")]
        cpu = torch.Generator().manual_seed(int(seed))
        reqs = []
        for k in range(case["requests"]):
            u = torch.rand(3, generator=cpu).tolist()
            e = torch.randn(3, generator=cpu)
            eye = (0.5 + 1.5 * e / e.norm()).tolist()
            # resolutions and sample counts of the burst: spread over their logarithms
            res = int(case["res_lo"] * (case["res_hi"] / case["res_lo"]) ** (0.618 * (k + 1) % 1.0))
            spp = max(1, int(case["spp_hi"] ** (0.414 * (k + 1) % 1.0)))
            lod = api.lod("cutoff", int(4 * u[1]))
            reqs.append((int(2 * u[2]), _camera(res, res, eye),
                         api.render_opts("scatter", spp, case["bounces"]), lod, int(seed) * 100 + k,
                         torch.empty(res, res).pin_memory()))
        return {"kind": kind, "server": api.Server(ctx, fields, mem_budget=64 << 20), "reqs": reqs}
    f = api.Field(ctx, _params(case, g), precision=case["precision"])
    f.set_lod(_lod(case))
    if kind == "trans":
        return {"kind": kind, "field": f, "rays": _rays(case, g), "mode": case["mode"], "seed": seed}
    opts = api.render_opts(case["integrator"], case["spp"], max(1, case["bounces"]),
                           free_flight=case["flight"])
    return {"kind": kind, "field": f, "cam": _camera(case["width"], case["height"]), "opts": opts,
            "seed": seed}


def run(state):
    kind = state["kind"]
    if kind == "trans":
        T, tau = state["field"].transmittance(*state["rays"], mode=state["mode"], seed=state["seed"])
        return {"T": T} if tau is None else {"T": T, "tau": tau}
    if kind == "render":
        return {"image": state["field"].render(state["cam"], state["opts"], seed=state["seed"])}
    if kind == "serve":
        srv = state["server"]
        tickets = [srv.submit(a, cam, opts, lod, seed=s, out=out)[0]
                   for a, cam, opts, lod, s, out in state["reqs"]]
        for t in tickets:
            srv.wait(t)
        return {"images": [r[-1] for r in state["reqs"]]}
    c, leaves = state["case"], state["leaves"]
    if c["integrator"] == "tomo":
        img = api.TomoRender.apply(*leaves, state["ctx"], state["cam"], c["spp"], state["seed"],
                                   "local", "peak", K_SIGMA)
    else:
        img = api.RadianceRender.apply(*leaves, state["ctx"], state["cam"], c["spp"], state["seed"],
                                       state["seed"] + 1, api.lod(), api.lod(), "local", "peak",
                                       K_SIGMA, 0.8, (1.0, 1.0, -1.0), c["bounces"])
    loss = ((img - state["target"]) ** 2).sum()
    grads = torch.autograd.grad(loss, leaves)
    return {"image": img.detach(), **dict(zip(KEYS, grads))}


# --------------------------------------------------------------------------
# work: kernels crossed by a ray of unit length (a kernel of scales s is crossed
# with probability pi (k s)^2), a chord set-up of about 60 operations each, a
# quadrature of about 12 nodes of 10 operations where the chord is integrated
# --------------------------------------------------------------------------
def _crossed(case, n):
    if case.get("field") == "absorb":
        return n * math.pi * K_SIGMA ** 2 * MEAN_S2
    counts = _octave_counts(n, case["octaves"])
    bands = len(counts)
    if case.get("freq") == "cutoff":
        bands = min(bands, case["max_band"] + 1)
    elif case.get("freq", "all") != "all":
        bands = 2  # the Gaussians and one band of one or more cones
    return bands * counts[0] * math.pi * K_SIGMA ** 2 * MEAN_S2


def work(case):
    kind, n = case["kind"], case["n"]
    rec = 64 if case.get("precision", "fp32") == "fp32" else 32
    if kind == "trans":
        per = 60 if case["mode"] == "rt" else 180
        outs = 1 if case["mode"] == "rt" else 2
        return {"bytes": rec * n + case["rays"] * (32 + 4 * outs),
                "flops": case["rays"] * _crossed(case, n) * per}
    if kind == "serve":
        # log-uniform resolution and samples, both assets alike
        lo, hi, sp = case["res_lo"], case["res_hi"], case["spp_hi"]
        pix = case["requests"] * (hi ** 2 - lo ** 2) / (2 * math.log(hi / lo))
        crossed = 0.5 * (_crossed(case, n) + _crossed(case, case["n2"]))
        return {"bytes": 64 * (n + case["n2"]) + 4 * pix,
                "flops": pix * (sp - 1) / math.log(sp) * 2 * 0.6 * crossed * 60}
    pix = case["width"] * case["height"]
    samples = pix * case["spp"]
    if kind == "render":
        rays = samples if case["integrator"] == "tomo" else 2 * samples
        per = 180 if case["integrator"] == "tomo" or case["flight"] != "delta" else 60
        return {"bytes": rec * n + 4 * pix, "flops": rays * _crossed(case, n) * per}
    # parameters in, gradients out; forward and adjoint passes over every ray
    rays = samples if case["integrator"] == "tomo" else 2 * samples
    per = 180 if case["integrator"] == "tomo" else 60
    return {"bytes": 2 * 60 * n + 12 * pix, "flops": 3 * rays * _crossed(case, n) * per}


# --------------------------------------------------------------------------
# 64-bit values: optical depths of deterministic masks, every kernel tried on
# every ray, chords by 96-node Gauss-Legendre; and the tomography step through
# torch's autograd over the same integral
# --------------------------------------------------------------------------
def _packed64(p, band_max):
    """Per kernel: mean, whitening matrix S^-1 R^T, whitened carrier, phase, amplitude."""
    q = p["quat"].double()
    q = q / q.norm(dim=1, keepdim=True)
    w, x, y, z = q.unbind(1)
    R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                     2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                     2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    s = p["log_scale"].double().exp()
    W = R.transpose(1, 2) / s[:, :, None]
    om = p["omega"].double()
    kw = om if p["omega_frame"] == "local" else s * (R.transpose(1, 2) @ om[:, :, None])[..., 0]
    A = p["weight"].double()
    if p["band"] is not None:
        A = torch.where(p["band"] <= band_max, A, torch.zeros_like(A))
    return p["mu"].double(), W, kw, p["phase"].double(), A


_GL = None


def _gl():
    global _GL
    if _GL is None:
        import numpy as np
        _GL = tuple(torch.from_numpy(a).cuda() for a in np.polynomial.legendre.leggauss(96))
    return _GL


def _pairs(P, o, v, tmin, tmax, budget=24_000_000):
    """(ray, kernel) pairs whose chords are not empty, a slice of rays at a time."""
    mu, W, _, _, A = P
    live = torch.nonzero(A)[:, 0]
    B = torch.einsum("nij,nik->njk", W[live], W[live])
    Bm, c = torch.einsum("njk,nk->nj", B, mu[live]), torch.einsum("nj,njk,nk->n", mu[live], B, mu[live])
    iu = [(0, 0, 1), (0, 1, 2), (0, 2, 2), (1, 1, 1), (1, 2, 2), (2, 2, 1)]
    Bs = torch.stack([f * B[:, i, j] for i, j, f in iu], 1)
    step = max(1, budget // max(1, live.numel()))
    for r0 in range(0, o.shape[0], step):
        oo, vv = o[r0:r0 + step], v[r0:r0 + step]
        sq = lambda a, b: torch.stack([a[:, i] * b[:, j] * 0.5 + a[:, j] * b[:, i] * 0.5 for i, j, _ in iu], 1)  # noqa: E731
        a = sq(vv, vv) @ Bs.T
        b = sq(oo, vv) @ Bs.T - vv @ Bm.T
        g = sq(oo, oo) @ Bs.T - 2 * oo @ Bm.T + c
        disc = b * b - a * (g - K_SIGMA ** 2)
        hw = disc.clamp(min=0).sqrt()
        near = (disc > 0) & (-b - hw < a * tmax) & (-b + hw > a * tmin)
        r, j = torch.nonzero(near, as_tuple=True)
        yield r0, min(step, o.shape[0] - r0), r, live[j]


def _chord_integrals(P, o, v, tmin, tmax):
    """Chord integrals of (ray, kernel) pairs given as gathered rows."""
    mu, W, kw, phi, A = P
    u = (W @ v[:, :, None])[..., 0]
    p = (W @ (o - mu)[:, :, None])[..., 0]
    a = (u * u).sum(1)
    ts = -(u * p).sum(1) / a
    d = p + ts[:, None] * u
    disc = K_SIGMA ** 2 - (d * d).sum(1)
    hw = (disc.clamp(min=1e-300) / a).sqrt()
    t0, t1 = (ts - hw).clamp(min=tmin), (ts + hw).clamp(max=tmax)
    x, wt = _gl()
    half = 0.5 * (t1 - t0)
    s = (0.5 * (t0 + t1) - ts)[:, None] + half[:, None] * x
    B, th = (kw * u).sum(1), (kw * d).sum(1) + phi
    f = torch.exp(-0.5 * ((d * d).sum(1)[:, None] + a[:, None] * s * s)) * torch.cos(B[:, None] * s + th[:, None])
    return torch.where((disc > 0) & (t1 > t0), A * half * (f @ wt), torch.zeros_like(A))


def _philox_camera(seed, pix, sample):
    """First two words of the Philox4x32-10 block of a sample's camera stream."""
    M = 0xFFFFFFFF
    c = [torch.zeros_like(pix), torch.full_like(pix, M), pix, torch.full_like(pix, (sample << 12) | 1)]
    k0, k1 = seed & M, (seed >> 32) & M

    def mul(m, x):  # high and low words of a 32 x 32 bit product
        lo = (x & 0xFFFF) * m
        hi = (x >> 16) * m + (lo >> 16)
        return (hi >> 16) & M, ((hi & 0xFFFF) << 16 | (lo & 0xFFFF)) & M

    for r in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return [(w >> 8).double() / 16777216.0 for w in c[:2]]


def _camera_rays(w, h, seed, sample):
    pix = torch.arange(w * h, device="cuda")
    jx, jy = _philox_camera(seed, pix, sample)
    tan = math.tan(0.5 * math.radians(VFOV))
    sx = (2 * ((pix % w) + jx) / w - 1) * tan * w / h
    sy = (1 - 2 * (torch.div(pix, w, rounding_mode="floor") + jy) / h) * tan
    # the camera looks along +z with +y up, so its right-hand axis is up x forward = +x
    d = torch.stack([sx, sy, torch.ones_like(sx)], 1)
    return torch.tensor(EYE, device="cuda").double().expand(w * h, 3), d / d.norm(dim=1, keepdim=True)


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    g = _gen(seed)
    if kind == "trans" and case["mode"] != "rt":
        if case["rays"] * n > 2.0e10:
            return None
        p = _params(case, g)
        o, d, tr = (t.double() for t in _rays(case, g))
        v = (d / d.norm(dim=1, keepdim=True)).float().double()  # rays run along the rounded direction
        P = _packed64(p, case["max_band"] if case["freq"] == "cutoff" else 7)
        tau = torch.zeros(case["rays"], dtype=torch.float64, device="cuda")
        for r0, m, r, j in _pairs(P, o, v, float(tr[0, 0]), float(tr[0, 1])):
            for k in range(0, r.numel(), 1 << 20):
                rr, jj = r[k:k + (1 << 20)] + r0, j[k:k + (1 << 20)]
                tau.index_add_(0, rr, _chord_integrals([t[jj] for t in P], o[rr], v[rr],
                                                       float(tr[0, 0]), float(tr[0, 1])))
        return {"T": torch.exp(-tau), "tau": tau}
    if case.get("integrator") != "tomo":
        return None  # Monte Carlo estimates: defined by their random streams
    w, h, spp = case["width"], case["height"], case["spp"]
    if w * h * spp * n > 6.0e9 or (kind == "render" and case["freq"] not in ("all", "cutoff")):
        return None
    p = _params(case, g)
    step = kind == "step"
    leaves = [p[k].detach().double().requires_grad_(step) for k in KEYS]
    P = _packed64({**p, **dict(zip(KEYS, leaves))},
                  case["max_band"] if case.get("freq") == "cutoff" else 7)
    D = [t.detach().requires_grad_(step) for t in P]
    img = torch.zeros(w * h, dtype=torch.float64, device="cuda")
    taus = []
    for s in range(spp):
        o, v = _camera_rays(w, h, int(seed), s)
        tau = torch.zeros(w * h, dtype=torch.float64, device="cuda")
        with torch.no_grad():
            for r0, m, r, j in _pairs(D, o, v, 0.0, math.inf):
                for k in range(0, r.numel(), 1 << 20):
                    rr, jj = r[k:k + (1 << 20)] + r0, j[k:k + (1 << 20)]
                    tau.index_add_(0, rr, _chord_integrals([t[jj] for t in D], o[rr], v[rr], 0.0, math.inf))
        taus.append(tau)
        img += torch.exp(-tau) / spp
    if not step:
        return {"image": img.view(h, w)}
    target = _uniform(g, 0.0, 1.0, h, w).double()
    dI = 2 * (img - target.view(-1))
    for s in range(spp):
        o, v = _camera_rays(w, h, int(seed), s)
        up = -dI * torch.exp(-taus[s]) / spp
        for r0, m, r, j in _pairs([t.detach() for t in D], o, v, 0.0, math.inf):
            for k in range(0, r.numel(), 1 << 18):
                rr, jj = r[k:k + (1 << 18)] + r0, j[k:k + (1 << 18)]
                (_chord_integrals([t[jj] for t in D], o[rr], v[rr], 0.0, math.inf) * up[rr]).sum().backward()
    torch.autograd.backward(P, [t.grad if t.grad is not None else torch.zeros_like(t) for t in D])
    return {"image": img.view(h, w), **{k: t.grad for k, t in zip(KEYS, leaves)}}
