"""The work that programs have this framework do, as measurable cases.

Every case goes through the public entry points (``Plan``, ``Batch`` and the
differentiable ``autograd.degrid``) with the sizes of the repository's own
workloads (``synth.py``: tiny, survey, reduced cost, differentiable, batched)
or generic ones of the same kind.  A case is a dict of

  op      what a pass calls: "degrid", "grid", "pair" (one of each, as an
          iterative imager does), "gradient" (chi^2 and its gradient with
          respect to a real image) or "batch" (both directions of a ``Batch``)
  N, x0, W, fov           the plan (image side, crop, kernel width, field)
  track, ants, times, hours, flagged   earth-rotation tracks of a flat array:
          ants (ants - 1) / 2 baselines at `times` hour angles over `hours`
          hours, less `flagged` samples (flagged data make the counts ragged)
  M, w    instead of tracks: M points uniform in a (u, v) disc with w uniform
          in +- w R, R the disc's radius
  flags   names of the plan's options, joined by "+"
  sources point sources of the model image
"""
from __future__ import annotations

import math

import torch

from paper_2101_11172_gb300 import _lib, autograd
from paper_2101_11172_gb300.batch import Batch
from paper_2101_11172_gb300.wstack import Plan

FLAGS = {"async": _lib.WS_FLAG_ASYNC, "real_sky": _lib.WS_FLAG_HERMITIAN,
         "deterministic": _lib.WS_FLAG_DETERMINISTIC, "fp64": _lib.WS_FLAG_FP64}


def _case(name, op, N, W, fov, x0=0.25, flags="", sources=50, bound=False, M=0, w=0.0, ants=0, times=0, hours=8.0,
          flagged=0, instances=0):
    c = {"op": op, "N": N, "x0": x0, "W": W, "fov": fov, "flags": flags, "sources": sources, "bound": bound}
    if instances:
        c["instances"] = instances
    if ants:
        c.update(ants=ants, times=times, hours=hours, flagged=flagged)
    else:
        c.update(M=M, w=w)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # One short observation predicted from a model: the smallest call, where latency and launches count.
        _case("snapshot degrid", "degrid", 256, 7, 0.2, M=10_000, w=0.05),
        # A quick look at a field of an odd size with a narrower kernel, calls queued one behind the other.
        _case("odd snapshot grid", "grid", 200, 6, 0.3, flags="async", M=9_973, w=0.06),
        # A small map over a large w-range: hundreds of planes for few visibilities.
        _case("many planes", "pair", 256, 7, 0.2, M=10_000, w=12.8),
        # FP64 plans measure the method's own error (W up to 14): small maps, a wide kernel.
        _case("fp64 accuracy", "pair", 128, 12, 0.3, flags="fp64", M=4_001, w=1.0),
        # Reproducible dirty images for regression runs of an imaging pipeline.
        _case("reproducible grid", "grid", 512, 7, 0.4, flags="deterministic", ants=64, times=60, flagged=311),
        # A map size that is not a power of two (mixed-radix transforms), a wider kernel, flagged data.
        _case("ragged map", "pair", 1000, 8, 0.25, ants=90, times=30, hours=5.0, flagged=1_237),
        # chi^2 and its gradient in an optimisation over a real sky; its uvw is bound to the plan once.
        _case("imaging gradient", "gradient", 1024, 7, 0.5, ants=256, times=61, sources=200, bound=True),
        # Many fields or channels served at once.
        _case("served batch", "batch", 1024, 7, 0.5, instances=8, ants=128, times=40),
        # A real sky (w < 0 folded), an hour and a half of a survey.
        _case("real sky", "pair", 2048, 7, 0.5, flags="real_sky", ants=256, times=60, hours=6.0, sources=500),
        # The survey workload, each direction on its own: model prediction ...
        _case("survey degrid", "degrid", 2048, 7, 0.5, ants=256, times=306, sources=500),
        # ... and dirty imaging.
        _case("survey grid", "grid", 2048, 7, 0.5, ants=256, times=306, sources=500),
        # The reduced-cost setting: the largest images and visibility sets.
        _case("reduced cost", "pair", 4096, 5, 0.5, x0=0.375, ants=256, times=1532, hours=4.0, sources=500),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["snapshot", "planes", "tracks", "tracks", "tracks", "gradient", "real", "large", "fp64",
                       "deterministic", "batch"])
    fov = round(rng.uniform(0.2, 0.5), 3)
    W = rng.choice([4, 5, 6, 7, 7, 7, 8])
    x0 = rng.choice([0.25, 0.25, 0.25, 0.3, 0.375])
    sources = rng.randint(20, 500)
    op = rng.choice(["degrid", "grid", "pair"])
    if kind == "snapshot":
        return _case("", op, 8 * _log(rng, 8, 64), W, fov, x0, sources=20, M=_log(rng, 1_000, 60_000),
                     w=round(rng.uniform(0.02, 0.2), 3), flags=rng.choice(["", "async"]))
    if kind == "planes":
        return _case("", op, 8 * _log(rng, 16, 48), W, fov, sources=20, M=_log(rng, 4_000, 60_000),
                     w=round(rng.uniform(2.0, 10.0), 3))
    if kind == "fp64":
        return _case("", "pair", rng.choice([64, 128, 256]), rng.choice([8, 10, 12, 14]), fov, flags="fp64",
                     sources=20, M=_log(rng, 1_000, 8_000), w=round(rng.uniform(0.1, 1.0), 3))
    track = dict(hours=round(rng.uniform(1.0, 8.0), 2), sources=sources)
    flagged = rng.randint(0, 400)
    if kind == "deterministic":
        return _case("", "grid", 8 * _log(rng, 32, 192), W, fov, x0, flags="deterministic", ants=rng.randint(40, 160),
                     times=rng.randint(10, 80), flagged=flagged, **track)
    if kind == "gradient":
        return _case("", "gradient", rng.choice([512, 1000, 1024, 1536]), W, fov, bound=rng.choice([True, False]),
                     ants=rng.randint(64, 256), times=rng.randint(10, 61), flagged=flagged, **track)
    if kind == "batch":
        return _case("", "batch", rng.choice([512, 768, 1024]), W, fov, instances=rng.randint(2, 8),
                     ants=rng.randint(40, 128), times=rng.randint(10, 40), **track)
    if kind == "real":
        return _case("", op, 8 * _log(rng, 64, 256), W, fov, x0, flags="real_sky", ants=rng.randint(64, 256),
                     times=rng.randint(10, 100), flagged=flagged, **track)
    if kind == "large":
        return _case("", op, rng.choice([2048, 2304, 3000, 4096]), W if W < 8 else 5, fov, 0.375,
                     ants=rng.randint(128, 256), times=rng.randint(30, 400), flagged=flagged, **track)
    return _case("", op, 8 * _log(rng, 32, 256), W, fov, x0, flags=rng.choice(["", "async"]), ants=rng.randint(32, 256),
                 times=rng.randint(4, 300), flagged=flagged, **track)


# -- inputs --------------------------------------------------------------------


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(1_000_003 * int(seed) + 17)


def _uniform(n, lo, hi, g):
    return lo + (hi - lo) * torch.rand(n, dtype=torch.float64, device="cuda", generator=g)


def _uvw(case, g):
    """Wavelengths, the longest (u, v) at 0.45 N / fov."""
    R = 0.45 * case["N"] / case["fov"]
    if "M" in case:
        r, th = R * _uniform(case["M"], 0, 1, g).sqrt(), _uniform(case["M"], 0, 2 * math.pi, g)
        w = _uniform(case["M"], -case["w"] * R, case["w"] * R, g)
        return torch.stack([r * th.cos(), r * th.sin(), w], 1).contiguous()
    n = case["ants"]
    rad, th = _uniform(n, 0, 1, g).sqrt(), _uniform(n, 0, 2 * math.pi, g)
    east, north = rad * th.cos(), rad * th.sin()
    lat = dec = math.radians(-30.0)
    X, Y, Z = -north * math.sin(lat), east, north * math.cos(lat)
    i, j = torch.triu_indices(n, n, 1, device="cuda")
    Bx, By, Bz = (v[j] - v[i] for v in (X, Y, Z))
    H = torch.deg2rad(15.0 * torch.linspace(-case["hours"] / 2, case["hours"] / 2, case["times"], dtype=torch.float64,
                                            device="cuda"))[:, None]
    sH, cH = H.sin(), H.cos()
    u = sH * Bx + cH * By
    v = -math.sin(dec) * (cH * Bx - sH * By) + math.cos(dec) * Bz
    w = math.cos(dec) * (cH * Bx - sH * By) + math.sin(dec) * Bz
    uvw = torch.stack([u.reshape(-1), v.reshape(-1), w.reshape(-1)], 1)
    uvw *= R / (uvw[:, 0].square() + uvw[:, 1].square()).max().sqrt()
    return uvw[:uvw.shape[0] - case["flagged"]].contiguous()


def _sky(case, g):
    """Pixels (flat) and amplitudes of the model's point sources."""
    pix = torch.randperm(case["N"] ** 2, device="cuda", generator=g)[:case["sources"]]
    return pix, _uniform(case["sources"], 0.1, 1.0, g).float().double()


def _inputs(case, seed):
    g = _generator(seed)
    uvw = _uvw(case, g)
    pix, amp = _sky(case, g)
    M = uvw.shape[0]
    vis = torch.view_as_complex(torch.randn(M, 2, dtype=torch.float32, device="cuda", generator=g) * math.sqrt(0.5))
    return uvw, pix, amp, vis


def _image(case, pix, amp, dtype):
    image = torch.zeros(case["N"] ** 2, dtype=dtype, device="cuda")
    image[pix] = amp.to(dtype)
    return image.reshape(case["N"], case["N"])


def _flags(case):
    return sum(FLAGS[f] for f in case["flags"].split("+") if f)


def _instances(case):
    """The instances of a batch: the first of the case's size, the others smaller and shorter."""
    out = []
    for i in range(case["instances"]):
        one = {k: v for k, v in case.items() if k not in ("instances", "name")}
        one.update(N=case["N"] >> (i % 2), ants=max(16, case["ants"] - 9 * i), times=max(2, case["times"] - 3 * i),
                   flagged=7 * i)
        out.append(one)
    return out


def _plan(case, uvw):
    return Plan(case["N"], case["x0"], case["W"], case["fov"], float(uvw[:, 2].min()), float(uvw[:, 2].max()),
                flags=_flags(case))


def prepare(case, seed):
    if case["op"] == "batch":
        parts = [(one, *_inputs(one, 100 * seed + i)) for i, one in enumerate(_instances(case))]
        uvw = [p[1] for p in parts]
        batch = Batch([(one["N"], one["fov"], float(t[:, 2].min()), float(t[:, 2].max()), t.shape[0])
                       for (one, *_), t in zip(parts, uvw)], case["x0"], case["W"], branches=4)
        images = [_image(one, pix, amp, torch.complex64) for one, _, pix, amp, _ in parts]
        return {"op": "batch", "batch": batch, "uvw": uvw, "images": images, "vis": [p[4] for p in parts],
                "out_vis": [torch.empty_like(p[4]) for p in parts], "out_dirty": [torch.empty_like(i) for i in images]}
    uvw, pix, amp, vis = _inputs(case, seed)
    plan = _plan(case, uvw)
    if case["bound"]:
        plan.bind(uvw)
    if case["op"] == "gradient":
        image = _image(case, pix, amp, torch.float32).requires_grad_(True)
    else:
        image = _image(case, pix, amp, plan.cdtype)
    return {"op": case["op"], "plan": plan, "uvw": uvw, "image": image, "vis": vis.to(plan.cdtype)}


def run(state):
    op = state["op"]
    if op == "batch":
        vis = state["batch"].degrid(state["images"], state["uvw"], out=state["out_vis"])
        return [vis, state["batch"].grid(state["uvw"], state["vis"], out=state["out_dirty"])]
    plan, uvw = state["plan"], state["uvw"]
    if op == "gradient":
        model = autograd.degrid(plan, state["image"], uvw)
        r = torch.view_as_real(model - state["vis"])
        chi2 = r.square().sum(dtype=torch.float64)
        (grad,) = torch.autograd.grad(chi2, state["image"])
        return [model.detach(), chi2.detach(), grad]
    out = []
    if op in ("degrid", "pair"):
        out.append(plan.degrid(state["image"], uvw))
    if op in ("grid", "pair"):
        out.append(plan.grid(uvw, state["vis"]))
    return out


# -- work ----------------------------------------------------------------------


def _count(case):
    return case["M"] if "M" in case else case["ants"] * (case["ants"] - 1) // 2 * case["times"] - case["flagged"]


def _one_work(case):
    N, W, M, x0 = case["N"], case["W"], _count(case), case["x0"]
    R = 0.45 * N / case["fov"]
    w = case["w"] * R if "M" in case else 0.6 * R * math.sin(math.radians(15.0 * min(case["hours"], 8.0) / 2)) + 0.1 * R
    lm2 = case["fov"] ** 2 / 2
    dn = lm2 / (1 + math.sqrt(1 - lm2))
    span = w if "real_sky" in case["flags"] else 2 * w
    planes = int(dn * span / (2 * x0)) + W
    Np = N / (2 * x0)
    # per plane, transforms along one axis of the N image lines and along the other of the N' grid lines
    fft = planes * (N + Np) * 5 * Np * math.log2(Np)
    flops = fft + M * W ** 3 * 4 + planes * N * N * 8
    value = 16 if "fp64" in case["flags"] else 8
    return 24 * M + value * (M + N * N), flops


def work(case):
    parts = [_one_work(one) for one in (_instances(case) if case["op"] == "batch" else [case])]
    times = 2 if case["op"] in ("pair", "gradient", "batch") else 1
    return {"bytes": float(times * sum(p[0] for p in parts)), "flops": float(times * sum(p[1] for p in parts))}


# -- the same in 64 bits -------------------------------------------------------


def _lm(case):
    return (torch.arange(case["N"], dtype=torch.float64, device="cuda") - case["N"] // 2) * (case["fov"] / case["N"])


def _nm1(r2):
    return -r2 / (1 + (1 - r2).sqrt())


def _cis(turns):
    turns = turns - turns.round()
    return torch.polar(torch.ones_like(turns), 2 * math.pi * turns)


def _exact_degrid(case, uvw, pix, amp):
    """V_k = sum over the sources of f exp(-2 pi i (u l + v m + w (n - 1)))."""
    x, N = _lm(case), case["N"]
    l, m = x[pix % N], x[pix // N]
    lmn = torch.stack([l, m, _nm1(l * l + m * m)])
    f, step = amp.to(torch.complex128), max(1, (1 << 26) // len(pix))
    return torch.cat([_cis(-(uvw[k:k + step] @ lmn)) @ f for k in range(0, uvw.shape[0], step)])


def _exact_grid(case, uvw, vis):
    """D[i][j] = sum over k of V_k exp(+2 pi i (u l_j + v m_i + w (n_ij - 1)))."""
    x, N = _lm(case), case["N"]
    i = torch.arange(N, device="cuda") - N // 2
    r2, where = torch.unique(i[:, None] ** 2 + i[None, :] ** 2, return_inverse=True)   # n - 1 depends on l^2 + m^2 alone
    nm1 = _nm1(r2.double() * (case["fov"] / N) ** 2)
    out = torch.zeros(N, N, dtype=torch.complex128, device="cuda")
    step = max(1, (1 << 25) // (N * N))
    for k in range(0, uvw.shape[0], step):
        c = uvw[k:k + step]
        t = _cis(c[:, 2:] * nm1)[:, where]
        t *= _cis(c[:, :1] * x)[:, None, :]
        t *= (vis[k:k + step, None] * _cis(c[:, 1:2] * x))[:, :, None]
        out += t.sum(0)
    real = "real_sky" in case["flags"]
    return torch.complex(out.real, torch.zeros_like(out.real)) if real else out


def exact(case, seed):
    def both(one, s):
        uvw, pix, amp, vis = _inputs(one, s)
        vis = vis.to(torch.complex128)
        affordable = uvw.shape[0] * one["N"] ** 2 < 2e11
        model = _exact_degrid(one, uvw, pix, amp) if one["op"] != "grid" and uvw.shape[0] * one["sources"] < 3e10 else None
        return model, _exact_grid(one, uvw, vis) if one["op"] not in ("degrid", "gradient") and affordable else None, vis

    if case["op"] == "batch":
        some = [both(dict(one, op="degrid"), 100 * seed + i)[0] for i, one in enumerate(_instances(case))]
        return [some, [None] * len(some)]
    model, dirty, vis = both(case, seed)
    if case["op"] == "gradient":
        return [model, torch.view_as_real(model - vis).square().sum(), None]
    out = ([model] if case["op"] != "grid" else []) + ([dirty] if case["op"] != "degrid" else [])
    return None if all(v is None for v in out) else out
