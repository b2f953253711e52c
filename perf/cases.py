"""The calls that programs make of this package, as cases to time.

Every case goes through the public entry points (api, splat) the way the
README's examples do, with the library's default launch shapes. Kinds:

  roots     api.roots_batched: roots and status of a uniform-degree batch
  density   api.roots_density: roots binned into a fresh 1920 x 1080 image
  uneven    api.roots_uneven: a packed batch of degrees 2..12, roots, status and image
  grad      api.roots, a loss on the roots, and the adjoint through autograd
  loss      the soft-density loss step: roots, splat, splat pull-back, adjoint
  l2        api.l2_approx: least-squares fits from samples on sub-disks
  pipeline  api.l2_approx, then api.roots_density with the own-tile clip
  field     api.field_density: the whole path for sin(z^3) + z/2 in one launch

The three views of the plane (pipeline, field, l2) pan and zoom with the seed,
as a user who moves through the plane does.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2507_02164_gb300 import api, splat

DEV = "cuda"
W, H = 1920, 1080
DTYPES = {"c64": torch.complex64, "c128": torch.complex128}
NR, NT = 16, 32  # the quadrature of the full pipeline: 16 radii x 32 angles


def listed():
    return [
        # an interactive tool that asks for a few hundred polynomials' roots: the smallest call
        dict(name="roots_few_c128", kind="roots", degree=6, n=771, dtype="c128", mode="mixed", polish="fp64", inputs="gauss"),
        # the small plain-FP64 configuration: 65,536 polynomials expanded from roots in the unit disk
        dict(name="density_plain_disk", kind="density", degree=6, n=65536, dtype="c128", mode="plain", polish="fp64",
             inputs="disk", half_width=1.5),
        # the headline: 2^26 Littlewood-type polynomials into one image; the largest call
        dict(name="density_littlewood", kind="density", degree=6, n=1 << 26, dtype="c64", mode="mixed", polish="fp64",
             inputs="littlewood", half_width=2.0),
        # a ragged batch of middling degree with the FP32-pipe polish
        dict(name="roots_deg8_df", kind="roots", degree=8, n=300007, dtype="c64", mode="mixed", polish="df", inputs="gauss"),
        # the largest degree, complex128 storage, a ragged batch
        dict(name="roots_deg12_c128", kind="roots", degree=12, n=100003, dtype="c128", mode="mixed", polish="fp64",
             inputs="gauss"),
        # a small packed batch of mixed degrees, where the number of launches counts
        dict(name="uneven_few_c128", kind="uneven", n=3001, dtype="c128", mode="mixed", polish="fp64"),
        # the batching configuration: mixed degrees, complex64 storage, image and roots
        dict(name="uneven_many_c64", kind="uneven", n=(1 << 22) + 5, dtype="c64", mode="mixed", polish="fp64"),
        # a training step on the roots of 2^20 complex64 polynomials: forward and adjoint
        dict(name="grad_c64", kind="grad", degree=6, n=1 << 20, dtype="c64"),
        # the differentiation configuration's loss step in double precision: solve, splat, both pull-backs
        dict(name="loss_c128", kind="loss", degree=6, n=1 << 20, dtype="c128", sigma=1.5, width=256, height=144),
        # fits from samples alone, double-precision sums, a ragged number of sub-disks
        dict(name="l2_fp64", kind="l2", degree=6, n=50021, nr=16, precision="fp64"),
        # the full pipeline from samples of sin(z^3) + z/2 on 480 x 270 sub-disks
        dict(name="pipeline_480x270", kind="pipeline", nx=480, ny=270),
        # the same view in one launch, f evaluated in the kernel
        dict(name="field_480x270", kind="field", nx=480, ny=270),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["roots", "roots", "density", "density", "uneven", "grad", "loss", "l2", "pipeline", "field"])
    dtype = rng.choice(["c64", "c128"])
    if kind in ("roots", "density"):
        mode = rng.choice(["mixed", "mixed", "mixed", "plain"])
        degree = rng.randint(1, 12)
        # plain FP64 sweeps cost about 12 times the mixed ones, and the work grows about as degree^2.5
        top = (1 << 23) * min(1.0, (6.0 / degree) ** 2.5) / (12 if mode == "plain" else 1)
        c = dict(kind=kind, degree=degree, n=_log_int(rng, 200, top), dtype=dtype, mode=mode,
                 polish=rng.choice(["fp64", "fp64", "df"]) if mode == "mixed" else "fp64", inputs="gauss")
        if kind == "density":
            c.update(half_width=round(rng.uniform(1.5, 3.0), 3))
        return c
    if kind == "uneven":
        return dict(kind=kind, n=_log_int(rng, 1000, 1 << 22), dtype=dtype, mode="mixed",
                    polish=rng.choice(["fp64", "fp64", "df"]))
    if kind == "grad":
        degree = rng.randint(2, 12)
        return dict(kind=kind, degree=degree, n=_log_int(rng, 1000, (1 << 20) * min(1.0, (6.0 / degree) ** 2)), dtype=dtype)
    if kind == "loss":
        width = rng.randint(96, 400)
        return dict(kind=kind, degree=rng.randint(3, 8), n=_log_int(rng, 1000, 1 << 19), dtype=dtype,
                    sigma=round(rng.uniform(0.6, 2.0), 3), width=width, height=int(width * 9 / 16))
    if kind == "l2":
        return dict(kind=kind, degree=rng.randint(2, 12), n=_log_int(rng, 500, 60000), nr=rng.randint(6, 24),
                    precision=rng.choice(["fp64", "df"]))
    nx = _log_int(rng, 40, 480)
    return dict(kind=kind, nx=nx, ny=max(8, int(nx * 9 / 16)))


# ---- inputs -----------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _gauss(g, shape, dtype):
    real = torch.float32 if dtype == torch.complex64 else torch.float64
    return torch.complex(torch.randn(shape, generator=g, device=DEV, dtype=real),
                         torch.randn(shape, generator=g, device=DEV, dtype=real))


def _coeffs(case, seed):
    """Coefficient-major [degree + 1, n]."""
    g, d, n, dtype = _gen(seed), case["degree"], case["n"], DTYPES[case["dtype"]]
    inputs = case.get("inputs", "gauss")
    if inputs == "littlewood":  # every coefficient one of 1, -1, i, -i
        table = torch.tensor([1, -1, 1j, -1j], dtype=dtype, device=DEV)
        out = torch.empty((d + 1, n), dtype=dtype, device=DEV)
        for k in range(d + 1):
            out[k] = table[torch.randint(0, 4, (n,), generator=g, device=DEV)]
        return out
    if inputs == "disk":  # monic, from roots uniform in the unit disk
        r = torch.sqrt(torch.rand((d, n), generator=g, device=DEV, dtype=torch.float64))
        z = torch.polar(r, 2.0 * math.pi * torch.rand((d, n), generator=g, device=DEV, dtype=torch.float64))
        c = torch.zeros((d + 1, n), dtype=torch.complex128, device=DEV)
        c[0] = 1.0
        for k in range(d):
            up = torch.zeros_like(c)
            up[1:] = c[:-1]
            c = up - z[k] * c
        return c.to(dtype)
    return _gauss(g, (d + 1, n), dtype)


def _packed(case, seed):
    g, n = _gen(seed), case["n"]
    # degrees 2..12 in equal shares, in random order
    degrees = 2 + torch.randperm(n, generator=g, device=DEV) % 11
    offsets = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(degrees + 1, dim=0, out=offsets[1:])
    return _gauss(g, (int(offsets[-1]),), DTYPES[case["dtype"]]), degrees.to(torch.uint8), offsets


def _view(seed):
    """A 16:9 view of the plane: the whole region or part of it, panned."""
    u = torch.rand(3, generator=torch.Generator().manual_seed(int(seed)), dtype=torch.float64).tolist()
    half = 4.0 * (0.4 + 0.6 * u[0])
    cx, cy = 0.8 * (u[1] - 0.5), 0.5 * (u[2] - 0.5)
    return api.Window(cx - half, cx + half, cy - half * 9 / 16, cy + half * 9 / 16)


def _centres(view, nx, ny):
    w, h = (view.xmax - view.xmin) / nx, (view.ymax - view.ymin) / ny
    x = view.xmin + (torch.arange(nx, device=DEV, dtype=torch.float64) + 0.5) * w
    y = view.ymax - (torch.arange(ny, device=DEV, dtype=torch.float64) + 0.5) * h
    return torch.complex(x[None, :].expand(ny, nx), y[:, None].expand(ny, nx)).reshape(-1).contiguous(), 0.5 * math.hypot(w, h)


def _sample(centres, radius, points):
    out = torch.empty((centres.numel(), points.numel()), dtype=torch.complex128, device=DEV)
    for s in range(0, centres.numel(), 16384):
        z = centres[s:s + 16384, None] + radius * points[None, :]
        out[s:s + 16384] = torch.sin(z * z * z) + 0.5 * z
    return out


def _radii(nr):
    """Gauss-Legendre radii and weights on [0, 1]."""
    x, w = np.polynomial.legendre.leggauss(nr)
    return 0.5 * (x + 1.0), 0.5 * w


def _points(nr):
    r = torch.from_numpy(_radii(nr)[0]).to(DEV)
    return torch.polar(r[:, None].expand(nr, NT), (2.0 * math.pi / NT) * torch.arange(NT, device=DEV, dtype=torch.float64)
                       .expand(nr, NT)).reshape(-1)


def _l2_inputs(case, seed):
    nx = int(math.sqrt(case["n"] * 16 / 9)) + 1
    centres, radius = _centres(_view(seed), nx, -(-case["n"] // nx))
    return _sample(centres[:case["n"]], radius, _points(case["nr"]))


# ---- a case's state, one pass, and its work ------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": case}
    if kind in ("roots", "density", "grad", "loss"):
        s["coeffs"] = _coeffs(case, seed)
    if kind in ("roots", "density", "uneven"):
        s["params"] = api.params(case["mode"], **({"polish_mode": case["polish"]} if case["mode"] == "mixed" else {}))
    if kind == "density":
        hw = case["half_width"]
        s["window"] = api.Window(-hw, hw, -hw * 9 / 16, hw * 9 / 16)
        s["hist"], s["stats"] = api.new_hist(W, H, DEV), api.new_stats(DEV)
    if kind == "uneven":
        s["coeffs"], s["degrees"], s["offsets"] = _packed(case, seed)
        s["workspace"] = api.new_uneven_workspace(case["n"], s["coeffs"].numel(), s["coeffs"].dtype, DEV)
        s["window"], s["hist"] = api.Window(-3.0, 3.0, -1.6875, 1.6875), api.new_hist(W, H, DEV)
    if kind in ("grad", "loss"):
        s["coeffs"].requires_grad_(True)
    if kind == "loss":
        s["target"] = 2e-5 * torch.rand((case["height"], case["width"]), generator=_gen(seed + 1), device=DEV,
                                        dtype=torch.float64)
    if kind == "l2":
        s["samples"] = _l2_inputs(case, seed)
    if kind in ("pipeline", "field"):
        s["view"], s["hist"] = _view(seed), api.new_hist(W, H, DEV)
        s["status"] = torch.empty(case["nx"] * case["ny"], dtype=torch.uint8, device=DEV)
    if kind == "pipeline":
        s["centres"], s["radius"] = _centres(s["view"], case["nx"], case["ny"])
        s["samples"] = _sample(s["centres"], s["radius"], _points(NR))
        s["clip"] = api.make_clip(s["centres"], s["radius"], case["nx"], case["ny"], s["view"])
    if kind == "field":
        s["spec"] = api.field_spec(s["view"], case["nx"], case["ny"])
        s["coeffs"] = torch.empty((7, case["nx"] * case["ny"]), dtype=torch.complex128, device=DEV)
    return s


def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "roots":
        roots, status = api.roots_batched(s["coeffs"], mode=case["mode"], params_=s["params"])
        return {"roots": roots, "status": status}
    if kind == "density":
        api.hist_clear(s["hist"])
        api.hist_clear(s["stats"])
        api.roots_density(s["coeffs"], s["window"], s["hist"], mode=case["mode"], params_=s["params"], stats=s["stats"])
        return {"hist": s["hist"], "stats": s["stats"]}
    if kind == "uneven":
        api.hist_clear(s["hist"])
        roots, status = api.roots_uneven(s["coeffs"], s["degrees"], s["offsets"], s["workspace"], mode=case["mode"],
                                         params_=s["params"], window=s["window"], hist=s["hist"])
        return {"roots": roots, "status": status, "hist": s["hist"]}
    if kind == "grad":
        s["coeffs"].grad = None
        z, status = api.roots(s["coeffs"], "mixed")
        z.backward(2.0 * z.detach())  # the loss is the sum of |z|^2
        return {"roots": z.detach(), "status": status, "grad": s["coeffs"].grad}
    if kind == "loss":
        s["coeffs"].grad = None
        z, _ = api.roots(s["coeffs"], "mixed")
        loss = splat.loss(z, s["target"], W=case["width"], H=case["height"], sigma=case["sigma"],
                          precision="fp64" if case["dtype"] == "c128" else "fp32")
        loss.backward()
        return {"loss": loss.detach(), "grad": s["coeffs"].grad}
    if kind == "l2":
        return {"coeffs": api.l2_approx(s["samples"], case["nr"], NT, case["degree"], precision=case["precision"])}
    api.hist_clear(s["hist"])
    if kind == "pipeline":
        c = api.l2_approx(s["samples"], NR, NT, 6, precision="df")
        api.roots_density(c, s["view"], s["hist"], mode="mixed", clip=s["clip"], status=s["status"])
        return {"coeffs": c, "hist": s["hist"], "status": s["status"]}
    api.field_density(s["spec"], s["view"], s["hist"], coeffs=s["coeffs"], status=s["status"])
    return {"coeffs": s["coeffs"], "hist": s["hist"], "status": s["status"]}


def _solve_flops(d, mode="mixed", polish="fp64"):
    """Flops of one polynomial of degree d: about 2.8 sweeps per eigenvalue of
    20 flops per rotated pair, 24 per rotation and 60 for the shift, then 3
    Newton steps and the residual of 8 d flops per root."""
    sweeps = sum(2.8 * (20 * (m * (m + 1) - 2) + 24 * (m - 1) + 60) for m in range(2, d + 1))
    newton = 0 if mode == "plain" else d * (8 * d + (3 * 66 * d if polish == "df" else 3 * 16 * d))
    return sweeps + newton


def work(case):
    kind = case["kind"]
    el = 8 if case.get("dtype") == "c64" else 16
    image = 4 * W * H
    if kind in ("roots", "density", "grad", "loss"):
        d, n = case["degree"], case["n"]
        solve = n * _solve_flops(d, case.get("mode", "mixed"), case.get("polish", "fp64"))
        cin, zout = n * (d + 1) * el, n * d * 16
        adjoint = n * d * (24 * d + 14)
        if kind == "roots":
            return {"bytes": cin + zout + n, "flops": solve}
        if kind == "density":
            return {"bytes": cin + image, "flops": solve}
        if kind == "grad":
            return {"bytes": 2 * cin + zout + n, "flops": solve + adjoint}
        stencil = math.pi * (3 * case["sigma"]) ** 2  # pixels that a root reaches: 4 flops each way
        return {"bytes": 2 * cin + 8 * case["width"] * case["height"], "flops": solve + adjoint + n * d * stencil * 8}
    if kind == "uneven":
        n = case["n"]
        solve = n * sum(_solve_flops(d, case["mode"], case["polish"]) for d in range(2, 13)) / 11
        return {"bytes": n * (8 * el + 7 * 16 + 1 + 8 + 1) + image, "flops": solve}
    if kind == "l2":
        return {"bytes": case["n"] * (case["nr"] * NT + case["degree"] + 1) * 16,
                "flops": case["n"] * case["nr"] * NT * 4 * (case["degree"] + 1)}
    n = case["nx"] * case["ny"]
    fit = n * NR * NT * 4 * 7
    if kind == "pipeline":
        return {"bytes": n * (NR * NT + 7) * 16 + n * 17 + image, "flops": fit + n * _solve_flops(6)}
    return {"bytes": n * 113 + image, "flops": fit + n * (_solve_flops(6) + NR * NT * 60)}


# ---- what the outputs are in 64 bits --------------------------------------------

def _aberth(c, iters=90):
    """All roots of every column of c ([d + 1, n], complex128) by the
    Ehrlich-Aberth iteration from a circle of the Fujiwara radius's scale."""
    d, n = c.shape[0] - 1, c.shape[1]
    radius = (c[0].abs() / c[d].abs()).pow(1.0 / d)
    angle = 2.0 * math.pi * (torch.arange(d, device=c.device, dtype=torch.float64) + 0.37) / d
    z = torch.polar(torch.ones_like(angle), angle)[:, None] * radius[None, :]

    def ratio(z):
        p, q = c[d].expand_as(z), torch.zeros_like(z)
        for k in range(d - 1, -1, -1):
            q = q * z + p
            p = p * z + c[k]
        return p / q

    for it in range(iters + 3):
        nw = ratio(z)
        if it < iters:
            s = torch.zeros_like(z)
            for j in range(d):
                diff = z - z[j]
                diff[j] = 1.0
                inv = 1.0 / diff
                inv[j] = 0.0
                s += inv
            nw = nw / (1.0 - nw * s)
        nw = torch.where(torch.isfinite(nw.real) & torch.isfinite(nw.imag), nw, torch.zeros_like(nw))
        z = z - nw
    return z


def _adjoint(c, z, gz):
    d = c.shape[0] - 1
    dp = torch.zeros_like(z)
    for k in range(d, 0, -1):
        dp = dp * z + k * c[k]
    u, zc = torch.conj(-1.0 / dp) * gz, torch.conj(z)
    out, pw = [], u
    for _ in range(d + 1):
        out.append(pw.sum(dim=0))
        pw = pw * zc
    return torch.stack(out)


def _splat_exact(z, case, target):
    """The soft-density loss of the roots z (flat) and its gradient on them."""
    wd, hg, sg = case["width"], case["height"], case["sigma"]
    xmin, xmax, ymin, ymax = splat.WINDOW
    px, py, norm = (xmax - xmin) / wd, (ymax - ymin) / hg, 1.0 / z.numel()
    u, v = (z.real - xmin) / px, (ymax - z.imag) / py
    x0, y0 = torch.ceil(u - 0.5 - 3.0 * sg).to(torch.int64), torch.ceil(v - 0.5 - 3.0 * sg).to(torch.int64)
    reach, cut = int(math.floor(6.0 * sg)) + 1, math.exp(-4.5)

    def stencil():
        for ky in range(reach):
            dv, iy = v - (y0 + ky) - 0.5, y0 + ky
            ev = torch.exp(-dv * dv / (2.0 * sg * sg))
            for kx in range(reach):
                du, ix = u - (x0 + kx) - 0.5, x0 + kx
                e = ev * torch.exp(-du * du / (2.0 * sg * sg))
                inside = (e > cut) & (ix >= 0) & (ix < wd) & (iy >= 0) & (iy < hg)
                yield du, dv, e, inside, torch.where(inside, iy * wd + ix, torch.zeros_like(ix))

    img = torch.zeros(wd * hg, dtype=torch.float64, device=z.device)
    for _, _, e, inside, at in stencil():
        img += torch.bincount(at, weights=torch.where(inside, norm * (e - cut), torch.zeros_like(e)), minlength=wd * hg)
    diff = img - target.reshape(-1)
    loss = (z.real ** 2 + z.imag ** 2).sum() + (diff * diff).sum()
    gu, gv = torch.zeros_like(u), torch.zeros_like(v)
    for du, dv, e, inside, at in stencil():
        t = torch.where(inside, 2.0 * diff[at] * e, torch.zeros_like(e))
        gu += t * du
        gv += t * dv
    k = -norm / (sg * sg)
    return loss, 2.0 * z + torch.complex(k * gu / px, -k * gv / py)


def _fit_exact(samples, nr, degree):
    """a_j = (j + 1) / pi <g, w^j>: Gauss-Legendre radii on [0, 1], 32 angles."""
    r, w = _radii(nr)
    th = 2.0 * math.pi * np.arange(NT) / NT
    m = np.empty((nr * NT, degree + 1), dtype=np.complex128)
    for j in range(degree + 1):
        m[:, j] = ((j + 1) / math.pi * (2.0 * math.pi / NT) * (w * r ** (j + 1))[:, None] * np.exp(-1j * j * th)[None, :]).reshape(-1)
    return (samples @ torch.from_numpy(m).to(samples.device)).T.contiguous()


def exact(case, seed):
    """What has one value in 64 bits: gradients, the loss, fitted
    coefficients. Roots come in no fixed order, images and codes are whole
    numbers: None."""
    kind = case["kind"]
    if kind == "grad":
        c = _coeffs(case, seed).to(torch.complex128)
        z = _aberth(c)
        return {"roots": None, "status": None, "grad": _adjoint(c, z, 2.0 * z)}
    if kind == "loss":
        c = _coeffs(case, seed).to(torch.complex128)
        target = 2e-5 * torch.rand((case["height"], case["width"]), generator=_gen(seed + 1), device=DEV, dtype=torch.float64)
        z = _aberth(c)
        loss, gz = _splat_exact(z.reshape(-1), case, target)
        return {"loss": loss, "grad": _adjoint(c, z, gz.reshape(z.shape))}
    if kind == "l2":
        return {"coeffs": _fit_exact(_l2_inputs(case, seed), case["nr"], case["degree"])}
    if kind in ("pipeline", "field"):
        centres, radius = _centres(_view(seed), case["nx"], case["ny"])
        points = _points(NR)
        c = torch.cat([_fit_exact(_sample(centres[s:s + 16384], radius, points), NR, 6)
                       for s in range(0, centres.numel(), 16384)], dim=1)
        return {"coeffs": c, "hist": None, "status": None}
    return None
