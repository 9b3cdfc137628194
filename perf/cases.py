"""The work that a user of this framework has it do, as cases that can be timed and compared.

Every case goes through the public operators (``Radon``, ``RadonFanbeam``, ``Landweber``, ``cgne``,
``BatchPlan``) at sizes of the repository's own workloads and tests, or generic ones.  Images are
seeded sums of ellipses, sinograms their closed-form line integrals plus noise (what a scanner
measures), so no input depends on the projectors.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_2009_14788_gb300 import BatchPlan, Landweber, Radon, RadonFanbeam, cgne

DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}


def _case(name, op, **kw):
    c = dict(name=name, op=op, kind="parallel", n=0, views=0, det=0, batch=1, dtype="f32", spacing=1.0, step=1.0,
             source=0.0, detector=0.0, table=False, iterations=0, items="")
    c.update(kw)
    return c


def listed():
    fan = dict(kind="fan", n=512, views=720, det=1024, batch=16, spacing=1.5, source=1000.0, detector=500.0)
    return [
        # one small image there and back: the call a test or a notebook makes; launches and latency count
        _case("small_pair_b1_n64_f32", "pair", n=64, views=64, det=91),
        # the fan-beam batch of the headline workload, each direction by itself
        _case("fan_forward_b16_n512_f16", "forward", dtype="f16", **fan),
        _case("fan_adjoint_b16_n512_f16", "backprojection", dtype="f16", **fan),
        # the same backprojection by a program that keeps the geometry's weight table
        _case("fan_adjoint_table_b16_n512_bf16", "backprojection", dtype="bf16", table=True, **fan),
        # one least-squares training step through autograd on the FP32 batch workload
        _case("step_b32_n256_f32", "step", n=256, views=256, det=363, batch=32),
        # the paper's benchmark shape: a large half-precision batch projected and back-projected
        _case("paper_pair_b32_n512_f16", "pair", n=512, views=512, det=512, batch=32, dtype="f16"),
        # sparse-view unrolled reconstruction with gradients to its input (a whole call)
        _case("landweber_b8_n512_bf16", "landweber", n=512, views=60, det=725, batch=8, dtype="bf16", iterations=10),
        # filtered backprojection of one slice
        _case("fbp_b1_n512_f32", "fbp", n=512, views=512, det=725),
        # the start of a conjugate-gradient reconstruction of one slice (a whole call)
        _case("cgne_b1_n512_f32", "cgne", n=512, views=512, det=725, iterations=3),
        # images of mixed sizes, each with its own geometry, in one launch per direction
        _case("uneven_forward_f16", "plan_forward", dtype="f16",
              items="128:214,128:905,256:611,256:131,512:433,512:987,1024:344,1024:818"),
        _case("uneven_adjoint_f16", "plan_adjoint", dtype="f16",
              items="128:214,128:905,256:611,256:131,512:433,512:987,1024:344,1024:818"),
        # odd sizes that fill no tile, group or vector: a few fan-beam images in single precision
        _case("odd_fan_pair_b5_n243_f32", "pair", kind="fan", n=243, views=181, det=367, batch=5, spacing=1.3,
              source=420.0, detector=310.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["forward", "forward", "backprojection", "backprojection", "pair", "pair", "step", "landweber", "fbp",
                     "cgne", "plan_forward", "plan_adjoint"])
    dtype = rng.choice(["f32", "f16", "bf16"])
    if op in ("plan_forward", "plan_adjoint"):
        items = ["%d:%d" % (_log_int(rng, 48, 800), _log_int(rng, 60, 900)) for _ in range(rng.randint(2, 6))]
        c = _case("", op, dtype=dtype, items=",".join(items))
        del c["name"]
        return c
    n, views, batch = _log_int(rng, 48, 768), _log_int(rng, 24, 800), _log_int(rng, 1, 32)
    kw = dict(n=n, views=views, det=max(8, int(n * rng.uniform(0.9, 1.6))), batch=batch, dtype=dtype)
    kw["spacing"] = round(rng.uniform(0.9, 1.4), 3) if rng.random() < 0.5 else 1.0
    kw["step"] = 0.75 if rng.random() < 0.15 else 1.0
    if op not in ("fbp", "cgne", "landweber") and rng.random() < 0.5:
        s, d = round(n * rng.uniform(1.3, 2.5), 1), round(n * rng.uniform(0.5, 1.5), 1)
        kw.update(kind="fan", source=s, detector=d, spacing=round(kw["spacing"] * (s + d) / s, 3))
    if op in ("step", "cgne"):
        kw["dtype"] = "f32"
    if op == "landweber":
        kw["iterations"] = rng.randint(2, 6)
    if op == "cgne":
        kw["iterations"] = rng.randint(1, 3)
    if op == "backprojection" and kw["step"] == 1.0:
        kw["table"] = rng.random() < 0.3
    at = kw["spacing"] * (kw["source"] / (kw["source"] + kw["detector"]) if kw.get("kind") == "fan" else 1.0)
    passes = {"pair": 2, "step": 2}.get(op, 1) + 4 * kw.get("iterations", 0)
    while _samples(n, kw["det"], kw["views"], at, kw["step"]) * kw["batch"] * passes > 1.5e9:
        if kw["batch"] > 1:
            kw["batch"] = max(1, kw["batch"] * 2 // 3)
        else:
            kw["views"] = max(24, kw["views"] * 2 // 3)
    c = _case("", op, **kw)
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------- inputs


def _angles(views, kind):
    return np.arange(views) * ((2.0 if kind == "fan" else 1.0) * math.pi / views)


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _ellipses(n, batch, gen):
    """[batch, 10] ellipses inside the image's inscribed circle: centre, semi-axes, rotation, intensity
    (attenuation per pixel: line integrals of order one, so that 16-bit results stay in range)."""
    u = torch.rand((6, batch, 10), generator=gen, device="cuda", dtype=torch.float64)
    a, b = n * (0.0625 + 0.25 * u[0]), n * (0.0625 + 0.25 * u[1])
    r = (0.5 * n - 1.0 - torch.maximum(a, b)).clamp_min(0.0) * u[2].sqrt()
    t = 2.0 * math.pi * u[3]
    return r * t.cos(), r * t.sin(), a, b, math.pi * u[4], 2.0 / n * u[5]


def _image(n, e, dtype):
    cx, cy, a, b, rot, rho = (v[:, :, None, None] for v in e)
    p = torch.arange(n, device="cuda", dtype=torch.float64) - 0.5 * (n - 1)
    out = torch.zeros((cx.shape[0], n, n), device="cuda", dtype=torch.float64)
    for k in range(cx.shape[1]):
        x, y = p[None, None, :] - cx[:, k], p[None, :, None] - cy[:, k]
        c, s = rot[:, k].cos(), rot[:, k].sin()
        out += rho[:, k] * ((((c * x + s * y) / a[:, k]) ** 2 + ((c * y - s * x) / b[:, k]) ** 2) <= 1.0)
    return out.to(dtype)


def _lines(kind, views, det, spacing, source, detector):
    """Every ray as (foot point, direction), [V, D] each, in pixels about the rotation centre."""
    th = torch.from_numpy(_angles(views, kind)).cuda()[:, None]
    nx, ny, ux, uy = th.cos(), th.sin(), -th.sin(), th.cos()
    s = ((torch.arange(det, device="cuda", dtype=torch.float64) - 0.5 * (det - 1)) * spacing)[None, :]
    if kind == "parallel":
        one = torch.ones_like(s)
        return s * nx, s * ny, ux * one, uy * one
    ex, ey = (source + detector) * ux + s * nx, (source + detector) * uy + s * ny
    ln = torch.sqrt(ex * ex + ey * ey)
    ex, ey = ex / ln, ey / ln
    along = -source * (ux * ex + uy * ey)
    return -source * ux - along * ex, -source * uy - along * ey, ex, ey


def _measured(c, n, views, det, e, gen, dtype):
    """The ellipses' closed-form line integrals with noise of 0.1 % of the largest."""
    mx, my, ex, ey = _lines(c["kind"], views, det, c["spacing"], c["source"], c["detector"])
    cx, cy, a, b, rot, rho = (v[:, :, None, None] for v in e)
    y = torch.zeros((cx.shape[0],) + tuple(mx.shape), device="cuda", dtype=torch.float64)
    for k in range(cx.shape[1]):
        cs, sn = rot[:, k].cos(), rot[:, k].sin()
        px, py = mx - cx[:, k], my - cy[:, k]
        ox, oy = (cs * px + sn * py) / a[:, k], (cs * py - sn * px) / b[:, k]
        dx, dy = (cs * ex + sn * ey) / a[:, k], (cs * ey - sn * ex) / b[:, k]
        q = dx * dx + dy * dy
        disc = (q - (ox * dy - oy * dx) ** 2).clamp_min(0.0)
        y += 2.0 * rho[:, k] * disc.sqrt() / q
    y += 1e-3 * y.max() * torch.randn(y.shape, generator=gen, device="cuda", dtype=torch.float64)
    return y.to(dtype)


def _items(c):
    """(side, views, detectors) of a mixed batch's images."""
    out = []
    for t in c["items"].split(","):
        n, v = (int(q) for q in t.split(":"))
        out.append((n, v, int(math.ceil(n * math.sqrt(2.0)))))
    return out


def _data(c, seed):
    """The case's input tensors, in the order its run takes them."""
    gen, dtype = _gen(seed), DTYPES[c["dtype"]]
    n, v, d, op = c["n"], c["views"], c["det"], c["op"]
    if c["items"]:
        out = []
        for m, w, k in _items(c):
            e = _ellipses(m, 1, gen)
            out.append(_image(m, e, dtype) if op == "plan_forward" else _measured(c, m, w, k, e, gen, dtype))
        return out
    e = _ellipses(n, c["batch"], gen)
    if op in ("forward", "pair"):
        return [_image(n, e, dtype)]
    y = _measured(c, n, v, d, e, gen, dtype)
    if op in ("backprojection", "fbp"):
        return [y]
    if op == "step":   # a guess and the data of another image
        return [_image(n, _ellipses(n, c["batch"], gen), dtype), y]
    x0 = torch.zeros((c["batch"], n, n), device="cuda", dtype=dtype)
    if op == "landweber":   # and the gradient that the rest of a network sends back
        return [x0, y, torch.randn(x0.shape, generator=gen, device="cuda", dtype=torch.float64).to(dtype)]
    return [x0, y]


def _alpha(c):
    """A step below 1 / lambda_max: lambda_max of A^T A is close to views x side / (spacing) / step."""
    return float(np.float32(0.8 * c["spacing"] / (c["views"] * c["n"])))


def _operator(c, n, v, d):
    ang = _angles(v, c["kind"])
    if c["kind"] == "fan":
        return RadonFanbeam(n, ang, c["source"], det_distance=c["detector"], det_count=d, det_spacing=c["spacing"],
                            step=c["step"])
    return Radon(n, ang, det_count=d, det_spacing=c["spacing"], step=c["step"])


def prepare(case, seed):
    c = dict(case)
    data = _data(c, seed)
    s = {"case": c, "data": data}
    if c["items"]:
        forward, keep = c["op"] == "plan_forward", []
        for (n, v, d), t in zip(_items(c), data):
            out = torch.empty((1, v, d) if forward else (1, n, n), device="cuda", dtype=t.dtype)
            keep.append((_operator(c, n, v, d).geometry, t, out))
        s["outs"] = [k[2] for k in keep]
        s["plan"] = BatchPlan(keep, "forward" if forward else "adjoint", autotune=False)
        return s
    s["radon"] = _operator(c, c["n"], c["views"], c["det"])
    if c["table"]:
        s["radon"].build_adjoint_table()
    if c["op"] == "landweber":
        s["solver"] = Landweber(s["radon"])
        s["data"] = [data[0].requires_grad_(True), data[1].requires_grad_(True), data[2]]
    return s


# ------------------------------------------------------------------------------------------- run


def run(s):
    c, op, data = s["case"], s["case"]["op"], s["data"]
    if "plan" in s:
        s["plan"].launch()
        return s["outs"]
    radon = s["radon"]
    if op == "forward":
        return radon.forward(data[0])
    if op == "backprojection":
        return radon.backprojection(data[0])
    if op == "pair":
        y = radon.forward(data[0])
        return [y, radon.backprojection(y)]
    if op == "fbp":
        return radon.fbp(data[0])
    if op == "cgne":
        return cgne(radon, data[0], data[1], c["iterations"])
    if op == "step":
        x = data[0].detach().requires_grad_(True)
        y = radon.forward(x)
        loss = ((y - data[1]) ** 2).sum()
        loss.backward()
        return [y.detach(), x.grad]
    x0, y, g = data
    x = s["solver"].run(x0, y, _alpha(c), c["iterations"])
    gy, gx = torch.autograd.grad(x, (y, x0), g)
    return [x.detach(), gy, gx]


# ------------------------------------------------------------------------------------------ work


def _samples(n, det, views, spacing, step):
    """About how many samples the rays of one image have: the support box where the detector sees it."""
    return views * (n + 1) * min(n + 1, det * spacing) / (spacing * step)


def work(case):
    """Each input read and each output written once; per projection, image and sample the 2.6 pairs of a
    pixel and a ray that have a weight, one multiply and one add each."""
    c = case
    es = 4 if c["dtype"] == "f32" else 2
    if c["items"]:
        its = _items(c)
        return {"bytes": es * sum(n * n + v * d for n, v, d in its),
                "flops": 5.2 * sum(_samples(n, d, v, 1.0, 1.0) for n, v, d in its)}
    b, n, v, d, op = c["batch"], c["n"], c["views"], c["det"], c["op"]
    img, sino = b * n * n, b * v * d
    # a fan's rays are spread over the image at the spacing they have at its centre
    at = c["spacing"] * (c["source"] / (c["source"] + c["detector"]) if c["kind"] == "fan" else 1.0)
    one = 5.2 * b * _samples(n, d, v, at, c["step"])
    if op in ("forward", "backprojection"):
        return {"bytes": es * (img + sino), "flops": one}
    if op == "pair":
        return {"bytes": es * (2 * img + sino), "flops": 2 * one}
    if op == "step":
        return {"bytes": es * (2 * img + 2 * sino), "flops": 2 * one + 3 * sino}
    if op == "fbp":   # the filter as a product of transforms
        return {"bytes": es * (img + sino), "flops": one + 10.0 * sino * math.log2(4.0 * d)}
    if op == "cgne":
        k = c["iterations"]
        return {"bytes": es * (2 * img + sino), "flops": (2 * k + 2) * one}
    return {"bytes": es * (4 * img + 2 * sino), "flops": 4 * c["iterations"] * one}


# ------------------------------------------------------------------------------ the same in 64 bits


class _Exact:
    """A and A^T as their definition states them, in FP64: every sample with its four bilinear weights."""

    def __init__(self, c, n, views, det):
        self.n, self.v, self.d, self.h = n, views, det, c["step"]
        self.rays = _lines(c["kind"], views, det, c["spacing"], c["source"], c["detector"])
        k = int(math.ceil(0.5 * (n + 1) * math.sqrt(2.0) / self.h)) + 1
        self.t = torch.arange(-k, k + 1, device="cuda", dtype=torch.float64)[None, :] * self.h

    def _view(self, v):
        mx, my, ux, uy = (r[v][:, None] for r in self.rays)
        x, y, half = mx + self.t * ux, my + self.t * uy, 0.5 * (self.n + 1)
        ok = (x.abs() < half) & (y.abs() < half)
        x, y = (torch.where(ok, q + 0.5 * (self.n - 1), torch.zeros_like(q)) for q in (x, y))
        fx, fy = x.floor(), y.floor()
        i = (fy.long() + 1) * (self.n + 2) + fx.long() + 1   # in the image with a border of one zero pixel
        x, y, h = x - fx, y - fy, ok * self.h
        return i, [(0, (1 - x) * (1 - y) * h), (1, x * (1 - y) * h), (self.n + 2, (1 - x) * y * h), (self.n + 3, x * y * h)]

    def forward(self, x):
        b = x.shape[0]
        p = torch.nn.functional.pad(x.double(), (1, 1, 1, 1)).reshape(b, -1).T.contiguous()
        y = torch.empty((self.v, self.d, b), device="cuda", dtype=torch.float64)
        for v in range(self.v):
            i, ws = self._view(v)
            acc = 0.0
            for o, w in ws:
                acc = acc + torch.bmm(w[:, None, :], p[(i + o).reshape(-1)].reshape(self.d, -1, b))[:, 0]
            y[v] = acc
        return y.permute(2, 0, 1).contiguous()

    def adjoint(self, y):
        b = y.shape[0]
        yt = y.double().permute(1, 2, 0).contiguous()
        p = torch.zeros(((self.n + 2) ** 2, b), device="cuda", dtype=torch.float64)
        for v in range(self.v):
            i, ws = self._view(v)
            for o, w in ws:
                at = (w != 0).nonzero(as_tuple=True)
                p.index_add_(0, i[at] + o, w[at][:, None] * yt[v][at[0]])
        return p.T.reshape(b, self.n + 2, self.n + 2)[:, 1:-1, 1:-1].contiguous()

    def ramp(self, y):
        """Ram-Lak: the band-limited ramp kernel over the zero-padded views, scaled by pi / V."""
        p = 1 << max(1, (2 * self.d - 2).bit_length())
        m = torch.arange(p, device="cuda", dtype=torch.float64)
        m = torch.where(m <= p // 2, m, m - p)
        k = torch.where(m % 2 != 0, -1.0 / (math.pi * torch.where(m == 0, torch.ones_like(m), m)) ** 2, torch.zeros_like(m))
        k[0] = 0.25
        f = torch.fft.rfft(y.double(), n=p) * torch.fft.rfft(k).real
        return torch.fft.irfft(f, n=p)[..., : self.d] * (math.pi / self.v)


def exact(case, seed):
    c, op = case, case["op"]
    data = [t.double() for t in _data(c, seed)]
    if c["items"]:
        ops = [_Exact(c, n, v, d) for n, v, d in _items(c)]
        return [a.forward(t) if op == "plan_forward" else a.adjoint(t) for a, t in zip(ops, data)]
    a = _Exact(c, c["n"], c["views"], c["det"])
    if op == "forward":
        return a.forward(data[0])
    if op == "backprojection":
        return a.adjoint(data[0])
    if op == "pair":
        y = a.forward(data[0])
        return [y, a.adjoint(y)]
    if op == "fbp":
        return a.adjoint(a.ramp(data[0]))
    if op == "step":
        y = a.forward(data[0])
        return [y, a.adjoint(2.0 * (y - data[1]))]
    if op == "cgne":
        x, r = data[0].clone(), data[1] - a.forward(data[0])
        s = a.adjoint(r)
        p, gamma = s.clone(), (s * s).sum((1, 2), keepdim=True)
        for _ in range(c["iterations"]):
            q = a.forward(p)
            step = gamma / (q * q).sum((1, 2), keepdim=True)
            x, r = x + step * p, r - step * q
            s = a.adjoint(r)
            new = (s * s).sum((1, 2), keepdim=True)
            p, gamma = s + (new / gamma) * p, new
        return x
    x, y, g = data
    alpha, gy = _alpha(c), torch.zeros_like(y)
    for _ in range(c["iterations"]):
        x = x - alpha * a.adjoint(a.forward(x) - y)
    for _ in range(c["iterations"]):
        t = a.forward(g)
        gy += alpha * t
        g = g - alpha * a.adjoint(t)
    return [x, gy, g]
