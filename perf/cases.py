"""The library's work in use, as cases that can be timed and checked.

A case is one call (or one call and its backward) through the public entry
points of `paper_2507_02401_gb300`: the forward map K and its adjoint K* on
2D and 3D grids, the wavelet embedding E_s and E_s*, the objective with its
gradient, the medium gradient and the batched CG.  Grids, orders, sensor
layouts and time axes are those of the repository's workloads
(synth/workloads.py); `draw` spreads sizes, orders, media and layers over the
same ranges, odd widths included.

`exact` states the same operators in FP64 with plain torch (the eliminated
pressure recurrence with the composed stencil, sensor sampling, the periodic
wavelet transform, CG), sharing nothing with the library.
"""
import math

import numpy as np
import torch

from paper_2507_02401_gb300 import Batch, Plan, autograd

H = 1.0e-4  # grid spacing [m]
CFL = 0.3
C0 = 1500.0
DEV = "cuda"


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest wave call: K of the 64 x 64 second-order test problem
        dict(name="forward_64", op="forward", nz=0, ny=64, nx=64, order=2, varc=False, layer=0, nt=250, ns=32,
             arc=False, levels=3, family=2, s=1.0),
        # one step of a gradient method (or of CG) on the 512 x 512 varying-medium problem: J(u) and its gradient,
        # i.e. E_s, K, K* and E_s* once each
        dict(name="objective_512", op="objective", nz=0, ny=512, nx=512, order=8, varc=True, layer=0, nt=1500, ns=512,
             arc=False, levels=5, family=4, s=1.0, alpha=0.5),
        # limited view inside an absorbing layer: K and its backward through autograd, sensors on an arc
        dict(name="layer_512", op="grad", nz=0, ny=512, nx=512, order=8, varc=False, layer=10, nt=1200, ns=80, arc=True,
             levels=5, family=4, s=1.0),
        # differentiation through a long record on a grid too large for one wave of on-chip tiles
        dict(name="grad_1024", op="grad", nz=0, ny=1024, nx=1024, order=8, varc=False, layer=0, nt=3000, ns=256,
             arc=True, levels=6, family=4, s=1.5),
        # a ragged grid with a row length that no vector width divides: K and its backward, varying medium
        dict(name="grad_1000x875", op="grad", nz=0, ny=1000, nx=875, order=4, varc=True, layer=0, nt=600, ns=200,
             arc=False, levels=0, family=4, s=1.0),
        # a 2D field larger than the L2 cache, partial tiles on both axes: K and its backward
        dict(name="grad_4000x3600", op="grad", nz=0, ny=4000, nx=3600, order=8, varc=False, layer=0, nt=300, ns=512,
             arc=False, levels=4, family=4, s=1.0),
        # 3D reconstruction: K and K* of the 256^3 problem (each half of every CG iteration there)
        dict(name="forward_256c", op="forward", nz=256, ny=256, nx=256, order=4, varc=False, layer=0, nt=800, ns=4096,
             arc=False, levels=4, family=4, s=1.0),
        dict(name="adjoint_256c", op="adjoint", nz=256, ny=256, nx=256, order=4, varc=False, layer=0, nt=800, ns=4096,
             arc=False, levels=4, family=4, s=1.0),
        # the embedding and its adjoint on an image and on a volume
        dict(name="wavelet_2048", op="wavelet", nz=0, ny=2048, nx=2048, order=2, varc=False, layer=0, nt=1, ns=4,
             arc=False, levels=5, family=4, s=1.0),
        dict(name="wavelet_256c", op="wavelet", nz=256, ny=256, nx=256, order=2, varc=False, layer=0, nt=1, ns=4,
             arc=False, levels=4, family=4, s=1.0),
        # sensitivity of the data to the medium (sound-speed estimation)
        dict(name="kappa_384", op="kappa", nz=0, ny=384, nx=384, order=8, varc=True, layer=0, nt=700, ns=256, arc=False,
             levels=4, family=4, s=1.0),
        # many independent reconstructions of uneven size at once (two CG iterations of each)
        dict(name="batch_32", op="batch", count=32, sizes="128 192 256 384 512", order=8,
             iters=2, levels=4, family=4, alpha=0.05),
    ]


def _shape(case):
    return ((case["nz"],) if case["nz"] else ()) + (case["ny"], case["nx"])


def _ext(shape):
    return dict(nz=shape[0] if len(shape) == 3 else 0, ny=shape[-2], nx=shape[-1])


def _sizes(case):
    pool = [int(n) for n in case["sizes"].split()]
    return [pool[k % len(pool)] for k in range(case["count"])]


# point-updates (cells x steps x wave applications) of the costliest listed case
MOST = 2 * 800 * 256 ** 3 // 2


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["forward", "adjoint", "grad", "grad", "objective", "wavelet", "vol", "vol", "kappa", "batch"])
    order = rng.choice([2, 4, 6, 8])
    family = rng.choice([1, 2, 4, 4])
    s = rng.choice([0.5, 1.0, 1.5, 2.0])
    if op == "batch":
        sizes = " ".join(str(n) for n in rng.sample([96, 128, 192, 256, 320, 384], rng.randint(1, 4)))
        return dict(op="batch", count=rng.randint(2, 16), sizes=sizes, order=order, iters=1, levels=3, family=family,
                    alpha=0.05)
    if op == "vol":
        op = rng.choice(["forward", "adjoint", "wavelet"])
        levels = rng.randint(1, 4)
        unit = 2 ** levels
        shape = [max(1, logint(48, 256) // unit) * unit for _ in range(3)]
        if op != "wavelet" and rng.random() < 0.3:  # a width that no vector width divides
            levels = 0
            shape[2] = 2 * (shape[2] // 2) - 1
        nt = logint(20, 200)
        return dict(op=op, **_ext(shape), order=rng.choice([2, 4, 4, 6]), varc=rng.random() < 0.25, layer=0, nt=nt,
                    ns=logint(64, 4096), arc=False, levels=levels, family=family, s=s)
    if op == "wavelet":
        levels = rng.randint(2, 6)
        unit = 2 ** levels
        shape = [max(1, logint(128, 4096) // unit) * unit for _ in range(2)]
        return dict(op=op, **_ext(shape), order=2, varc=False, layer=0, nt=1, ns=4, arc=False, levels=levels,
                    family=family, s=s)
    hi = {"kappa": 512, "objective": 1400}.get(op, 4000)
    levels = 3
    shape = [max(1, logint(64, hi) // 8) * 8 for _ in range(2)]
    if op in ("forward", "adjoint", "grad") and rng.random() < 0.3:
        levels = 0
        shape = [shape[0] + rng.randint(0, 7), shape[1] + rng.randint(1, 7)]
    apps = {"forward": 1, "adjoint": 1, "grad": 2, "objective": 2, "kappa": 8}[op]
    cells = shape[0] * shape[1]
    nt = min(int(math.ceil(math.sqrt(2.0) * max(shape) / CFL)), MOST // (16 * cells * apps), 2000)
    layer = 10 if op in ("forward", "grad") and order >= 4 and rng.random() < 0.25 else 0
    return dict(op=op, **_ext(shape), order=order, varc=rng.random() < 0.4, layer=layer, nt=max(nt, 2),
                ns=logint(32, 512), arc=rng.random() < 0.5, levels=levels, family=family, s=s, alpha=0.5)


# ------------------------------------------------------------ inputs of a case
def _sensors(shape, ns, arc):
    """Sensor coordinates (x, y[, z]) [m]: a circle or 180-degree arc of radius
    0.45 of the shorter side, or a Fibonacci sphere."""
    ext = np.array(shape[::-1], dtype=np.float64) - 1.0
    mid, rad = 0.5 * ext * H, 0.45 * ext.min() * H
    if len(shape) == 2:
        th = np.arange(ns) * ((math.pi / max(ns - 1, 1)) if arc else (2.0 * math.pi / ns))
        return np.stack([mid[0] + rad * np.cos(th), mid[1] + rad * np.sin(th)], axis=1)
    i = np.arange(ns) + 0.5
    z = 1.0 - 2.0 * i / ns
    th = math.pi * (1.0 + math.sqrt(5.0)) * i
    q = np.sqrt(1.0 - z * z)
    return np.stack([mid[0] + rad * q * np.cos(th), mid[1] + rad * q * np.sin(th), mid[2] + rad * z], axis=1)


def _speed(shape, rng):
    """Smooth random speed of sound in [1400, 1600] m/s: a few random plane waves."""
    ax = [torch.linspace(0.0, 1.0, n, device=DEV, dtype=torch.float64) for n in shape]
    f = torch.zeros(shape, device=DEV, dtype=torch.float64)
    for _ in range(8):
        k = rng.normal(0.0, 3.0, len(shape))
        ph = rng.uniform(0.0, 2.0 * math.pi)
        for a in range(len(shape)):
            ph = ph + (2.0 * math.pi * k[a] * ax[a]).reshape([-1 if b == a else 1 for b in range(len(shape))])
        f += torch.cos(ph)
    f = (f - f.min()) / (f.max() - f.min())
    return (1400.0 + 200.0 * f).cpu().numpy()


def _phantom(shape, rng, nt=0, blobs=4, vessels=4):
    """Initial pressure: Gaussian blobs (amplitude 0.5 .. 1, width 2 .. 6 cells)
    plus thin curved vessels, a float32 tensor on the GPU; and the blobs.  They
    lie within 0.3 of the shorter side; on a record of nt samples too short for
    waves to get from there to the sensors, the blobs lie near the sensors."""
    d = len(shape)
    ax = [torch.arange(n, device=DEV, dtype=torch.float32) for n in shape]
    x = torch.zeros(shape, device=DEV)
    mid = (np.array(shape) - 1) / 2.0
    rad = 0.3 * min(shape)

    def bump(p, w):
        g = [torch.exp(-((ax[a] - float(p[a])) ** 2) / (2.0 * w * w)) for a in range(d)]
        out = g[0]
        for a in range(1, d):
            out = out.unsqueeze(-1) * g[a]
        return out

    pts = []
    for _ in range(blobs):
        v = rng.normal(size=d)
        dist = rad * rng.random() ** (1.0 / d)
        if 0 < CFL * nt < 0.2 * min(shape):
            dist = 0.45 * min(shape) - 0.5 * CFL * nt * rng.random()
            v[0] = abs(v[0])  # the side of the grid that an arc of sensors covers
        p = mid + dist * v / np.linalg.norm(v)
        amp, w = rng.uniform(0.5, 1.0), rng.uniform(2.0, 6.0)
        pts.append((p, amp, w))
        x += amp * bump(p, w)
    for _ in range(vessels):
        ctl = mid + rng.uniform(-rad, rad, (4, d))
        amp, w = rng.uniform(0.5, 1.0), rng.uniform(0.7, 1.5)
        for t in np.linspace(0.0, 1.0, 24):
            b = np.array([(1 - t) ** 3, 3 * t * (1 - t) ** 2, 3 * t * t * (1 - t), t ** 3])
            x = torch.maximum(x, amp * bump(b @ ctl, w))
    return x, pts


def _traces(shape, sens, pts, dt, nt, rng, noise=0.02):
    """Sensor data (ns, nt), float32 on the GPU: the spherical-wave pulse of every
    blob, its echoes off the faces (pressure zero outside the grid) and noise."""
    r_s = torch.as_tensor(sens, device=DEV, dtype=torch.float32)
    ct = C0 * dt * torch.arange(nt, device=DEV, dtype=torch.float32)
    y = torch.zeros((len(sens), nt), device=DEV)
    for p, amp, w in pts:
        pos = np.array(p[::-1]) * H
        images = [(pos, 1.0)]
        for a, n in enumerate(shape[::-1]):
            for face in (0.0, (n - 1) * H):
                q = pos.copy()
                q[a] = 2.0 * face - q[a]
                images.append((q, -1.0))
        for q, sign in images:
            r = (r_s - torch.as_tensor(q, device=DEV, dtype=torch.float32)).norm(dim=1).clamp_min(H).unsqueeze(1)
            u = (r - ct) / (w * H)
            y += sign * amp * (0.25 + 0.5 * u) * w * H / r * torch.exp(-0.5 * u * u)
    g = torch.Generator(device=DEV)
    g.manual_seed(int(rng.integers(1 << 31)))
    return y + noise * y.abs().max() * torch.randn(y.shape, device=DEV, generator=g)


def _problem(case, rng):
    shape = _shape(case)
    c = _speed(shape, rng) if case["varc"] else C0
    return dict(shape=shape, c=c, dt=CFL * H / float(np.max(c)), nt=case["nt"], order=case["order"],
                sens=_sensors(shape, case["ns"], case["arc"]), layer=case["layer"], levels=case["levels"],
                family=case["family"])


def _plan(p):
    plan = Plan(p["shape"], H, p["dt"], p["nt"], p["order"], p["c"], p["sens"], family=p["family"],
                levels=p["levels"])
    if p["layer"]:
        plan.set_sponge(p["layer"])
    return plan


def _batch_problems(case, rng):
    out = []
    for n in _sizes(case):
        ns = int(rng.integers(64, 513))
        out.append(dict(shape=(n, n), c=C0, dt=CFL * H / C0, nt=int(math.ceil(math.sqrt(2.0) * n / CFL)),
                        order=case["order"], sens=_sensors((n, n), ns, bool(rng.random() < 0.5)), layer=0,
                        levels=case["levels"], family=case["family"], s=float(rng.choice([1.0, 1.5, 2.0])),
                        alpha=case["alpha"] * 10.0 ** rng.uniform(-1.0, 1.0)))
    return out


def _inputs(case, seed):
    """The case's problem(s) and input tensors, from the seed alone."""
    rng = np.random.default_rng(seed)
    op = case["op"]
    if op == "batch":
        ps = _batch_problems(case, rng)
        pts = [_phantom(p["shape"], rng, p["nt"], 3, 0)[1] for p in ps]
        ys = [_traces(p["shape"], p["sens"], b, p["dt"], p["nt"], rng) for p, b in zip(ps, pts)]
        return ps, ys
    p = _problem(case, rng)
    x, pts = _phantom(p["shape"], rng, p["nt"] if op != "wavelet" else 0)
    if op == "forward":
        return p, dict(x=x)
    if op == "adjoint":
        return p, dict(y=_traces(p["shape"], p["sens"], pts, p["dt"], p["nt"], rng))
    if op == "wavelet":
        u = analysis(x.unsqueeze(0), p["family"], p["levels"], case["s"])[0].float()
        return p, dict(u=u, gx=_phantom(p["shape"], rng)[0])
    y = _traces(p["shape"], p["sens"], pts, p["dt"], p["nt"], rng)
    if op == "objective":
        return p, dict(y=y, u=analysis(x.unsqueeze(0), p["family"], p["levels"], case["s"])[0].float())
    return p, dict(x=x, y=y)  # grad, kappa


def prepare(case, seed):
    p, t = _inputs(case, seed)
    if case["op"] == "batch":
        batch = Batch([_plan(q) for q in p])
        return dict(case=case, batch=batch, ys=t, alphas=[q["alpha"] for q in p], ss=[q["s"] for q in p])
    st = dict(case=case, plan=_plan(p), **t)
    if case["op"] == "grad":
        st["x"].requires_grad_(True)
    if case["op"] == "objective":
        st["u"].requires_grad_(True)
    return st


def run(st):
    case = st["case"]
    op = case["op"]
    if op == "forward":
        return st["plan"].forward(st["x"])
    if op == "adjoint":
        return st["plan"].adjoint(st["y"])
    if op == "grad":  # y = K x and gx = K* gy
        y = autograd.K(st["plan"], st["x"])
        (gx,) = torch.autograd.grad(y, st["x"], st["y"])
        return [y.detach(), gx]
    if op == "objective":
        J = autograd.reconstruction_loss(st["plan"], st["u"], st["y"], case["alpha"], case["s"])
        (gu,) = torch.autograd.grad(J, st["u"])
        return [J.detach(), gu]
    if op == "wavelet":
        return [st["plan"].Es(st["u"], case["s"]), st["plan"].EsT(st["gx"], case["s"])]
    if op == "kappa":
        return st["plan"].grad_kappa(st["x"].detach(), st["y"])
    return st["batch"].solve(st["ys"], st["alphas"], st["ss"], case["iters"])[0]


def work(case):
    """Each input read once and each output written once; two flops per stencil
    tap pair and axis beyond the pair's sum, per cell and step."""
    radius = {2: 1, 4: 3, 6: 5, 8: 7}[case["order"]]
    if case["op"] == "batch":
        b = f = 0
        for n in _sizes(case):
            nt = int(math.ceil(math.sqrt(2.0) * n / CFL))
            apps = 1 + 2 * case["iters"]
            b += 4 * (288 * nt + n * n)
            f += apps * nt * n * n * (2 * 3 * radius + 4)
        return {"bytes": b, "flops": f}
    cells, d = math.prod(_shape(case)), len(_shape(case))
    data = case["ns"] * case["nt"]
    per_step = cells * case["nt"] * (d * 3 * radius + 4)
    taps = cells * d * 2 * 2 * case["family"] * 2
    io = {"forward": cells + data, "adjoint": cells + data, "grad": 2 * cells + 2 * data,
          "objective": 2 * cells + data, "wavelet": 4 * cells, "kappa": 2 * cells + data}[case["op"]]
    if case["varc"]:
        io += 2 * cells
    f = {"forward": per_step, "adjoint": per_step, "grad": 2 * per_step, "objective": 2 * per_step + 2 * taps,
         "wavelet": 2 * taps, "kappa": 4 * per_step}[case["op"]]
    return {"bytes": 4 * io, "flops": f}


# --------------------------------------------------------------- FP64 statement
def _filters(family):
    """Daubechies scaling and wavelet filters by spectral factorisation."""
    n = family
    roots = []
    if n > 1:
        poly = [math.comb(n - 1 + k, k) for k in range(n)]
        for y in np.roots(poly[::-1]):
            b = 2.0 - 4.0 * y
            q = np.sqrt(b * b - 4.0 + 0j)
            z = max((b + q) / 2.0, (b - q) / 2.0, key=abs)
            roots.append(z)
    h = np.array([1.0 + 0j])
    for z in roots:
        h = np.convolve(h, [-z, 1.0])
    for _ in range(n):
        h = np.convolve(h, [1.0, 1.0])
    h = h.real * (math.sqrt(2.0) / h.real.sum())
    return h, np.array([(-1.0) ** j * h[2 * n - 1 - j] for j in range(2 * n)])


def _split(x, ax, f):
    """sum_j f_j x[(2k + j) mod n] along axis ax."""
    n = x.shape[ax]
    out = 0
    for j, c in enumerate(f):
        i = (2 * torch.arange(n // 2, device=x.device) + j) % n
        out = out + float(c) * x.index_select(ax, i)
    return out


def _merge(c, ax, f):
    """The transpose of _split."""
    n = 2 * c.shape[ax]
    shape = list(c.shape)
    shape[ax] = n
    out = torch.zeros(shape, device=c.device, dtype=c.dtype)
    for j, v in enumerate(f):
        i = (2 * torch.arange(n // 2, device=c.device) + j) % n
        out.index_add_(ax, i, float(v) * c)
    return out


def _order2(d):
    """(x high?, y high?, ...) of the detail bands in storage order."""
    if d == 2:
        return [(0, 1), (1, 0), (1, 1)]
    return [((b >> 0) & 1, (b >> 1) & 1, (b >> 2) & 1) for b in range(1, 8)]


def analysis(x, family, levels, s, offset=0):
    """E_s* of a stack of images: (B, *grid) -> (B, N)."""
    h, g = _filters(family)
    d = x.dim() - 1
    B = x.shape[0]
    out = []
    for i in range(1, levels + 1):
        wt = 2.0 ** (-s * (levels - i + offset))
        parts = {(): x}
        for a in range(d):  # axis a = 0 is x, the last array axis
            parts = {k + (b,): _split(v, d - a, f) for k, v in parts.items() for b, f in ((0, h), (1, g))}
        out.append([(wt * parts[k]).reshape(B, -1) for k in _order2(d)])
        x = parts[(0,) * d]
    return torch.cat([x.reshape(B, -1)] + [b for bands in out[::-1] for b in bands], dim=1)


def synthesis(u, grid, family, levels, s, offset=0):
    """E_s of a stack of coefficient vectors: (B, N) -> (B, *grid)."""
    h, g = _filters(family)
    d, B = len(grid), u.shape[0]
    ext = [n >> levels for n in grid]
    pos = math.prod(ext)
    x = u[:, :pos].reshape([B] + ext)
    for i in range(levels, 0, -1):
        wt = 2.0 ** (-s * (levels - i + offset))
        n = math.prod(ext)
        parts = {(0,) * d: x}
        for k in _order2(d):
            parts[k] = wt * u[:, pos:pos + n].reshape([B] + ext)
            pos += n
        for a in range(d - 1, -1, -1):
            parts = {k: _merge(parts[k + (0,)], d - a, h) + _merge(parts[k + (1,)], d - a, g)
                     for k in {q[:-1] for q in parts}}
        x = parts[()]
        ext = [2 * e for e in ext]
    return x


class Exact:
    """K and K* in FP64 for B problems of one grid, order and time axis."""

    STAG = {2: [1.0], 4: [9 / 8, -1 / 24], 6: [75 / 64, -25 / 384, 3 / 640],
            8: [1225 / 1024, -245 / 3072, 49 / 5120, -5 / 7168]}

    def __init__(self, problems):
        p = problems[0]
        self.B, self.shape, self.nt = len(problems), p["shape"], p["nt"]
        self.d = len(self.shape)
        half = self.STAG[p["order"]]
        g = np.array([-v for v in half[::-1]] + list(half))  # staggered first difference
        w = np.convolve(g, g)  # second difference: offsets -(2M-1) .. 2M-1
        self.R = len(half) * 2 - 1
        self.w = [float(v) for v in w[self.R:]]
        kap, one = [], np.ones(self.shape)
        for q in problems:
            kap.append((np.asarray(q["c"], dtype=np.float64) * q["dt"] / H) ** 2 * (one if np.ndim(q["c"]) else 1.0))
        big = any(np.ndim(q["c"]) for q in problems)
        if big:
            self.kappa = torch.as_tensor(np.stack([k * one for k in kap]), device=DEV)
        else:
            self.kappa = torch.as_tensor(np.array(kap), device=DEV).reshape([-1] + [1] * self.d)
        self.a = self.b = None
        if p["layer"]:
            W = p["layer"]
            smax = 3.0 * float(np.max(p["c"])) * math.log(1e3) / (2.0 * W * H)
            sig = np.zeros(self.shape)
            for ax, n in enumerate(self.shape):
                dist = np.minimum(np.arange(n), n - 1 - np.arange(n))
                pr = np.where(dist < W, smax * ((W - dist) / W) ** 2, 0.0)
                sig = sig + pr.reshape([-1 if a == ax else 1 for a in range(self.d)])
            q = 0.5 * sig * p["dt"]
            self.a = torch.as_tensor((1 - q) / (1 + q), device=DEV).unsqueeze(0)
            self.b = torch.as_tensor(1 / (1 + q), device=DEV).unsqueeze(0)
        cells = math.prod(self.shape)
        idx, wts, self.ns = [], [], [len(q["sens"]) for q in problems]
        for k, q in enumerate(problems):
            u = np.asarray(q["sens"], dtype=np.float64) / H
            n = np.array(self.shape[::-1])
            i0 = np.minimum(np.floor(u).astype(np.int64), n - 2)
            f = u - i0
            ii, ww = [], []
            for c in range(1 << self.d):
                lin, wt, stride = 0, 1.0, 1
                for a in range(self.d):
                    bit = (c >> a) & 1
                    lin = lin + (i0[:, a] + bit) * stride
                    wt = wt * (f[:, a] if bit else 1.0 - f[:, a])
                    stride *= int(n[a])
                ii.append(lin + k * cells)
                ww.append(wt)
            idx.append(np.stack(ii, axis=1))
            wts.append(np.stack(ww, axis=1))
        self.idx = torch.as_tensor(np.concatenate(idx), device=DEV)
        self.wts = torch.as_tensor(np.concatenate(wts), device=DEV)
        self.pad = torch.zeros([self.B] + [n + 2 * self.R for n in self.shape], device=DEV, dtype=torch.float64)
        self.core = self.pad[(slice(None),) + tuple(slice(self.R, self.R + n) for n in self.shape)]

    def lap(self, P):
        """L P, zero outside the grid."""
        self.core.copy_(P)
        out = P * (self.d * self.w[0])
        for ax in range(self.d):
            for m in range(1, self.R + 1):
                for sgn in (-m, m):
                    sl = [slice(None)] + [slice(self.R, self.R + n) for n in self.shape]
                    sl[ax + 1] = slice(self.R + sgn, self.R + sgn + self.shape[ax])
                    out.add_(self.pad[tuple(sl)], alpha=self.w[m])
        return out

    def sample(self, P):
        return (P.reshape(-1)[self.idx] * self.wts).sum(dim=1)

    def inject(self, P, v):
        P.reshape(-1).index_add_(0, self.idx.reshape(-1), (self.wts * v.unsqueeze(1)).reshape(-1))

    def fields(self, x):
        """P^0, P^1, ... P^{nt-1}, one at a time."""
        P, D = x.clone(), None
        for n in range(self.nt):
            yield P
            if n == self.nt - 1:
                return
            inc = self.lap(P).mul_(self.kappa)
            if n == 0:
                inc.mul_(0.5)
            if self.a is None:
                D = inc if D is None else D.add_(inc)
            else:
                inc.mul_(self.b)
                D = (self.a - 1.0) * P + inc if D is None else D.mul_(self.a).add_(inc)
            P = P + D

    def forward(self, x):
        """(B, *grid) -> (sum of ns, nt)."""
        return torch.stack([self.sample(P) for P in self.fields(x)], dim=1)

    def states(self, y):
        """(m, Q^m) for m = nt-1 .. 1, then (0, K* y)."""
        G = torch.zeros([self.B] + list(self.shape), device=DEV, dtype=torch.float64)
        Q = torch.zeros_like(G)
        yt = y.t().contiguous()
        for m in range(self.nt - 1, 0, -1):
            G = G + self.lap(self.kappa * Q)
            self.inject(G, yt[m])
            Q = Q + G if self.a is None else self.a * Q + self.b * G
            yield m, Q
        x = G + 0.5 * self.lap(self.kappa * Q)
        self.inject(x, yt[0])
        if self.a is not None:
            x = x + (self.a - 1.0) / self.b * Q
        yield 0, x

    def adjoint(self, y):
        for _, x in self.states(y):
            pass
        return x


def _cg(ex, y, alphas, ss, family, levels, iters):
    """x = E_s u after `iters` CG steps from u = 0, for every problem of `ex`."""
    def each(f, v):
        return torch.cat([f(v[k:k + 1], ss[k]) for k in range(ex.B)])

    def up(u):
        return each(lambda v, s: synthesis(v, ex.shape, family, levels, s), u)

    def down(x):
        return each(lambda v, s: analysis(v, family, levels, s), x)

    def dot(a, b):
        return (a * b).sum(dim=1, keepdim=True)

    al = torch.as_tensor(alphas, device=DEV, dtype=torch.float64).unsqueeze(1)
    r = down(ex.adjoint(y))
    p, u, rr = r.clone(), torch.zeros_like(r), dot(r, r)
    for _ in range(iters):
        q = down(ex.adjoint(ex.forward(up(p)))) + al * p
        a = rr / dot(p, q)
        u, r = u + a * p, r - a * q
        new = dot(r, r)
        p, rr = r + (new / rr) * p, new
    return up(u)


def exact(case, seed):
    op = case["op"]
    p, t = _inputs(case, seed)
    if op == "batch":
        out = [None] * len(p)
        for n in sorted(set(_sizes(case))):
            ks = [k for k, q in enumerate(p) if q["shape"][0] == n]
            x = _cg(Exact([p[k] for k in ks]), torch.cat([t[k] for k in ks]).double(), [p[k]["alpha"] for k in ks],
                    [p[k]["s"] for k in ks], case["family"], case["levels"], case["iters"])
            for i, k in enumerate(ks):
                out[k] = x[i]
        return out
    fam, lev, s = p["family"], p["levels"], case["s"]
    if op == "wavelet":
        x = synthesis(t["u"].double().unsqueeze(0), p["shape"], fam, lev, s)[0]
        return [x, analysis(t["gx"].double().unsqueeze(0), fam, lev, s)[0]]
    ex = Exact([p])
    if op == "forward":
        return ex.forward(t["x"].double().unsqueeze(0))
    if op == "adjoint":
        return ex.adjoint(t["y"].double())[0]
    if op == "grad":
        return [ex.forward(t["x"].double().unsqueeze(0)), ex.adjoint(t["y"].double())[0]]
    if op == "objective":
        u = t["u"].double().unsqueeze(0)
        res = ex.forward(synthesis(u, p["shape"], fam, lev, s)) - t["y"].double()
        J = 0.5 * (res * res).sum() + 0.5 * case["alpha"] * (u * u).sum()
        return [J, (analysis(ex.adjoint(res), fam, lev, s) + case["alpha"] * u)[0]]
    # kappa: sum_n Q^{n+1} .* L P^n, the first term halved
    LP = [ex.lap(P) for P in ex.fields(t["x"].double().unsqueeze(0))]
    g = torch.zeros_like(LP[0])
    for m, Q in ex.states(t["y"].double()):
        if m >= 1:
            g += (0.5 if m == 1 else 1.0) * Q * LP[m - 1]
    return g[0]
