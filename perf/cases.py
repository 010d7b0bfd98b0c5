"""What this framework is asked to do in earnest, as cases that can be timed and checked.

The work of the framework is the Fourier reconstruction of photoacoustic data: the image from line or
planar detector data (`Plan.reconstruct`, `reconstruct`), its exact transpose and gradients through it
(`Plan.adjoint`, `PAIRecon`), the detector data of an image (`ForwardModel`, with or without the smooth
cutoff of limited-view data), one problem at a time or many uneven ones in one plan.  A user makes a plan
for a geometry and calls it on frame after frame, so a plan is what `prepare` keeps and one call is a pass.

Keys of a case
  op       reconstruct | adjoint | gradient (image and its gradient through autograd) | limited (cutoff of
           the data, then the reconstruction) | forward | batch
  dim      2 line detector, 3 planar detector;  nx, ny, nt, nz: detectors, time samples, depth samples
  dt       time step (unit spacings and sound speed otherwise)
  K        window half width at oversampling 2; 0 leaves the window to the plan, the default of a geometry
  method   "kb" or one of the compared interpolation methods
  cutoff   parameter of the smooth data cutoff in squared sampling steps (0: none)
  count, sizes  (batch) number of problems and the seed their sizes come from
"""
import math
import random

import numpy as np
import torch

import paper_0808_3510_gb300 as pai


def _case(op, dim, nx, nt, nz, ny=1, dt=1.0, K=3, method="kb", cutoff=0, name=None):
    c = dict(op=op, dim=dim, nx=nx, ny=ny, nt=nt, nz=nz, dt=dt, K=K, method=method, cutoff=cutoff)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one small slice, as in a preview or a live view: a handful of launches
        _case("reconstruct", 2, 128, 256, 128, name="line 128x256"),
        # the large slice of the benchmark, both directions
        _case("reconstruct", 2, 2048, 4096, 2048, K=4, name="line 2048x4096"),
        _case("adjoint", 2, 2048, 4096, 2048, K=4, name="line 2048x4096 adjoint"),
        # a slice of a scanner whose detector count is what it is (2^2 5 71), window left to the plan
        _case("reconstruct", 2, 1420, 3784, 1892, K=0, name="line 1420x3784"),
        # a training or iterative step on such a slice: image and gradient through autograd
        _case("gradient", 2, 666, 1500, 750, dt=0.8, name="line 666x1500 gradient"),
        # limited-view data: smooth cutoff of the data, then the image, by the cheap compared method
        _case("limited", 2, 1024, 2048, 1024, method="linear", cutoff=16, name="line 1024x2048 limited, linear"),
        # a volume of the ordinary size
        _case("reconstruct", 3, 128, 256, 128, ny=128, name="plane 128^2x256"),
        # one gradient step of an iterative reconstruction of a large volume
        _case("gradient", 3, 256, 512, 256, ny=256, name="plane 256^2x512 gradient"),
        # a volume of a detector matrix of odd extents
        _case("gradient", 3, 100, 310, 150, ny=90, K=0, name="plane 100x90x310 gradient"),
        # simulated data of a volume, and of a large slice seen through the cutoff
        _case("forward", 3, 128, 256, 128, ny=128, name="plane 128^2x256 forward"),
        _case("forward", 2, 2048, 4096, 2048, K=4, cutoff=16, name="line 2048x4096 data model"),
        # many uneven slices in one plan
        dict(op="batch", count=64, sizes=0, name="batch of 64 lines"),
    ]


def _even(rng, lo, hi):
    return 2 * int(round(math.exp(rng.uniform(math.log(lo / 2), math.log(hi / 2)))))


def draw(rng):
    kind = rng.choice(["line", "line", "line", "plane", "plane", "forward", "batch"])
    if kind == "batch":
        return dict(op="batch", count=rng.randint(2, 64), sizes=rng.randrange(1, 1 << 20))
    dt = round(rng.uniform(0.5, 1.2), 3)
    pow2 = rng.random() < 0.4  # detector arrays come in powers of two more often than not by chance

    def size(lo, hi):
        n = _even(rng, lo, hi)
        return min(hi, 1 << round(math.log2(n))) if pow2 else n

    if kind == "forward":
        dim = rng.choice([2, 3])
        if dim == 2:
            n, nt = size(64, 2048), size(128, 4096)
            return _case("forward", 2, n, nt, size(64, 2048), dt=min(dt, 1.0), K=rng.choice([3, 4]),
                         cutoff=rng.choice([0, 16]))
        return _case("forward", 3, size(32, 128), size(64, 256), size(32, 128), ny=size(32, 128), dt=min(dt, 1.0))
    op = rng.choice(["reconstruct", "reconstruct", "adjoint", "gradient"])
    K = rng.choice([3, 3, 4, 0])
    if kind == "line":
        nt = size(128, 4096)
        if rng.random() < 0.2:
            return _case("limited", 2, size(64, 2048), nt, size(64, 2048), dt=dt, K=3,
                         method=rng.choice(["kb", "linear"]), cutoff=16)
        return _case(op, 2, size(64, 2048), nt, size(64, 2048), dt=dt, K=K)
    return _case(op, 3, size(32, 256), size(64, 512), size(32, 256), ny=size(32, 256), dt=dt, K=K)


# ---------------------------------------------------------------------------
# geometries and inputs
# ---------------------------------------------------------------------------

def _geometries(case):
    if case["op"] == "batch":
        rng = random.Random(1000 + case["sizes"])
        gs = []
        for _ in range(case["count"]):
            nx, nt = 2 * rng.randint(128, 1024), 2 * rng.randint(256, 2048)
            gs.append(dict(dim=2, nx=nx, ny=1, nt=nt, nz=(nt // 2) & ~1, dx=1.0, dy=1.0, dt=1.0, c=1.0, dz=1.0,
                           method="kb"))
        return gs
    g = {k: case[k] for k in ("dim", "nx", "ny", "nt", "nz", "dt", "method")}
    g.update(dx=1.0, dy=1.0, dz=1.0, c=1.0)
    if case["K"]:
        g.update(oversampling=2.0, K=float(case["K"]))
    elif case["method"] != "kb":
        g.update(oversampling=2.0)
    return [g]


def _data_shape(g):
    return (g["nx"], g["nt"]) if g["dim"] == 2 else (g["nx"], g["ny"], g["nt"])


def _image_shape(g):
    return (g["nx"], g["nz"]) if g["dim"] == 2 else (g["nx"], g["ny"], g["nz"])


def _data(g, rng, dev):
    """Detector data of a few round objects plus 1 % white noise: line data of f_circ discs (closed form), planar
    data of uniform balls (N-waves)."""
    gen = torch.Generator(device=dev)
    gen.manual_seed(rng.randrange(1 << 40))
    t = g["dt"] * torch.arange(g["nt"], device=dev, dtype=torch.float32)
    x = torch.arange(g["nx"], device=dev, dtype=torch.float32)
    p = torch.zeros(_data_shape(g), device=dev)
    depth = g["nz"]
    for _ in range(rng.randint(2, 6)):
        r = rng.uniform(2.0, max(2.5, min(15.0, depth / 5)))
        x0, z0, a = rng.uniform(0, g["nx"]), rng.uniform(r + 2, max(r + 3, depth - r)), rng.uniform(0.5, 1.0)
        if g["dim"] == 2:
            d = torch.sqrt((x - x0) ** 2 + z0 * z0)[:, None]
            hi, lo = t + r, torch.maximum(d, t - r)
            sh = torch.sqrt(torch.clamp(hi * hi - d * d, min=0.0))
            sl = torch.sqrt(torch.clamp(lo * lo - d * d, min=0.0))
            val = (sh - sl) - t * torch.log((hi + sh) / (lo + sl))
            p += torch.where(hi > lo, (a / (2 * r)) * val, torch.zeros((), device=dev))
        else:
            y = torch.arange(g["ny"], device=dev, dtype=torch.float32)
            d = torch.sqrt((x[:, None] - x0) ** 2 + (y[None, :] - rng.uniform(0, g["ny"])) ** 2 + z0 * z0)[:, :, None]
            p += torch.where((d - t).abs() < r, a * (d - t) / (2 * d), torch.zeros((), device=dev))
    noise = torch.empty_like(p).normal_(generator=gen)
    return p + (0.01 * p.abs().max()) * noise


def _image(g, rng, dev):
    """Smooth balls in an image with a little white noise (an initial pressure, or a residual image)."""
    gen = torch.Generator(device=dev)
    gen.manual_seed(rng.randrange(1 << 40))
    shape = _image_shape(g)
    axes = [torch.arange(n, device=dev, dtype=torch.float32) for n in shape]
    f = torch.zeros(shape, device=dev)
    for _ in range(rng.randint(3, 8)):
        r = rng.uniform(3.0, 15.0)
        s2 = torch.zeros((1,) * len(shape), device=dev)
        for k, ax in enumerate(axes):
            view = [1] * len(shape)
            view[k] = -1
            s2 = s2 + ((ax - rng.uniform(0, shape[k])) / r).view(view) ** 2
        f += rng.uniform(0.5, 1.0) * torch.clamp(1 - s2, min=0.0) ** 2
    return f + 0.01 * torch.empty_like(f).normal_(generator=gen)


def _inputs(case, seed, dev):
    """(data, image): what the operation takes, None where it does not take it."""
    rng = random.Random(int(seed))
    gs = _geometries(case)
    if case["op"] == "batch":
        return torch.cat([_data(g, rng, dev).reshape(-1) for g in gs]), None
    op = case["op"]
    p = _data(gs[0], rng, dev) if op in ("reconstruct", "limited", "gradient") else None
    h = _image(gs[0], rng, dev) if op in ("adjoint", "gradient", "forward") else None
    return p, h


def prepare(case, seed):
    p, h = _inputs(case, seed, torch.device("cuda"))
    gs = _geometries(case)
    if case["op"] == "batch":
        plan = pai.Plan(gs)
    elif case["op"] == "forward":
        plan = pai.ForwardModel(gs[0], cutoff=case["cutoff"] or None)
    else:
        plan = pai.Plan(gs[0])
        if case["op"] == "limited":
            plan.set_cutoff(case["cutoff"])
    if case["op"] == "gradient":
        p.requires_grad_(True)
    return dict(op=case["op"], plan=plan, p=p, h=h)


def run(s):
    op, plan = s["op"], s["plan"]
    if op in ("reconstruct", "batch"):
        return plan.reconstruct(s["p"])
    if op == "adjoint":
        return plan.adjoint(s["h"])
    if op == "gradient":
        f = pai.PAIRecon.apply(s["p"], plan)
        (grad,) = torch.autograd.grad(f, s["p"], s["h"])
        return f.detach(), grad
    if op == "limited":
        return plan.reconstruct(plan.cutoff(s["p"]))
    return plan(s["h"])  # forward


# ---------------------------------------------------------------------------
# the work a pass cannot do without
# ---------------------------------------------------------------------------

def _fft(n):
    return 5.0 * n * math.log2(max(n, 2))


def work(case):
    """Bytes: data and images, each read or written once.  Operations: the lateral transform of the real data, per
    lateral frequency one oversampled transform (padded by 2) and the window sums at the nodes (12 taps, real times
    complex), the inverse transform of the image."""
    total = {"bytes": 0.0, "flops": 0.0}
    op = case["op"]
    passes = 2 if op == "gradient" else 1
    for g in _geometries(case):
        lat = g["nx"] * (g["ny"] if g["dim"] == 3 else 1)
        data, image = 4.0 * lat * g["nt"], 4.0 * lat * g["nz"]
        taps = 12 if g["method"] == "kb" else 2
        ops = 0.5 * (g["nt"] + g["nz"]) * _fft(lat) + 0.5 * lat * (
            _fft(2 * g["nt"]) + _fft(g["nz"]) + 4.0 * taps * g["nz"])
        total["bytes"] += passes * (data + image)
        total["flops"] += passes * ops
        if op == "limited":
            total["flops"] += lat * g["nt"]
    return total


# ---------------------------------------------------------------------------
# the same in 64 bits, by direct sums (and library FFTs on the uniform grids)
# ---------------------------------------------------------------------------

def _rows(g, n, nt):
    """(half-lateral |K|^2 / (2 pi)^2 as a flat row axis, lateral extents n = box extents)."""
    kx = torch.fft.fftfreq(n[0], d=1.0, dtype=torch.float64)
    if g["dim"] == 2:
        return (torch.arange(n[0] // 2 + 1, dtype=torch.float64) / n[0]) ** 2
    ky = torch.arange(n[1] // 2 + 1, dtype=torch.float64) / n[1]
    return (kx[:, None] ** 2 + ky[None, :] ** 2).reshape(-1)


def _split(nt):
    b = 1 << max(1, math.ceil(math.log2(math.sqrt(nt))))
    return -(-nt // b), b  # samples n = a B + b


def _tables(nu, nt):
    """e^{-2 pi i nu b / nt} (b < B) and e^{-2 pi i nu a B / nt} (a < A) for nodes nu [rows][j]."""
    A, B = _split(nt)

    def e(m):
        cycles = nu[..., None] * (m.to(nu.device) / nt)
        return torch.polar(torch.ones_like(cycles), -2 * math.pi * (cycles - torch.round(cycles)))

    return e(torch.arange(B, dtype=torch.float64)), e(B * torch.arange(A, dtype=torch.float64)), A, B


def _type2(G, nu, nt):
    """sum_n G[row][n] e^{-2 pi i nu n / nt} at nu and at -nu."""
    T1, T2, A, B = _tables(nu, nt)
    Gp = torch.nn.functional.pad(torch.view_as_real(G), (0, 0, 0, A * B - nt))
    Gp = torch.view_as_complex(Gp.contiguous()).reshape(G.shape[0], A, B).transpose(1, 2)
    plus = (torch.bmm(T1, Gp) * T2).sum(-1)
    minus = (torch.bmm(T1, Gp.conj()) * T2).sum(-1).conj()
    return plus, minus


def _type1(yp, ym, nu, nt):
    """sum_j yp[j] e^{+2 pi i nu_j n / nt} + ym[j] e^{-2 pi i nu_j n / nt}, n < nt."""
    T1, T2, A, B = _tables(nu, nt)
    plus = torch.bmm((yp[..., None] * T2.conj()).transpose(1, 2), T1.conj())
    minus = torch.bmm((ym[..., None] * T2).transpose(1, 2), T1)
    return (plus + minus).reshape(yp.shape[0], A * B)[:, :nt]


def _linear2(G, nu, nt):
    """Linear interpolation of the zero-padded transform (length M, the power of two >= 2 nt) at +-nu."""
    M = 1 << max(5, math.ceil(math.log2(2 * nt)))
    D = torch.fft.fft(G, n=M, dim=1)
    x = nu * (M / nt)
    out = []
    for s in (x, -x):
        j = torch.floor(s)
        fr = (s - j).to(torch.complex128)
        j = j.long()
        out.append((1 - fr) * torch.gather(D, 1, j % M) + fr * torch.gather(D, 1, (j + 1) % M))
    return out


def _chunks(rows, nodes, nt):
    A, B = _split(nt)
    step = max(1, int(2e9 / (16 * (2 * nodes * (A + B) + 4 * nt))))
    return [slice(r, min(rows, r + step)) for r in range(0, rows, step)]


def _nodes(g, S, nz):
    """nu and weight at depth frequencies l = 1 .. nz/2 for rows of lateral |K|^2 / (2 pi)^2 = S."""
    kz = (torch.arange(1, nz // 2 + 1, dtype=torch.float64) / nz).to(S.device)
    K = torch.sqrt(S[:, None] + kz[None, :] ** 2)
    return g["dt"] * g["nt"] * K, g["dt"] * 2.0 * kz[None, :] / K


def _lateral(g, n):
    return (n[0],) if g["dim"] == 2 else (n[0], n[1])


def _exact_reconstruct(g, p):
    """f = Re of the inverse transform of W(k, l) times the temporal spectrum at nu(k, l); zero at l = 0, the mean of
    both Nyquist nodes at l = -nz/2."""
    n = _lateral(g, (g["nx"], g["ny"]))
    nt, nz = g["nt"], g["nz"]
    axes = tuple(range(len(n)))
    P = torch.fft.rfftn(p.double(), dim=axes).reshape(-1, nt)
    S = _rows(g, n, nt).to(p.device)
    F = torch.zeros((P.shape[0], nz), dtype=torch.complex128, device=p.device)
    for c in _chunks(P.shape[0], nz // 2, nt):
        nu, w = _nodes(g, S[c], nz)
        plus, minus = (_linear2 if g["method"] == "linear" else _type2)(P[c], nu, nt)
        plus, minus = plus * w, minus * w
        F[c, 1:nz // 2] = plus[:, :-1]
        F[c, nz // 2 + 1:] = minus[:, :-1].flip(1)
        F[c, nz // 2] = 0.5 * (plus[:, -1] + minus[:, -1])
    F = torch.fft.ifft(F, dim=1).reshape(*n[:-1], n[-1] // 2 + 1, nz)
    return torch.fft.irfftn(F, s=n, dim=axes)


def _exact_adjoint(g, h):
    n = _lateral(g, (g["nx"], g["ny"]))
    nt, nz = g["nt"], g["nz"]
    axes = tuple(range(len(n)))
    Y = torch.fft.fft(torch.fft.rfftn(h.double(), dim=axes), dim=-1).reshape(-1, nz) / nz
    S = _rows(g, n, nt).to(h.device)
    Q = torch.empty((Y.shape[0], nt), dtype=torch.complex128, device=h.device)
    for c in _chunks(Y.shape[0], nz // 2, nt):
        nu, w = _nodes(g, S[c], nz)
        yp = Y[c, 1:nz // 2 + 1].clone()
        ym = Y[c].flip(1)[:, :nz // 2].clone()
        ym[:, -1] = yp[:, -1]
        yp[:, -1] *= 0.5
        ym[:, -1] *= 0.5
        Q[c] = _type1(yp * w, ym * w, nu, nt)
    Q = Q.reshape(*n[:-1], n[-1] // 2 + 1, nt)
    return torch.fft.irfftn(Q, s=n, dim=axes)


def _box(n, reach):
    b, need = 32, n + math.ceil(reach - 1e-9) + 2
    while b < need:
        b *= 2
    return b


def _exact_forward(g, f):
    """Wave-equation solution for the trigonometric interpolant of the image in its zero-padded periodic box."""
    nt, reach = g["nt"], g["nt"] * g["dt"]
    full = _lateral(g, (g["nx"], g["ny"]))
    n = tuple(_box(m, reach) for m in full)
    nz = _box(g["nz"], reach)
    axes = tuple(range(len(n)))
    F = torch.fft.fft(f.double(), n=nz, dim=-1)
    F = torch.view_as_real(F)
    if len(n) == 2:
        Fr = [torch.fft.rfft(F[..., k], n=n[1], dim=1) for k in (0, 1)]
        F = torch.fft.fft(Fr[0] + 1j * Fr[1], n=n[0], dim=0)
    else:
        Fr = [torch.fft.rfft(F[..., k], n=n[0], dim=0) for k in (0, 1)]
        F = Fr[0] + 1j * Fr[1]
    F = F.reshape(-1, nz) / nz
    S = _rows(g, n, nt).to(f.device)
    Q = torch.empty((F.shape[0], nt), dtype=torch.complex128, device=f.device)
    kz = (torch.arange(nz // 2 + 1, dtype=torch.float64) / nz).to(f.device)
    for c in _chunks(F.shape[0], nz // 2 + 1, nt):
        nu = g["dt"] * nt * torch.sqrt(S[c][:, None] + kz[None, :] ** 2)
        y = F[c, : nz // 2 + 1].clone()
        y[:, 1:nz // 2] += F[c, nz // 2 + 1:].flip(1)
        Q[c] = _type1(0.5 * y, 0.5 * y, nu, nt)
    Q = Q.reshape(*n[:-1], n[-1] // 2 + 1, nt)
    p = torch.fft.irfftn(Q, s=n, dim=axes)
    return p[: g["nx"]] if g["dim"] == 2 else p[: g["nx"], : g["ny"]]


def _cutoff_weights(g, eps, dev):
    """The smooth cutoff at every data sample: the bump exp(-1/(1 - |v|^2/eps)^4) integrated over the offsets that
    stay inside the box [0, n_a] of every axis, over its full integral; distances in sampling steps."""
    r = math.sqrt(eps)
    R = math.ceil(r)
    dim = g["dim"]
    x, w = np.polynomial.legendre.leggauss(96)

    def integral(tops):
        pts = [(-r + (t + r) * (x + 1) / 2, w * (t + r) / 2) for t in tops]
        q, m = 0.0, 1.0
        for a, (v, wt) in enumerate(pts):
            shape = [1] * dim
            shape[a] = -1
            q, m = q + v.reshape(shape) ** 2, m * wt.reshape(shape)
        q = q / eps
        inside = q < 1
        return float((np.where(inside, np.exp(-1.0 / np.where(inside, 1 - q, 1.0) ** 4), 0.0) * m).sum())

    whole = integral((r,) * dim)
    table = np.empty((R + 1,) * dim)
    for s in np.ndindex(table.shape):
        table[s] = integral([min(r, float(v)) for v in s]) / whole
    index = []
    for a, n in enumerate(_data_shape(g)):
        i = np.arange(n)
        index.append(np.minimum(np.minimum(i, n - i), R))
    return torch.from_numpy(table[np.ix_(*index)]).to(dev)


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    p, h = _inputs(case, seed, dev)
    gs, op = _geometries(case), case["op"]
    if op == "batch":
        out, at = [], 0
        for g in gs:
            n = g["nx"] * g["nt"]
            out.append(_exact_reconstruct(g, p[at:at + n].reshape(g["nx"], g["nt"])).reshape(-1))
            at += n
        return torch.cat(out)
    g = gs[0]
    if op == "reconstruct":
        return _exact_reconstruct(g, p)
    if op == "adjoint":
        return _exact_adjoint(g, h)
    if op == "gradient":
        return _exact_reconstruct(g, p), _exact_adjoint(g, h)
    if op == "limited":
        return _exact_reconstruct(g, p.double() * _cutoff_weights(g, case["cutoff"], dev))
    q = _exact_forward(g, h)
    return q * _cutoff_weights(g, case["cutoff"], dev) if case["cutoff"] else q
