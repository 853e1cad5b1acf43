"""Performance cases: the calls that programs built on this library make, over the range of their sizes.

Grids, view counts, contrasts and optics are those of the repository's configurations, tests and benchmark
(phantoms/, bench.py): lambda = 0.532 um in water, voxels of lambda/8, illumination on a cone of NA 0.8,
contrasts up to 0.05.  `exact` is the same physics in complex128 torch: Prop. 1's kernel, plain FFTs and
BiCGStab to 1e-11.
"""
import math

import numpy as np
import torch

import paper_1910_13844_gb300 as ls
from paper_1910_13844_gb300 import recon

LAM, ETA_B, NA = 0.532, 1.333, 0.8
KB = 2.0 * math.pi * ETA_B / LAM
H = LAM / 8.0
AXES = (16, 24, 32, 48, 64, 72, 96, 128, 144, 192)
LARGEST = 60 * 128 ** 3                      # views x voxels of the largest listed case


def listed():
    return [
        # one operator application on the smallest everyday grid: a user's own iteration or a unit check
        _case("matvec_32", "matvec", 32),
        # quick-look solve of a small bead, one wave along z
        _case("forward_32x1", "forward", 32, views=1, na=0.0),
        # the served workload's small grids: one request's views in one call
        _case("forward_64x24", "forward", 64, views=24),
        # a burst of mixed forward and gradient requests at the continuous-batching server
        dict(_case("serve_burst", "serve", 64, views=16), requests=8),
        # the gradient half of a reconstruction step whose forward fields are kept
        _case("gradient_96x16", "gradient", 96, views=16),
        # a non-cubic grid, adjoint operator, an odd number of vectors
        _case("adjoint_ragged_7", "matvec_batch", (72, 48, 96), views=7, adjoint=True),
        # the benchmark's headline operator: 60 vectors at 128^3
        _case("matvec_128x60", "matvec_batch", 128, views=60),
        # detector-plane operators: far field through a pupil, and its adjoint
        _case("detector_96x20", "detector", 96, views=20, det=72),
        # a cell on a flat grid, 40 views, the data for a reconstruction
        _case("forward_cell_40", "forward", (96, 128, 128), views=40, phantom="cell"),
        # one reconstruction step (loss and gradient) at the benchmark's size: the largest case
        _case("step_128x60", "step", 128, views=60),
        # a large field of view with few views
        _case("forward_192x8", "forward", 192, views=8),
        # the bead convergence study's fine grid, one wave along z
        _case("forward_bead_144x1", "forward", 144, views=1, na=0.0, phantom="bead"),
    ]


def _case(name, kind, grid, views=1, adjoint=False, na=NA, det=0, phantom="ellipsoids"):
    nz, ny, nx = (grid,) * 3 if isinstance(grid, int) else grid
    return dict(name=name, kind=kind, nz=nz, ny=ny, nx=nx, views=views, adjoint=adjoint, na=na, det=det,
                phantom=phantom)


def draw(rng):
    kind = rng.choice(["matvec", "matvec_batch", "matvec_batch", "forward", "forward", "forward", "gradient",
                       "gradient", "step", "detector"])
    n = rng.choice(AXES)
    grid = [n, n, n]
    if rng.random() < 0.5:                       # flat and ragged grids: axes within a factor of two
        grid = [rng.choice([a for a in AXES if n / 2 <= a <= 2 * n]) for _ in range(3)]
    voxels = grid[0] * grid[1] * grid[2]
    most = max(1, min(60, LARGEST // (voxels * (1 if kind == "step" else 2))))
    views = 1 if kind == "matvec" else min(most, int(round(math.exp(rng.uniform(0.0, math.log(most + 0.49))))))
    det = rng.choice([0, 0, min(grid[1], grid[2]) - 2 * rng.randrange(0, 4)])
    if kind == "detector":                       # the pupil's transforms take the grid lengths
        det = rng.choice([0] + [a for a in AXES if a < min(grid[1:])])
    elif grid[1] != grid[2]:
        det = 0
    c = _case("", kind, tuple(grid), views=max(1, views), adjoint=rng.random() < 0.5, det=det,
              na=rng.choice([0.0, 0.4, NA]), phantom=rng.choice(["ellipsoids", "ellipsoids", "bead", "cell"]))
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------------- inputs
def _axis(n, dev):
    return (torch.arange(n, dtype=torch.float64, device=dev) - n // 2 + 1) * H


def _coords(shape, dev):
    nz, ny, nx = shape
    return _axis(nz, dev)[:, None, None], _axis(ny, dev)[None, :, None], _axis(nx, dev)[None, None, :]


def _potential(case, seed, dev):
    """Scattering potential of a seeded phantom, float32."""
    shape = (case["nz"], case["ny"], case["nx"])
    rng = np.random.default_rng(seed)
    z, y, x = _coords(shape, dev)
    dn = torch.zeros(shape, dtype=torch.float64, device=dev)
    half = np.array([n * H / 2 for n in shape])

    def add(centre, semi, contrast):
        q = ((z - centre[0]) / semi[0]) ** 2 + ((y - centre[1]) / semi[1]) ** 2 + ((x - centre[2]) / semi[2]) ** 2
        torch.maximum(dn, torch.where(q <= 1.0, float(contrast), 0.0), out=dn)

    if case["phantom"] == "bead":                # a homogeneous sphere a third of the box across
        add(rng.uniform(-0.5, 0.5, 3) * H, np.full(3, half.min() / 3), rng.uniform(0.08, 0.1))
    elif case["phantom"] == "cell":              # cytoplasm, nucleus, granules
        shell = 0.78 * half
        add(np.zeros(3), shell, rng.uniform(0.025, 0.03))
        add([0.0, 0.0, 0.12 * half[2]], 0.3 * half, 0.05)
        for _ in range(50):
            add(rng.uniform(-0.55, 0.55, 3) * shell, np.full(3, rng.uniform(0.03, 0.06) * half.min()), 0.08)
    else:                                        # 20 ellipsoids, contrast up to 0.05
        for _ in range(20):
            semi = rng.uniform(0.06, 0.32, 3) * half
            add(rng.uniform(-1, 1, 3) * (0.97 * half - semi.max()).clip(0), semi, rng.uniform(0.0, 0.05))
    return (KB * KB * (((ETA_B + dn) / ETA_B) ** 2 - 1.0)).float()


def _kvec(case, seed):
    """Wave vectors on the illumination cone, azimuths evenly spaced from a seeded start."""
    q = case["views"]
    s = case["na"] / ETA_B
    phi = 2 * np.pi * (np.arange(q) / q + np.random.default_rng(seed + 1).random())
    return KB * np.stack([s * np.cos(phi), s * np.sin(phi), np.full(q, math.sqrt(1 - s * s))], axis=1)


def _waves(case, kvec, dev):
    """Plane waves at the voxel centres, complex64 (views, nz, ny, nx)."""
    z, y, x = _coords((case["nz"], case["ny"], case["nx"]), dev)
    out = torch.empty((len(kvec),) + (case["nz"], case["ny"], case["nx"]), dtype=torch.complex64, device=dev)
    for q, k in enumerate(kvec):
        out[q] = torch.exp(1j * k[2] * z) * torch.exp(1j * k[1] * y) * torch.exp(1j * k[0] * x)
    return out


def _speckle(n, my, mx, seed, dev):
    """Band-limited complex fields on the detector (spatial frequencies within the cone's NA), rms 0.3."""
    g = torch.Generator(device=dev).manual_seed(seed + 2)
    s = torch.randn(n, my, mx, 2, generator=g, device=dev, dtype=torch.float64)
    wy = 2 * math.pi * torch.fft.fftfreq(my, H, device=dev, dtype=torch.float64)[:, None]
    wx = 2 * math.pi * torch.fft.fftfreq(mx, H, device=dev, dtype=torch.float64)[None, :]
    f = torch.fft.ifft2(torch.view_as_complex(s) * (wy ** 2 + wx ** 2 <= (KB * NA / ETA_B) ** 2))
    return (0.3 * f / f.abs().square().mean().sqrt()).to(torch.complex64)


def _vectors(case, seed, dev):
    """Krylov-like vectors: plane waves with noise."""
    g = torch.Generator(device=dev).manual_seed(seed + 3)
    v = _waves(case, _kvec(case, seed), dev)
    for q in range(v.shape[0]):
        v[q] += torch.view_as_complex(torch.randn(v.shape[1:] + (2,), generator=g, device=dev) * 0.3)
    return v


def _fields(case, f, kvec, dev):
    """Total fields as the phase approximation has them: the plane wave times exp(i/(2 kb) int f dz)."""
    u = _waves(case, kvec, dev)
    phase = torch.exp(1j * torch.cumsum(f.double(), 0) * (H / (2 * KB))).to(torch.complex64)
    return u * phase


def _inputs(case, seed, dev):
    """The seeded inputs of a case, shared by prepare() and exact()."""
    kind, q = case["kind"], case["views"]
    my, mx = (case["det"] or case["ny"]), (case["det"] or case["nx"])
    d = {"f": _potential(case, seed, dev)}
    if kind in ("matvec", "matvec_batch"):
        d["x"] = _vectors(case, seed, dev)
    if kind in ("forward", "gradient", "step", "serve"):
        d["kvec"] = _kvec(case, seed)
    if kind == "forward":
        d["u_in"] = _waves(case, d["kvec"], dev)
    if kind == "gradient":
        d["u"] = _fields(case, d["f"], d["kvec"], dev)
        d["w"] = [float(w) for w in 1.0 / (0.09 * my * mx * np.random.default_rng(seed).uniform(0.8, 1.2, q))]
    if kind == "detector":
        d["u"] = _fields(case, d["f"], _kvec(case, seed), dev)
    if kind in ("gradient", "detector", "step", "serve"):
        d["y"] = _speckle(q, my, mx, seed, dev)
    return d


def _requests(case):
    """(first view, views, gradient?) of a serving burst: uneven requests, about a third of them gradients."""
    q = case["views"]
    return [(i % 3, max(1, q - 2 * i), i % 3 == 2) for i in range(case["requests"])]


def prepare(case, seed):
    d = _inputs(case, seed, "cuda")
    kind, shape = case["kind"], (case["nz"], case["ny"], case["nx"])
    if kind == "serve":
        # a server that has been up for a while: its lane exists, as after any earlier request
        d["server"] = ls.Server(KB, H, hbm_budget_bytes=16 << 30, max_views_per_grid=8 * case["views"])
        far = torch.empty((1,) + shape[1:], dtype=torch.complex64, device="cuda")
        d["server"].wait(d["server"].submit_forward(d["f"], d["kvec"][:1], far=far))
        d["out"] = []
        for first, n, grad in _requests(case):
            n = min(n, case["views"] - first)
            out = {"far": torch.empty((n,) + shape[1:], dtype=torch.complex64, device="cuda")}
            if grad:
                out = {"grad": torch.empty(shape, dtype=torch.float32, device="cuda")}
            d["out"].append((first, n, grad, out))
        return dict(d, kind=kind)
    plan = ls.Plan(shape, KB, H, **({"det_mx": case["det"], "det_my": case["det"]} if case["det"] else {}))
    if kind == "detector":
        ls.ls_set_pupil(plan.handle, 2 * math.pi * NA / LAM, -plan_distance(case))
        d["far"], d["back"] = plan.detector(case["views"]), plan.field(case["views"])
    if kind == "step":
        d["problem"] = recon.Problem(plan, d["kvec"], d["y"])
    if kind in ("matvec", "matvec_batch"):
        d["out"] = torch.empty_like(d["x"])
    return dict(d, plan=plan, kind=kind, adjoint=case["adjoint"])


def plan_distance(case):
    """Distance of the detector plane from the grid's origin (the default, 3/4 of the box), um."""
    return 0.75 * case["nz"] * H


def run(s):
    kind = s["kind"]
    if kind == "matvec":
        ls.ls_matvec(s["plan"].handle, s["f"], s["x"][0], s["out"][0], s["adjoint"])
        return s["out"][0]
    if kind == "matvec_batch":
        ls.ls_matvec_batch(s["plan"].handle, s["f"], s["x"], s["out"], s["adjoint"])
        return s["out"]
    if kind == "forward":
        u, far, _, _ = s["plan"].forward(s["f"], s["u_in"])
        return {"u": u, "far": far}
    if kind == "gradient":
        g, _, _ = s["plan"].gradient(s["f"], s["y"], u_fwd=s["u"], weights=s["w"])
        return g
    if kind == "detector":
        ls.ls_farfield(s["plan"].handle, s["f"], s["u"], s["far"])
        ls.ls_farfield_adjoint(s["plan"].handle, s["y"], s["back"])
        return {"far": s["far"], "back": s["back"]}
    if kind == "step":
        loss, g = recon.data_grad(s["problem"], s["f"])
        return {"loss": np.float32(loss), "grad": g}
    server, tickets = s["server"], []
    for first, n, grad, out in s["out"]:
        k = s["kvec"][first:first + n]
        if grad:
            tickets.append(server.submit_gradient(s["f"], k, s["y"][first:first + n], out["grad"]))
        else:
            tickets.append(server.submit_forward(s["f"], k, far=out["far"]))
    for t in tickets:
        server.wait(t)
    return [out for _, _, _, out in s["out"]]


# ---------------------------------------------------------------------------------------------- work
def work(case):
    """One pass: each input read once, each output written once; the FFT arithmetic at 5 L log2 L a transform.

    A solve is counted as five BiCGStab iterations and its two residuals (twelve operator applications)."""
    nz, ny, nx = case["nz"], case["ny"], case["nx"]
    n, q, kind = nz * ny * nx, case["views"], case["kind"]
    m = (case["det"] or ny) * (case["det"] or nx)

    def fft(length, count):
        return 5.0 * length * math.log2(length) * count

    op = 2 * (fft(2 * nx, ny * nz) + fft(2 * ny, 2 * nx * nz) + fft(2 * nz, 4 * nx * ny)) + 6.0 * 8 * n
    far = (fft(2 * nx, ny * nz) + fft(2 * ny, 2 * nx * nz) + 8.0 * 4 * n)
    green, k2 = 8.0 * (nx + 1) * (ny + 1) * (nz + 1), 8.0 * 4 * n
    b, fl = {
        "matvec": (16.0 * n, op),
        "matvec_batch": (16.0 * n * q, op * q),
        "forward": (16.0 * n * q + 8.0 * m * q + k2, (12 * op + far) * q),
        "gradient": (8.0 * n * q + 8.0 * m * q + 4.0 * n + k2, (12 * op + far) * q),
        "step": (8.0 * m * q + 4.0 * n + k2, (24 * op + 2 * far) * q),
        "detector": (16.0 * n * q + 16.0 * m * q + k2, 2 * far * q),
        "serve": (0.0, 0.0),
    }[kind]
    if kind == "serve":
        for first, count, grad in _requests(case):
            count = min(count, q - first)
            b += 8.0 * m * count + 4.0 * n * (2 if grad else 1)
            fl += (12 * op + far) * count * (2 if grad else 1)
    return {"bytes": b + 4.0 * n + (green if kind != "detector" else 0.0), "flops": fl}


# ---------------------------------------------------------------------------------------------- 64 bits
class _Exact:
    """The operators in complex128: Prop. 1's kernel on the 2n grid, and the detector's per-slice kernels."""

    def __init__(self, shape, dev, p=4):
        self.shape, self.dev = shape, dev
        size = [n * H for n in shape]
        radius = math.sqrt(sum(v * v for v in size))
        q = [torch.fft.fftfreq(2 * n, 1.0 / (2 * n), device=dev, dtype=torch.float64) for n in shape]
        for n, v in zip(shape, q):
            v[n] = n                                   # centred index set [-n+1, n]
        kern = torch.zeros([2 * n for n in shape], dtype=torch.complex128, device=dev)
        for s in np.ndindex(*(p // 2,) * 3):
            w = [2 * math.pi / (p * v) * (p // 2 * qi - si) for v, qi, si in zip(size, q, s)]
            ph = [torch.exp(-2j * math.pi * qi * si / (n * p)) for qi, si, n in zip(q, s, shape)]
            r = (w[0][:, None, None] ** 2 + w[1][None, :, None] ** 2 + w[2][None, None, :] ** 2).sqrt()
            t = torch.fft.ifftn(self._ghat(r, radius))
            kern += t * ph[0][:, None, None] * ph[1][None, :, None] * ph[2][None, None, :]
        kern *= 8.0 / p ** 3
        kern[shape[0]] = 0
        kern[:, shape[1]] = 0
        kern[:, :, shape[2]] = 0
        self.ghat = torch.fft.fftn(kern)
        self.k2 = None

    @staticmethod
    def _ghat(w, radius):
        """int_0^R exp(i kb r) sin(w r)/w dr through E(s) = int_0^R exp(i s r) dr = R exp(i s R/2) sinc(s R/2)."""
        def e(s):
            return radius * torch.exp(0.5j * radius * s) * torch.sinc(s * (radius / (2 * math.pi)))
        zero = (complex(math.cos(KB * radius), math.sin(KB * radius)) * (1 - 1j * KB * radius) - 1) / KB ** 2
        safe = torch.where(w == 0, 1.0, w)
        return torch.where(w == 0, zero, (e(KB + safe) - e(KB - safe)) / (2j * safe))

    def green(self, v, adjoint):
        nz, ny, nx = self.shape
        a = torch.fft.fft(torch.fft.fft(torch.fft.fft(v, n=2 * nx, dim=2), n=2 * ny, dim=1), n=2 * nz, dim=0)
        a = torch.fft.ifft(a * (self.ghat.conj() if adjoint else self.ghat), dim=0)[:nz]
        return torch.fft.ifft(torch.fft.ifft(a, dim=1)[:, :ny], dim=2)[:, :, :nx]

    def op(self, f, x, adjoint=False):
        return x - self.green(f * x, adjoint)

    def solve(self, f, b, adjoint=False, tol=1e-11):
        x = b.clone()
        r = b - self.op(f, x, adjoint)
        rh, bn = r.clone(), b.norm()
        rho = alpha = omega = 1.0
        v = p = torch.zeros_like(b)
        for _ in range(200):
            if float(r.norm()) <= tol * float(bn):
                break
            new = torch.vdot(rh.flatten(), r.flatten())
            p = r + (new / rho) * (alpha / omega) * (p - omega * v)
            v = self.op(f, p, adjoint)
            alpha = new / torch.vdot(rh.flatten(), v.flatten())
            s = r - alpha * v
            t = self.op(f, s, adjoint)
            omega = torch.vdot(t.flatten(), s.flatten()) / torch.vdot(t.flatten(), t.flatten())
            x = x + alpha * p + omega * s
            r, rho = s - omega * t, new
        return x

    def _slices(self):
        if self.k2 is None:
            nz, ny, nx = self.shape
            d = [torch.fft.fftfreq(2 * n, 1.0 / (2 * n), device=self.dev, dtype=torch.float64) * H for n in (ny, nx)]
            r = ((0.75 * nz * H - _axis(nz, self.dev))[:, None, None] ** 2 + d[0][None, :, None] ** 2
                 + d[1][None, None, :] ** 2).sqrt()
            k = torch.exp(1j * KB * r) / (4 * math.pi * r) * H ** 3
            k[:, ny] = 0
            k[:, :, nx] = 0
            self.k2 = torch.fft.fft2(k)
        return self.k2

    def far(self, v, det):
        nz, ny, nx = self.shape
        my, mx = det or ny, det or nx
        oy, ox = (ny - my) // 2, (nx - mx) // 2
        a = (self._slices() * torch.fft.fft2(v, s=(2 * ny, 2 * nx))).sum(0)
        return torch.fft.ifft2(a)[oy:oy + my, ox:ox + mx]

    def far_adjoint(self, r):
        nz, ny, nx = self.shape
        my, mx = r.shape
        oy, ox = (ny - my) // 2, (nx - mx) // 2
        pad = torch.zeros((2 * ny, 2 * nx), dtype=torch.complex128, device=self.dev)
        pad[oy:oy + my, ox:ox + mx] = r
        return torch.fft.ifft2(self._slices().conj() * torch.fft.fft2(pad))[:, :ny, :nx]

    def pupil(self, y, distance, adjoint=False):
        my, mx = y.shape
        w = [2 * math.pi * torch.fft.fftfreq(2 * m, H, device=self.dev, dtype=torch.float64) for m in (my, mx)]
        w2 = w[0][:, None] ** 2 + w[1][None, :] ** 2
        h = torch.where(w2 <= (2 * math.pi * NA / LAM) ** 2,
                        torch.exp(1j * distance * (KB * KB - w2).clamp(min=0).sqrt()), 0.0)
        return torch.fft.ifft2((h.conj() if adjoint else h) * torch.fft.fft2(y, s=(2 * my, 2 * mx)))[:my, :mx]

    def gradient(self, f, u, r, weights):
        g = torch.zeros(self.shape, dtype=torch.float64, device=self.dev)
        for q in range(len(r)):
            w = self.solve(f, self.far_adjoint(r[q].to(torch.complex128)), True)
            g += float(weights[q]) * (u[q].to(torch.complex128).conj() * w).real
        return g

    def wave(self, case, k):
        z, y, x = _coords(self.shape, self.dev)
        return torch.exp(1j * k[2] * z) * torch.exp(1j * k[1] * y) * torch.exp(1j * k[0] * x)


def exact(case, seed):
    kind, shape, q = case["kind"], (case["nz"], case["ny"], case["nx"]), case["views"]
    solves = {"forward": q, "gradient": q, "step": 2 * q, "serve": 3 * q}.get(kind, 0)
    if solves * shape[0] * shape[1] * shape[2] > LARGEST:
        return None                                    # over about 20 seconds
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    d, e = _inputs(case, seed, dev), _Exact(shape, dev)
    f = d["f"].double()
    wide = torch.complex128
    if kind in ("matvec", "matvec_batch"):
        out = torch.stack([e.op(f, v.to(wide), case["adjoint"]) for v in d["x"]])
        return out[0] if kind == "matvec" else out
    if kind == "forward":
        u = torch.stack([e.solve(f, v.to(wide)) for v in d["u_in"]])
        return {"u": u, "far": torch.stack([e.far(f * v, case["det"]) for v in u])}
    if kind == "gradient":
        return e.gradient(f, d["u"], d["y"], d["w"])
    if kind == "detector":
        away = -plan_distance(case)
        far = torch.stack([e.pupil(e.far(f * v.to(wide), case["det"]), away) for v in d["u"]])
        return {"far": far, "back": torch.stack([e.far_adjoint(e.pupil(v.to(wide), away, True)) for v in d["y"]])}

    def loss_and_gradient(kvec, y):
        u = [e.solve(f, e.wave(case, k)) for k in kvec]
        y = y.to(wide)
        r = [e.far(f * v, case["det"]) - m for v, m in zip(u, y)]
        w = [1.0 / float(m.abs().square().sum()) for m in y]
        loss = 0.5 * sum(c * float(v.abs().square().sum()) for c, v in zip(w, r))
        return loss, e.gradient(f, u, r, w)

    if kind == "step":
        loss, g = loss_and_gradient(d["kvec"], d["y"])
        return {"loss": loss, "grad": g}
    out = []
    for first, n, grad in _requests(case):
        last = first + min(n, q - first)
        if grad:
            out.append({"grad": loss_and_gradient(d["kvec"][first:last], d["y"][first:last])[1]})
        else:
            out.append({"far": torch.stack([e.far(f * e.solve(f, e.wave(case, k)), 0) for k in d["kvec"][first:last]])})
    return out
