"""The work a user of the library has it do, as measured cases.

One pass of a string case is what a program does between two looks at its strings: set the paths, run some
iterations, read the paths (and the barrier or the energy curve) back.  One pass of the gradient case is a
forward and backward of ``autograd.string_energies``.  Contexts, which a program keeps, are made in
``prepare``.  Outputs of single-precision trajectories are handed over in single precision (their energies
are evaluated in FP64, but the states they belong to carry FP32 digits).

``exact`` restates the method in plain torch FP64 (the dipole field through torch.fft): Eqs. 1-13 of
arXiv:1804.07135 and the variants as include/ss.h describes them.
"""
import math

import numpy as np
import torch

from paper_1804_07135_gb300 import autograd, binding

# The uneven parameter study's four lattices with the strings its seeded draw gives to each (20 in all).
STUDY = ((192, 192, 8, 4), (128, 128, 8, 6), (96, 96, 4, 6), (64, 64, 4, 4))


def listed():
    return [
        # The smallest calls: the quick-start and smoke workload (16x16x1, 16 images, 200 iterations, one
        # barrier), where launches and latencies are all there is.
        _string("tiny-16x16x1", 16, 16, 1, 16, 200, D=0.3, K=0.05, w=0.01, R=4.0, read="barrier"),
        # The plain method at its smallest, FP64 with the direct dipole sum, as a check path is run.
        _string("tiny-fp64-direct-16x16x1", 16, 16, 1, 16, 50, D=0.3, K=0.05, w=0.01, R=4.0, precision="fp64",
                dipole="direct", read="energies"),
        # The paper's own monolayer: one string of 60 images, the barrier checked every 100 iterations.
        _string("monolayer-112x112x1", 112, 112, 1, 60, 100, D=5.30 / 54.23, K=1.0 / 54.23, w=2.787e-4, R=14.0,
                read="barrier"),
        # The same with the refinements of the phase-diagram driver: spline interpolation, climbing image.
        _string("monolayer-spline-climb", 112, 112, 1, 60, 64, D=5.30 / 54.23, K=1.2 / 54.23, w=2.787e-4, R=14.0,
                interp="spline", climb=True),
        # A lattice nobody tuned for: odd extents, three layers, an odd number of images.
        _string("ragged-75x45x3", 75, 45, 3, 21, 100, D=0.25, K=0.1, w=0.02, R=9.0),
        # The Bloch-point collapse string, the ordinary single-string run.
        _string("bloch-64x64x8", 64, 64, 8, 32, 100, D=0.25, K=0.1, w=0.02, R=8.0, read="barrier"),
        # Its adaptive Dormand-Prince evolution.
        _string("dopri5-64x64x8", 64, 64, 8, 32, 8, D=0.25, K=0.1, w=0.02, R=8.0, integrator="dopri5"),
        # Precessional dynamics of independent images (damping 0.5 at a step of 0.05, where the explicit step is
        # stable for the shortest waves too).
        _string("llg-96x96x4", 96, 96, 4, 16, 100, D=0.25, K=0.1, w=0.01, R=12.0, dynamics="llg"),
        # The plain FP64 method on a film.
        _string("fp64-64x64x4", 64, 64, 4, 16, 16, D=0.25, K=0.1, w=0.02, R=8.0, precision="fp64", read="energies"),
        # dE/ds of every image and dE/d(J, D, K, w): the differentiation workload, forward and backward.
        dict(name="gradient-64x64x8", kind="gradient", nx=64, ny=64, nz=8, images=32, D=0.25, K=0.1, w=0.02, R=8.0),
        # The boundary-annihilation sweep: eight strings of 48 images in one batch.
        _string("sweep-128x128x4-8x48", 128, 128, 4, 48, 32, D=0.2, K=0.05, w=0.01, R=10.0, strings=8, path="boundary"),
        # The largest: the uneven study, 20 strings on four lattices in one batch.
        dict(name="study-20x32", kind="study", images=32, iters=24),
    ]


def _string(name, nx, ny, nz, images, iters, D, K, w, R, strings=1, path="bloch", precision="fp32", dipole="fft",
            interp="linear", climb=False, integrator="euler", dynamics="string", read="curve"):
    c = dict(kind="string", nx=nx, ny=ny, nz=nz, images=images, strings=strings, iters=iters, D=D, K=K, w=w, R=R,
             path=path, precision=precision, dipole=dipole, interp=interp, climb=climb, integrator=integrator,
             dynamics=dynamics, read=read)
    if name is not None:
        c["name"] = name
    return c


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: films of 12 to 200 sites a side and 1 to 8 layers, 8 to 64 images, one to
    eight strings, every option; iterations such that a pass stays near a tenth of a second."""
    mode = rng.choice(["plain", "plain", "plain", "plain", "plain", "batch", "batch", "variant", "rk", "llg", "fp64",
                       "gradient"])
    fp64 = mode == "fp64"
    nx = _log_int(rng, 12, 72 if fp64 else 200)
    ny = nx if rng.random() < 0.4 else max(12, min(200, int(nx * rng.uniform(0.5, 1.5))))
    nz = rng.choice([1, 1, 2, 3, 4, 4, 5, 6, 8, 8])
    images = rng.randint(8, 64)
    strings = rng.randint(2, 8) if mode == "batch" else 1
    cap = 400_000 if fp64 else 15_000_000
    while strings > 1 and nx * ny * nz * images * strings > cap:
        strings -= 1
    while nx * ny * nz * images > cap and images > 8:
        images -= 1
    while nx * ny * nz * images > cap and nz > 1:
        nz -= 1
    sites = nx * ny * nz * images * strings
    D, K, w = rng.uniform(0.15, 0.4), rng.uniform(0.02, 0.2), rng.choice([2.787e-4, 0.01, 0.02])
    R = max(3.0, min(nx, ny) / 8.0)
    if mode == "gradient":
        return dict(kind="gradient", nx=nx, ny=ny, nz=nz, images=min(images, max(2, 2_000_000 // (nx * ny * nz))), D=D, K=K,
                    w=w, R=R)
    per = {"fp64": 4e6, "rk": 3e7}.get(mode, 4e8)
    iters = max(4 if mode == "rk" else 10, min(16 if mode == "rk" else 100, int(per / sites)))
    more = {}
    if mode == "variant":
        more = dict(interp=rng.choice(["linear", "spline"]), climb=True)
    elif mode == "rk":
        more = dict(integrator=rng.choice(["dopri5", "rkf45"]))
    elif mode == "llg":
        more = dict(dynamics="llg")
    elif fp64:
        more = dict(precision="fp64", read="energies")
    elif mode == "plain":
        more = dict(read=rng.choice(["curve", "barrier"]))
    if mode in ("plain", "batch"):
        more["path"] = rng.choice(["bloch", "boundary"])
    return _string(None, nx, ny, nz, images, iters, D, K, w, R, strings=strings, **more)


# ---- inputs ------------------------------------------------------------------------------------------

def _specs(case):
    """The strings of a case: (nx, ny, nz, J, D, K, w, images) and (path, R) of each."""
    if case["kind"] == "study":
        out, i = [], 0
        for nx, ny, nz, count in STUDY:
            for _ in range(count):
                # K ~ [0, 0.2], D ~ [0.15, 0.4] spread over the strings, both paths in turn
                out.append(((nx, ny, nz, 1.0, 0.15 + 0.25 * ((7 * i) % 20) / 19, 0.2 * ((3 * i) % 20) / 19, 0.01,
                             case["images"]), ("boundary" if i % 2 else "bloch", nx / 8.0)))
                i += 1
        return out
    n = case.get("strings", 1)
    return [((case["nx"], case["ny"], case["nz"], 1.0, case["D"] * (1 + 0.05 * i), case["K"] * (1 + 0.1 * i), case["w"],
              case["images"]), (case.get("path", "bloch"), case["R"])) for i in range(n)]


LLG_ALPHA = 0.5


def _dt(case):
    return 0.05 if case.get("dynamics") == "llg" else 0.1


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _paths(case, seed):
    """The initial paths, [images][sites][3]: a Neel skyrmion (core down, linear profile of radius R) that
    shrinks into the ferromagnet or leaves through the edge, with a slight random tilt of every spin."""
    gen = torch.Generator(device=_device()).manual_seed(int(seed))
    dtype = torch.float64 if case.get("precision") == "fp64" else torch.float32
    out = []
    for (nx, ny, nz, _, _, _, _, images), (kind, R) in _specs(case):
        f = dict(dtype=torch.float32, device=_device())
        k = torch.arange(images, **f) / (images - 1)
        x, y = torch.arange(nx, **f)[None, None, :], torch.arange(ny, **f)[None, :, None]
        x0, y0 = (nx - 1) / 2.0, (ny - 1) / 2.0
        xc = x0 + (k * ((nx - 1) + R - x0) if kind == "boundary" else 0.0 * k)
        dx, dy = x - xc[:, None, None], y - y0
        r = torch.sqrt(dx * dx + dy * dy)
        theta = torch.where(r < R, math.pi * (1.0 - r / R), torch.zeros_like(r))
        if kind != "boundary":
            theta = theta * (1.0 - k)[:, None, None]
        phi = torch.atan2(dy + 0.0 * dx, dx + 0.0 * dy) + math.pi
        s = torch.stack([torch.sin(theta) * torch.cos(phi), torch.sin(theta) * torch.sin(phi), torch.cos(theta)], -1)
        s = s[:, None].expand(images, nz, ny, nx, 3).reshape(images, nz * ny * nx, 3)
        s = s + 0.02 * torch.randn(s.shape, generator=gen, **f)
        out.append((s / s.norm(dim=-1, keepdim=True)).to(dtype).contiguous())
    return out


def prepare(case, seed):
    specs = _specs(case)
    paths = _paths(case, seed)
    kw = dict(dt=_dt(case))
    if case.get("precision") == "fp64":
        kw["precision"] = binding.SS_PREC_FP64
    if case.get("dipole") == "direct":
        kw["dipole"] = binding.SS_DIPOLE_DIRECT
    sm = binding.StringMethod([s for s, _ in specs], **kw)
    if case.get("interp") == "spline" or case.get("climb"):
        sm.set_reparam(binding.SS_INTERP_SPLINE if case["interp"] == "spline" else binding.SS_INTERP_LINEAR, case["climb"])
    if case.get("integrator", "euler") != "euler":
        sm.set_integrator({"dopri5": binding.SS_INT_DOPRI5, "rkf45": binding.SS_INT_RKF45}[case["integrator"]], 1e-6, 1e-8)
    if case.get("dynamics") == "llg":
        sm.set_dynamics(binding.SS_DYN_LLG, LLG_ALPHA)
    state = dict(case=case, sm=sm, paths=paths)
    if case["kind"] == "gradient":
        state["spins"] = paths[0].requires_grad_(True)
        state["params"] = torch.tensor([1.0, case["D"], case["K"], case["w"]], dtype=torch.float64, requires_grad=True)
        state["weights"] = torch.linspace(0.5, 1.5, case["images"], dtype=torch.float64, device=_device())
    else:
        state["out"] = [torch.empty_like(p) for p in paths]
    return state


def run(state):
    case, sm = state["case"], state["sm"]
    if case["kind"] == "gradient":
        spins, params = state["spins"], state["params"]
        energies = autograd.string_energies(sm, 0, spins, params)
        g_spins, g_params = torch.autograd.grad((energies * state["weights"]).sum(), (spins, params))
        return dict(energies=energies.detach(), spins=g_spins, params=g_params)
    for i, p in enumerate(state["paths"]):
        sm.set_path(i, p)
    sm.step(case["iters"])
    out = {}
    n = len(state["paths"])
    single = case.get("precision") != "fp64"
    read = case.get("read", "curve")
    if read == "barrier":
        out["barrier"] = np.array([sm.barrier(i)[0] for i in range(n)], dtype=np.float32)
    elif read == "energies":
        out["energies"] = np.stack([sm.energies(i) for i in range(n)])
    else:
        e = np.stack([sm.step_energies(i) for i in range(n)])
        out["curve"] = e.astype(np.float32) if single else e
    for i, o in enumerate(state["out"]):
        binding.ss_get_path(sm.ctx, i, o)
    out["paths"] = state["out"]
    return out


def work(case):
    """Bytes of the paths in and out and of the constants; FLOPs of the iterations: per site and image the
    local terms, step and redistribution (about 150), the padded x and y transforms of the three components
    both ways (real data) and the layer convolution."""
    total_b = total_f = 0.0
    rounds = {"dopri5": 7, "rkf45": 6}.get(case.get("integrator"), 1)
    iters = case.get("iters", 1)
    size = 8 if case.get("precision") == "fp64" else 4
    for (nx, ny, nz, _, _, _, _, images), _ in _specs(case):
        sites = nx * ny * nz * images
        f = 150.0
        if case.get("dipole") == "direct":
            f += 25.0 * nx * ny * nz
        else:
            f += 6 * (5 * math.log2(max(2, 2 * nx)) + 10 * math.log2(max(2, 2 * ny))) + 72.0 * nz
        total_b += 2 * 3 * size * sites + 8 * images
        total_f += f * sites * (iters * rounds if case["kind"] != "gradient" else 1)
    return {"bytes": total_b, "flops": total_f}


# ---- the method in plain torch, 64 bits ------------------------------------------------------------------

class _Exact:
    """One string: the effective field of a batch of images [K][nz][ny][nx][3]."""

    def __init__(self, spec):
        self.nx, self.ny, self.nz, self.J, self.D, self.K, self.w, self.images = spec
        self.shape = (self.nz, self.ny, self.nx, 3)
        self.hat = None
        if self.w != 0.0:
            f = dict(dtype=torch.float64, device=_device())
            ax = [torch.cat([torch.arange(n, **f), torch.zeros(1, **f), torch.arange(-(n - 1), 0, **f)]) for n in
                  (self.nz, self.ny, self.nx)]
            z, y, x = torch.meshgrid(*ax, indexing="ij")
            keep = torch.ones_like(x)
            keep[self.nz], keep[:, self.ny], keep[:, :, self.nx] = 0.0, 0.0, 0.0
            keep[0, 0, 0] = 0.0
            r2 = (x * x + y * y + z * z).clamp(min=0.5)
            r5 = keep * r2 ** -2.5
            r3 = keep * r2 ** -1.5
            t = {}
            for a, p in enumerate((x, y, z)):
                for b, q in enumerate((x, y, z)):
                    if b >= a:
                        t[a, b] = torch.fft.rfftn(3.0 * p * q * r5 - (r3 if a == b else 0.0))
            self.hat = t

    def conv(self, s):
        if self.hat is None:
            return torch.zeros_like(s)
        out = torch.empty_like(s)
        size = (2 * self.nz, 2 * self.ny, 2 * self.nx)
        for k in range(s.shape[0]):  # image by image: the padded spectra of a whole string are large
            f = [torch.fft.rfftn(s[k, ..., b], s=size) for b in range(3)]
            for a in range(3):
                g = sum(self.hat[min(a, b), max(a, b)] * f[b] for b in range(3))
                out[k, ..., a] = torch.fft.irfftn(g, s=size)[: self.nz, : self.ny, : self.nx]
        return out

    def field(self, s, conv=None):
        h = self.w * (self.conv(s) if conv is None else conv)
        h[..., 2] += 2.0 * self.K * s[..., 2]
        J, D = self.J, self.D
        for ax in (1, 2, 3):
            n = s.shape[ax]
            if n > 1:
                lo, hi = [slice(None)] * 4, [slice(None)] * 4
                lo[ax], hi[ax] = slice(0, n - 1), slice(1, n)
                lo, hi = tuple(lo), tuple(hi)
                h[lo] += J * s[hi]
                h[hi] += J * s[lo]
                if ax == 1:
                    continue  # no interlayer DMI
                c = 0 if ax == 3 else 1
                h[lo + (c,)] -= D * s[hi + (2,)]
                h[hi + (c,)] += D * s[lo + (2,)]
                h[lo + (2,)] += D * s[hi + (c,)]
                h[hi + (2,)] -= D * s[lo + (c,)]
        return h

    def terms(self, s):
        """Per image dE/d(J, D, K, w)."""
        c = self.conv(s)
        keep = self.J, self.D, self.K, self.w
        out = []
        for q in range(4):
            self.J, self.D, self.K, self.w = [1.0 if i == q else 0.0 for i in range(4)]
            out.append(-0.5 * (self.field(s, c) * s).sum(dim=(1, 2, 3, 4)))
        self.J, self.D, self.K, self.w = keep
        return torch.stack(out, 1)


def _unit(s):
    return s / s.norm(dim=-1, keepdim=True)


def _force(s, h):
    return h - (s * h).sum(-1, keepdim=True) * s


def _llg(s, h, alpha):
    return -torch.cross(s, h, dim=-1) / (1 + alpha * alpha) + alpha / (1 + alpha * alpha) * _force(s, h)


def _spline_weights(x, t):
    """phi(t_i) = sum_q W_iq y_q of the natural cubic spline through knots x."""
    n = len(x) - 1
    h = x[1:] - x[:-1]
    A, B = np.eye(n + 1), np.zeros((n + 1, n + 1))
    for i in range(1, n):
        A[i, i - 1], A[i, i], A[i, i + 1] = h[i - 1], 2 * (h[i - 1] + h[i]), h[i]
        B[i, i - 1], B[i, i], B[i, i + 1] = 6 / h[i - 1], -6 / h[i - 1] - 6 / h[i], 6 / h[i]
    P = np.linalg.solve(A, B)
    W = np.zeros((len(t), n + 1))
    for i, v in enumerate(t):
        j = min(max(int(np.searchsorted(x, v, side="right")) - 1, 0), n - 1)
        a, b = (x[j + 1] - v) / h[j], (v - x[j]) / h[j]
        W[i, j] += a
        W[i, j + 1] += b
        W[i] += h[j] ** 2 / 6 * ((a ** 3 - a) * P[j] + (b ** 3 - b) * P[j + 1])
    return W


def _redistribute(s, spline, kc):
    """Equal arc length over the string, or over its two parts on either side of a climbing image."""
    n = s.shape[0]
    d = [float((s[k] - s[k - 1]).norm()) for k in range(1, n)]
    arc = np.concatenate([[0.0], np.cumsum(d)])
    out = s.clone()
    for a, b in [(0, kc), (kc, n - 1)] if 0 < kc < n - 1 else [(0, n - 1)]:
        length = arc[b] - arc[a]
        if b - a < 2 or not length > 0:
            continue
        x = (arc[a:b + 1] - arc[a]) / length
        t = np.arange(1, b - a) / (b - a)
        if spline:
            W = _spline_weights(x, t)
        else:
            W = np.zeros((len(t), b - a + 1))
            for i, v in enumerate(t):
                j = min(int(np.searchsorted(x, v, side="right")) - 1, b - a - 1)
                W[i, j + 1] = (v - x[j]) / (x[j + 1] - x[j])
                W[i, j] = 1 - W[i, j + 1]
        if spline:
            part = torch.tensordot(torch.from_numpy(W).to(s.device), s[a:b + 1], dims=1)
            out[a + 1:b] = _unit(part)
        else:
            for i in range(len(t)):
                j = int(np.nonzero(W[i])[0][0])
                mix = W[i, j] * s[a + j] + (W[i, j + 1] * s[a + j + 1] if j + 1 <= b - a else 0.0)
                out[a + 1 + i] = _unit(mix)
    return out


_DOPRI = ([[], [1 / 5], [3 / 40, 9 / 40], [44 / 45, -56 / 15, 32 / 9],
           [19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729],
           [9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656],
           [35 / 384, 0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84]],
          [35 / 384, 0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84, 0],
          [5179 / 57600, 0, 7571 / 16695, 393 / 640, -92097 / 339200, 187 / 2100, 1 / 40])
_RKF = ([[], [1 / 4], [3 / 32, 9 / 32], [1932 / 2197, -7200 / 2197, 7296 / 2197], [439 / 216, -8, 3680 / 513, -845 / 4104],
         [-8 / 27, 2, -3544 / 2565, 1859 / 4104, -11 / 40]],
        [25 / 216, 0, 1408 / 2565, 2197 / 4104, -1 / 5, 0],
        [16 / 135, 0, 6656 / 12825, 28561 / 56430, -9 / 50, 2 / 55])


def _rk_interval(m, y, T, step, tab, rtol=1e-6, atol=1e-8):
    a, b, b2 = tab
    t = 0.0
    while t < T:
        hs = min(step, T - t)
        k = []
        for row in a:
            Y = y
            for c, q in zip(row, k):
                Y = Y + (hs * c) * q
            k.append(_force(Y, m.field(Y)))
        y5 = y + hs * sum(c * q for c, q in zip(b, k))
        e = hs * sum((c - c2) * q for c, c2, q in zip(b, b2, k))
        err = float((e / (atol + rtol * torch.maximum(y.abs(), y5.abs()))).square().mean().sqrt())
        fac = min(5.0, max(0.2, 0.9 * err ** -0.2 if err > 0 else 5.0))
        if err <= 1:
            t = T if hs == T - t else t + hs
            y = _unit(y5)
        else:
            fac = min(1.0, fac)
        step = hs * fac
    return y, step


def _run_exact(case, spec, path):
    m = _Exact(spec)
    s = _unit(path.to(torch.float64)).reshape((spec[7],) + m.shape)
    spline, climb = case.get("interp") == "spline", bool(case.get("climb"))
    llg, rk = case.get("dynamics") == "llg", case.get("integrator", "euler")
    dt, kc, curve, step = _dt(case), -1, None, _dt(case)
    for _ in range(case["iters"]):
        h = m.field(s)
        curve = -0.5 * (h * s).sum(dim=(1, 2, 3, 4))
        if rk != "euler":
            s2, step = _rk_interval(m, s, dt, step, _DOPRI if rk == "dopri5" else _RKF)
        elif llg:
            s = _unit(s + dt * _llg(s, h, LLG_ALPHA))
            continue
        else:
            F = _force(s, h)
            if 0 < kc < spec[7] - 1:
                tau = s[kc + 1] - s[kc - 1]
                tau = tau - (tau * s[kc]).sum(-1, keepdim=True) * s[kc]
                F[kc] -= 2 * float((F[kc] * tau).sum()) / float((tau * tau).sum()) * tau
            s2 = _unit(s + dt * F)
        s = _redistribute(s2, spline, kc)
        if climb:
            kc = 1 + int(torch.argmax(curve[1:-1]))
    return m, s, curve


def exact(case, seed):
    paths = _paths(case, seed)
    if case["kind"] == "gradient":
        spec = _specs(case)[0][0]
        m = _Exact(spec)
        s = paths[0].to(torch.float64).reshape((spec[7],) + m.shape)
        wts = torch.linspace(0.5, 1.5, case["images"], dtype=torch.float64, device=_device())
        s = _unit(s)
        h = m.field(s)
        t = m.terms(s)
        return dict(energies=-0.5 * (h * s).sum(dim=(1, 2, 3, 4)),
                    spins=-(wts[:, None, None, None, None] * h).reshape(spec[7], -1, 3),
                    params=(wts[:, None] * t).sum(0))
    out, energies, curves, barriers = [], [], [], []
    read = case.get("read", "curve")
    for (spec, _), path in zip(_specs(case), paths):
        m, s, curve = _run_exact(case, spec, path)
        out.append(s.reshape(spec[7], -1, 3))
        curves.append(curve)
        if read != "curve":
            e = -0.5 * (m.field(s) * s).sum(dim=(1, 2, 3, 4))
            energies.append(e)
            barriers.append(float(e.max() - e[0]))
    res = dict(paths=out)
    if read == "barrier":
        res["barrier"] = np.array(barriers)
    elif read == "energies":
        res["energies"] = torch.stack(energies)
    else:
        res["curve"] = torch.stack(curves)
    return res
