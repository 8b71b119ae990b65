"""The work whose speed is measured: calls that a user of this library makes, over the sizes and options it
serves (grids 16..2048, coherent / IOTF / 9 or 25 source modes, one projection to a whole series).

Every case goes through the Python entry points of ``paper_2503_20146_gb300`` on inputs made from the seed alone:
projections of random spheroids (phases of some ten radians), a shared phase-screen diffuser with a 3 px correlation
length, Poisson counts of the blurred speckle. Solves start from an earlier estimate of the same object (0.9 of its
phase and attenuation), as a run that refines or resumes a reconstruction does (gradients are taken at 0.5), except
``solve_host``, which starts from zero like Algorithm S1. ``exact`` restates each call in 64 bits from the paper's equations, in plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2503_20146_gb300 import pwf
from paper_2503_20146_gb300.autograd import physical_model

PIXEL, WAVELENGTH, L1, L2 = 1.0e-6, 1.23984198e-6 / 2.0e4, 0.1, 0.4  # 20 keV, metres
SIGMA_PX = 2.0                                                       # std of the source blur at the detector
XCOH = SIGMA_PX * math.sqrt(4.0 * math.pi) * PIXEL
GAMMA, ALPHA = 1.0, 0.1 + 0.01j
GROUP_SIZES = (256, 768, 1536, 2048)
FBP_WIDTHS = (16, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024)


def listed():
    return [
        # one small projection's modelled intensity: the shortest call, where latency is all
        {"name": "forward_128", "kind": "forward", "batch": 1, "ny": 128, "nx": 128, "modes": 0, "coherent": False},
        # a preview solve of one small coherent projection
        {"name": "solve_128", "kind": "solve", "batch": 1, "ny": 128, "nx": 128, "modes": 0, "coherent": True, "iters": 20},
        # a solve of one ordinary projection
        {"name": "solve_512", "kind": "solve", "batch": 1, "ny": 512, "nx": 512, "modes": 0, "coherent": False, "iters": 20},
        # the Wirtinger gradient of a few wide, low strips (a radix-3 detector row, an uneven batch), for a caller's own optimiser
        {"name": "gradient_96x768", "kind": "gradient", "batch": 9, "ny": 96, "nx": 768, "modes": 0, "coherent": False},
        # the tomographic series: 180 angles at 1024^2 in one plan
        {"name": "solve_180x1024", "kind": "solve", "batch": 180, "ny": 1024, "nx": 1024, "modes": 0, "coherent": False, "iters": 5},
        # part of the same series with 9 source modes
        {"name": "solve_24x1024_k9", "kind": "solve", "batch": 24, "ny": 1024, "nx": 1024, "modes": 9, "coherent": False, "iters": 2},
        # projections of four sizes solved together, 25 source modes
        {"name": "group_mixed_k25", "kind": "group", "batch": 4, "modes": 25, "iters": 1},
        # a series in host memory streamed through the GPU: pinned buffers in and out
        {"name": "solve_host_180x128", "kind": "solve_host", "batch": 180, "ny": 128, "nx": 128, "modes": 0, "coherent": False, "iters": 10},
        # differentiation: forward and backward of the physical model at the largest grid
        {"name": "autograd_16x2048", "kind": "autograd", "batch": 16, "ny": 2048, "nx": 2048, "modes": 0, "coherent": False},
        # the same with 25 source modes
        {"name": "autograd_2x2048_k25", "kind": "autograd", "batch": 2, "ny": 2048, "nx": 2048, "modes": 25, "coherent": False},
        # filtered back projection of the whole retrieved series into a 1024^3 volume
        {"name": "fbp_180x1024", "kind": "fbp", "angles": 180, "ny": 1024, "nx": 1024},
        # and of a small ablation series
        {"name": "fbp_32x128", "kind": "fbp", "angles": 32, "ny": 128, "nx": 128},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))) - 0.5))))


def draw(rng):
    """One more case: any of the listed kinds, any grid the library serves (rectangles too), batches and iteration
    counts spread over their logarithm under a cap on the work."""
    kind = rng.choice(["forward", "solve", "solve", "gradient", "solve_host", "group", "autograd", "autograd", "fbp", "fbp"])
    if kind == "fbp":
        angles, nx = _log_int(rng, 8, 400), rng.choice(FBP_WIDTHS)
        return {"kind": kind, "angles": angles, "ny": _log_int(rng, 1, max(1, min(1024, int(1.2e11 / (angles * nx * nx))))), "nx": nx}
    if kind == "group":
        return {"kind": kind, "batch": rng.randint(1, 5), "modes": rng.choice([0, 9, 25]), "iters": rng.randint(1, 2)}
    sizes = pwf.SIZES if kind != "solve_host" else [n for n in pwf.SIZES if n <= 128]
    ny, nx = rng.choice(sizes), rng.choice(sizes)
    if rng.random() < 0.5:
        nx = ny
    modes = 0 if kind == "solve_host" else rng.choice([0, 0, 0, 9, 25])
    iters = rng.randint(1, 10) if kind in ("solve", "solve_host") else 1
    cap = 1.5e8 / (iters * (1 if modes == 0 else 1.5 * modes) * (4 if kind == "solve_host" else 1))
    case = {"kind": kind, "batch": _log_int(rng, 1, max(1, min(256, int(cap / (ny * nx))))), "ny": ny, "nx": nx, "modes": modes,
            "coherent": modes == 0 and rng.random() < 0.25}
    if kind in ("solve", "solve_host"):
        case["iters"] = iters
    return case


# ---- inputs ----------------------------------------------------------------------------------------------------------
def _eta(case):
    return 2.0 ** -10 if case.get("coherent") else 2.0 ** -9


def _sizes(case):
    return [(n, n) for n in GROUP_SIZES] if case["kind"] == "group" else [(case["ny"], case["nx"])]


def _objects(batch, ny, nx, g):
    """psi of `batch` parallel projections over 180 degrees of 16 random spheroids (as wide, for their height, as the
    detector): chords times up to 15 rad."""
    r = 0.04 + 0.16 * torch.rand(16, generator=g)
    pos = torch.rand(16, 3, generator=g) - 0.5
    amp = 3.0 + 12.0 * torch.rand(16, generator=g)
    y = torch.arange(ny, device="cuda", dtype=torch.float32)[:, None] - (ny - 1) / 2
    x = torch.arange(nx, device="cuda", dtype=torch.float32)[None, :] - (nx - 1) / 2
    psi = torch.empty((batch, ny, nx), dtype=torch.complex64, device="cuda")
    for b0 in range(0, batch, 16):
        th = math.pi * torch.arange(b0, min(batch, b0 + 16), dtype=torch.float32) / batch
        phase = torch.zeros((len(th), ny, nx), device="cuda")
        for k in range(16):
            cx = (0.8 * nx * (pos[k, 0] * torch.cos(th) + pos[k, 2] * torch.sin(th))).cuda()[:, None, None]
            d2 = ((x - cx) / (float(r[k]) * nx)).square() + ((y / ny - 0.8 * float(pos[k, 1])) / float(r[k])).square()
            phase += float(amp[k]) * (1.0 - d2).clamp_(min=0.0).sqrt_()
        psi[b0:b0 + len(th)] = torch.complex(-0.01 * phase, -phase)
    return psi


def _diffuser(ny, nx, g):
    """exp(i theta): white noise smoothed to 3 px, standard deviation 1 rad."""
    w = torch.randn(ny, nx, generator=g, dtype=torch.float32).cuda()
    u, v = torch.fft.fftfreq(nx, device="cuda")[None, :], torch.fft.fftfreq(ny, device="cuda")[:, None]
    th = torch.fft.ifft2(torch.fft.fft2(w) * torch.exp(-2.0 * (math.pi * 3.0) ** 2 * (u * u + v * v))).real
    th = (th - th.mean()) / th.std()
    return torch.polar(torch.ones_like(th), th)


def _inputs(case, seed, ny, nx):
    """(psi_true, t, y, cotangent): the object, the diffuser, the counts and model minus counts at 0.9 of the object."""
    g = torch.Generator().manual_seed(seed * 7919 + ny * 31 + nx)
    psi, t = _objects(case["batch"], ny, nx, g), _diffuser(ny, nx, g)
    M = _Model(case, ny, nx, t, torch.float32, modes=0)  # the counts of a blurred (or coherent) speckle, whatever model is fitted
    y, cot = torch.empty(psi.shape, device="cuda"), None
    if case["kind"] == "autograd":
        cot = torch.empty(psi.shape, device="cuda")
    torch.cuda.manual_seed(seed)
    for b in range(0, len(psi), 16):
        y[b:b + 16] = torch.poisson(1e4 * M.forward(psi[b:b + 16]).clamp(min=0.0)) / 1e4
        if cot is not None:
            cot[b:b + 16] = M.forward(_start(case) * psi[b:b + 16]) - y[b:b + 16]
    return psi, t, y, cot


def _plan(case, ny, nx):
    coh = 0.0 if case.get("coherent") else XCOH
    return pwf.Plan(pwf.PlanDesc(case["batch"], ny, nx, PIXEL, WAVELENGTH, L1, L2, coh, coh, GAMMA, ALPHA.real, ALPHA.imag,
                                 _eta(case), 0, case["modes"], SIGMA_PX if case["modes"] else 0.0))


class _Group:
    """Several plans joined in one group."""

    def __init__(self, plans):
        self.plans, self.handle = plans, pwf.pwf_group_create(plans)

    def __del__(self):
        pwf.pwf_group_destroy(self.handle)


def _angles(n):
    return np.arange(n) * (math.pi / n)


def _start(case):
    return 0.5 if case["kind"] == "gradient" else 0.9


def prepare(case, seed):
    kind = case["kind"]
    if kind == "fbp":
        g = torch.Generator().manual_seed(seed)
        return {"case": case, "psi": _objects(case["angles"], case["ny"], case["nx"], g), "angles": _angles(case["angles"])}
    s = {"case": case}
    data = [_inputs(case, seed, ny, nx) for ny, nx in _sizes(case)]
    plans = [_plan(case, ny, nx) for ny, nx in _sizes(case)]
    psi, t, y, cot = data[0]
    if kind == "group":
        s |= {"group": _Group(plans), "psi0": [_start(case) * d[0] for d in data], "t": [d[1] for d in data], "y": [d[2] for d in data]}
    elif kind == "solve_host":
        s |= {"plan": plans[0], "t": t.cpu().pin_memory(), "y": y.cpu().pin_memory(),
              "psi": torch.empty(psi.shape, dtype=psi.dtype).pin_memory()}
    else:
        s |= {"plan": plans[0], "psi0": _start(case) * psi, "t": t, "y": y, "cot": cot}
        if kind == "autograd":
            s["psi0"].requires_grad_(True)
            s["t"].requires_grad_(True)
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "forward":
        return s["plan"].forward(s["psi0"], s["t"])
    if kind == "gradient":
        g, loss = s["plan"].gradient(s["psi0"], s["t"], s["y"])
        return g, loss.float()  # a sum of FP32 terms: single precision is what its digits mean
    if kind == "solve":
        psi = s["psi0"].clone()
        s["plan"].solve(s["y"], s["t"], psi, case["iters"], read_back=False)
        return psi
    if kind == "solve_host":
        iters, _ = s["plan"].solve_host(s["y"], s["t"], s["psi"], case["iters"], psi_is_input=False)
        return s["psi"], iters
    if kind == "group":
        psis = [p.clone() for p in s["psi0"]]
        pwf.pwf_group_solve(s["group"].handle, s["y"], s["t"], psis, case["iters"])
        return psis
    if kind == "autograd":
        f = physical_model(s["psi0"], s["t"], s["plan"])
        return (f.detach(), *torch.autograd.grad(f, (s["psi0"], s["t"]), s["cot"]))
    return pwf.pwf_fbp(s["psi"], s["angles"], WAVELENGTH, PIXEL)


def work(case):
    """Inputs read once and outputs written once; the real operations of the transforms that the method's filters need
    (5 N log2 N for a complex one) and of the back projection (a linear interpolation and a sum, complex)."""
    if case["kind"] == "fbp":
        a, ny, nx = case["angles"], case["ny"], case["nx"]
        return {"bytes": 8.0 * (a * ny * nx + ny * nx * nx),
                "flops": 8.0 * a * ny * nx * nx + a * ny * 2 * 5.0 * 2 * nx * math.log2(2 * nx)}
    total = {"bytes": 0.0, "flops": 0.0}
    for ny, nx in _sizes(case):
        px, k = case["batch"] * ny * nx, max(1, case["modes"])
        fft = 5.0 * px * math.log2(ny * nx)
        blur = 0 if case.get("coherent") or case["modes"] else 1  # real filters of the intensity: half a complex transform pair each
        ffts = {"forward": 4 * k + blur, "gradient": 8 * k + 2 * blur, "autograd": 8 * k + 2 * blur}.get(case["kind"], 8 * k + 2 * blur + 2)
        per_px = {"forward": 8 + 4, "gradient": 8 + 4 + 8, "autograd": 8 + 4 + 4 + 8, "solve_host": 4 + 8}.get(case["kind"], 8 + 4 + 8)
        total["bytes"] += per_px * px + 8.0 * ny * nx * (2 if case["kind"] == "autograd" else 1)
        total["flops"] += ffts * fft * case.get("iters", 1)
    return total


# ---- the method in 64 bits -------------------------------------------------------------------------------------------
def _hermite(k):
    """Nodes and weights of the Gauss-Hermite rule for the standard normal density, k points."""
    x, w = np.polynomial.hermite_e.hermegauss(k)
    return x, w / w.sum()


class _Model:
    """Eq. (1) and its reverse sweep for one grid and diffuser: angular-spectrum propagators Q (piston dropped), the
    IOTF of Eq. (5) or the weighted tilted source modes, the preconditioner of Eq. (11), the window of Eqs. (14)-(15)."""

    def __init__(self, case, ny, nx, t, real, modes=None):
        k = case["modes"] if modes is None else modes
        coh = 0.0 if case.get("coherent") else XCOH
        u = torch.fft.fftfreq(nx, PIXEL, dtype=torch.float64, device="cuda")[None, :]
        v = torch.fft.fftfreq(ny, PIXEL, dtype=torch.float64, device="cuda")[:, None]
        rho2 = u * u + v * v
        cplx = torch.complex128 if real == torch.float64 else torch.complex64
        phase = -rho2 / (1.0 / WAVELENGTH + torch.sqrt(WAVELENGTH ** -2 - rho2)) * 2.0 * math.pi
        self.q1, self.q2 = (torch.polar(torch.ones_like(phase), phase * L).to(cplx) for L in (L1, L2))
        self.iotf = None if coh == 0.0 or k else torch.exp(-0.5 * math.pi * rho2 * coh ** 2).to(real)
        self.window = (-torch.expm1(-math.pi * GAMMA * rho2 * coh ** 2)).to(real)
        p2 = rho2 * PIXEL ** 2
        self.pinv = torch.where(p2 > 0, 1.0 / p2.clamp(min=1e-30), torch.zeros_like(p2)).to(real)
        self.t, self.maxt2 = t.detach().to(cplx), float(t.detach().to(cplx).abs().square().max())
        self.modes = [(0, 0, 1.0)]
        if k:
            z, (xs, ws) = WAVELENGTH * (L1 + L2), _hermite(math.isqrt(k))
            self.modes = [(int(np.rint(SIGMA_PX * a * PIXEL / z * nx * PIXEL)), int(np.rint(SIGMA_PX * b * PIXEL / z * ny * PIXEL)), wa * wb)
                          for b, wb in zip(xs, ws) for a, wa in zip(xs, ws)]

    @staticmethod
    def _filter(x, w):
        return torch.fft.ifft2(torch.fft.fft2(x) * w)

    def _real(self, x):
        return x if self.iotf is None else self._filter(x, self.iotf).real

    def _fields(self, X, mx, my):
        """(P1{x s}, P2{t P1{x s}}) of one mode: a tilt by whole bins shifts the spectrum X of x."""
        u1 = torch.fft.ifft2(torch.roll(X, (my, mx), (-2, -1)) * self.q1)
        return u1, self._filter(self.t * u1, self.q2)

    def forward(self, psi):
        X = torch.fft.fft2(torch.exp(psi))
        return self._real(sum(w * self._fields(X, mx, my)[1].abs().square() for mx, my, w in self.modes))

    def pullback(self, psi, df):
        """dl/dconj(psi) and dl/dconj(t) (per projection) of a real l with dl/df = df."""
        x = torch.exp(psi)
        X, dI = torch.fft.fft2(x), self._real(df)
        dX, dt = torch.zeros_like(X), torch.zeros_like(X)
        for mx, my, w in self.modes:
            u1, v = self._fields(X, mx, my)
            du2 = self._filter(w * dI * v, self.q2.conj())
            dt += u1.conj() * du2
            dX += torch.roll(torch.fft.fft2(self.t.conj() * du2) * self.q1.conj(), (-my, -mx), (-2, -1))
        return x.conj() * torch.fft.ifft2(dX), dt

    def gradient(self, psi, y):
        """The search direction g and the loss of Eq. (2)."""
        e = self.forward(psi) - y
        return self.pullback(psi, e)[0] / self.maxt2, e.square().sum((-2, -1))

    def solve(self, psi, y, iters, eta):
        """Algorithm S1 for a fixed count."""
        phi, mu = torch.zeros_like(psi), 1.0
        for _ in range(iters):
            g, reg = self.gradient(psi, y)[0], self._filter(psi, self.window)
            d = torch.complex(g.real + ALPHA.real * reg.real, self._filter(g.imag, self.pinv).real + ALPHA.imag * reg.imag)
            new, mu_new = psi - eta * d, (1.0 + math.sqrt(1.0 + 4.0 * mu * mu)) / 2.0
            psi, phi, mu = new + ((mu - 1.0) / mu_new) * (new - phi), new, mu_new
        return psi


def _exact_fbp(psi, angles):
    """Ram-Lak filtered back projection, linear interpolation, zero outside the detector, times -lambda / (2 pi p)."""
    n_ang, ny, nx = psi.shape
    L = 2 * nx
    h = torch.zeros(L, dtype=torch.float64, device="cuda")
    odd = torch.arange(1, nx, 2, device="cuda")
    h[0], h[odd], h[L - odd] = 0.25, -1.0 / (math.pi * odd.double()) ** 2, -1.0 / (math.pi * odd.double()) ** 2
    H = torch.fft.fft(h).real
    out = torch.empty((ny, nx * nx), dtype=torch.complex128, device="cuda")
    c = torch.arange(nx, dtype=torch.float64, device="cuda") - nx / 2 + 0.5
    for y0 in range(0, ny, 64):
        q = torch.fft.ifft(torch.fft.fft(psi[:, y0:y0 + 64].to(torch.complex128), n=L) * H)[..., :nx]
        q = torch.nn.functional.pad(q.transpose(1, 2), (0, 0, 1, 2))  # [angle][sample, one zero before and two after][slice]
        acc = torch.zeros((nx * nx, q.shape[2]), dtype=torch.complex128, device="cuda")
        for a in range(n_ang):
            u = (c[None, :] * math.cos(angles[a]) + c[:, None] * math.sin(angles[a])).reshape(-1) + (nx / 2 - 0.5)
            j = torch.floor(u)
            w = (u - j)[:, None]
            j = (j.long() + 1).clamp(-1, nx + 1)  # beyond one sample outside, both taps are zero
            q0, q1 = q[a][j.clamp(min=0)], q[a][j + 1]
            acc += torch.lerp(torch.where(j[:, None] < 0, torch.zeros_like(q0), q0), q1, w.to(torch.complex128))
        out[y0:y0 + 64] = acc.T
    return out.view(ny, nx, nx) * (math.pi / n_ang * -WAVELENGTH / (2.0 * math.pi * PIXEL))


def exact(case, seed):
    kind = case["kind"]
    if kind == "fbp":
        return _exact_fbp(_objects(case["angles"], case["ny"], case["nx"], torch.Generator().manual_seed(seed)), _angles(case["angles"]))
    outs = []
    for ny, nx in _sizes(case):
        psi, t, y, cot = _inputs(case, seed, ny, nx)
        psi0, M = (_start(case) * psi).to(torch.complex128), _Model(case, ny, nx, t, torch.float64)
        parts = []
        for b in range(0, len(psi), 8):
            p, m = psi0[b:b + 8], y[b:b + 8].double()
            if kind == "forward":
                parts.append(M.forward(p))
            elif kind == "gradient":
                parts.append(M.gradient(p, m))
            elif kind == "autograd":
                dpsi, dt = M.pullback(p, cot[b:b + 8].double())
                parts.append((M.forward(p), 2.0 * dpsi, 2.0 * dt.sum(0)))
            else:
                parts.append(M.solve(torch.zeros_like(p) if kind == "solve_host" else p, m, case["iters"], _eta(case)))
        if kind == "gradient":
            return tuple(torch.cat(p) for p in zip(*parts))
        if kind == "autograd":
            f, gp, gt = zip(*parts)
            return torch.cat(f), torch.cat(gp), sum(gt)
        outs.append(torch.cat(parts))
    return outs if kind == "group" else (outs[0], None) if kind == "solve_host" else outs[0]
