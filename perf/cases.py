"""The work a user of this framework has it do, as cases whose time can be measured.

Every case goes through the public entry points of paper_2304_03306_gb300.ttsh: stepping one
domain with or without a recorded time series, stepping a sweep of domains as a batch, stepping
caller-owned buffers without allocation, diagnostics of a state, and the learned corrector
(forward pass, training, corrected rollout).  Sizes are those of the repository's workloads
(ttsh_inputs.WORKLOADS, ttsh_inputs.sweep_domains, corrector.py, the tests); draw() spreads
further cases over the same ranges.

Values that a single-precision domain hands out as double-precision host arrays are exact
copies of single-precision values; run() returns them in the domain's own precision.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2304_03306_gb300 import ttsh

TABLE1 = dict(a=0.5, b=1.6, lam=9.0, gamma_v=40.0, gamma_w=4.0)


# ---------------------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------------------
def _step(name, n, dx, radius, precision, steps, every=0, tuned=False, amplitude=0.01, dt=0.01):
    c = dict(kind="step", n=n, dx=dx, radius=radius, precision=precision, steps=steps, every=every,
             tuned=tuned, amplitude=amplitude, dt=dt)
    return dict(c, name=name) if name else c


def _noalloc(name, n, dx, radius, precision, steps, amplitude=0.3):
    c = dict(kind="noalloc", n=n, dx=dx, radius=radius, precision=precision, steps=steps, amplitude=amplitude, dt=0.01)
    return dict(c, name=name) if name else c


def _sweep(name, ndom, steps, precision=32):
    c = dict(kind="sweep", ndom=ndom, steps=steps, precision=precision, amplitude=0.01)
    return dict(c, name=name) if name else c


def _diag(name, n, dx, radius, precision, nbins):
    c = dict(kind="diag", n=n, dx=dx, radius=radius, precision=precision, nbins=nbins, amplitude=0.3, dt=0.01)
    return dict(c, name=name) if name else c


def _fno(name, kind, n, modes, layers, batch, iters=0):
    c = dict(kind=kind, n=n, modes=modes, layers=layers, batch=batch, iters=iters)
    return dict(c, name=name) if name else c


def _rollout(name, n, dx, radius, modes, layers, steps, every):
    c = dict(kind="rollout", n=n, dx=dx, radius=radius, modes=modes, layers=layers, steps=steps, every=every,
             precision=32, amplitude=0.3, dt=0.04)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one step of a small double-precision state in the caller's buffers: the smallest call
        _noalloc("noalloc64_fp64", 64, 0.25, 5.2, 64, 1),
        # a burst of steps inside a caller's own loop (its memory pool, no allocation)
        _noalloc("noalloc256_fp32", 256, 0.08, 5.4, 32, 25),
        # the flagship run: oscillating vortex pair at 512^2, energy, enstrophy and order
        # parameter recorded every 10 steps, tile shapes autotuned once, state checkpointed
        _step("circle512_fp32_recorded", 512, 0.04, 5.4, 32, 200, every=10, tuned=True),
        # the same domain in double precision (reference runs, parity)
        _step("circle512_fp64", 512, 0.04, 5.4, 64, 50),
        # the transient of a hysteresis stage at 1024^2, default tile shapes
        _step("circle1024_fp32", 1024, 0.02, 5.32, 32, 100),
        # the turbulent case
        _step("circle2048_fp32", 2048, 0.02, 12.0, 32, 100, tuned=True),
        # the paper's production grid, series recorded, state checkpointed
        _step("circle8192_fp32_recorded", 8192, 0.005, 12.0, 32, 100, every=10),
        # the radius and dumbbell sweep: 48 domains of 128^2 to 512^2 advanced together
        _sweep("sweep48_fp32", 48, 160),
        # observables and shell spectrum of a turbulent state
        _diag("diagnostics2048_fp32", 2048, 0.02, 12.0, 32, 513),
        # the corrector network as configured: one state forward
        _fno("corrector_forward256_b1", "fno_forward", 256, 16, 4, 1),
        # its training: mini-batches of 8 samples, loss, gradients, Adam
        _fno("corrector_train256_b8", "fno_train", 256, 16, 4, 8, iters=4),
        # coarse solver corrected after every step
        _rollout("corrected_rollout256", 256, 0.08, 5.5, 16, 4, 50, 1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "noalloc", "sweep", "diag", "fno_forward", "fno_train", "rollout"])
    box = rng.uniform(16.0, 41.0)
    frac = rng.uniform(0.22, 0.32)
    if kind == "step":
        precision = rng.choice([32, 32, 64])
        n = 2 ** rng.randint(6, 12 if precision == 32 else 10)
        most = min(200, max(4, int((2.4e9 if precision == 32 else 1.2e8) / (n * n))))
        return _step(None, n, box / n, frac * box, precision, _log_int(rng, 2, most) | 1, every=rng.choice([0, 0, 1, 7, 10, 100]),
                     tuned=rng.random() < 0.4)
    if kind == "noalloc":
        precision = rng.choice([32, 64])
        n = 2 ** rng.randint(4, 9)
        return _noalloc(None, n, box / n, frac * box, precision, _log_int(rng, 1, 40))
    if kind == "sweep":
        precision = rng.choice([32, 32, 32, 64])
        return _sweep(None, rng.randint(3, 48), _log_int(rng, 5, 160 if precision == 32 else 20), precision)
    if kind == "diag":
        n = 2 ** rng.randint(6, 12)
        return _diag(None, n, box / n, frac * box, rng.choice([32, 64]) if n <= 1024 else 32, rng.choice([0, 33, n // 4 + 1]))
    n = 2 ** rng.randint(5, 9)
    modes = rng.choice([m for m in (4, 6, 8, 12, 16) if 4 * m <= n])
    layers = rng.randint(1, 4)
    if kind == "fno_forward":
        return _fno(None, kind, n, modes, layers, rng.randint(1, 8))
    if kind == "fno_train":
        return _fno(None, kind, n, modes, layers, rng.randint(1, 8 if n <= 256 else 2), iters=rng.randint(1, 5))
    return _rollout(None, n, box / n, frac * box, modes, layers, rng.randint(3, 60), rng.choice([1, 1, 2, 5]))


# ---------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(1000003 + int(seed))


def _mask(n, dx, radius, sep=0.0):
    """1 = outside: a disc, or the union of two discs `sep` apart along x."""
    c = (torch.arange(n, device="cuda", dtype=torch.float64) - n // 2) * dx
    y2 = c[:, None] ** 2
    out = (c[None, :] - 0.5 * sep) ** 2 + y2 >= radius * radius
    if sep:
        out &= (c[None, :] + 0.5 * sep) ** 2 + y2 >= radius * radius
    return out


def _noise(mask, amplitude, gen):
    """The paper's random initial state: uniform velocity noise inside the domain."""
    n = mask.shape[0]
    v = torch.rand((2, n, n), device="cuda", dtype=torch.float64, generator=gen)
    return v.mul_(2 * amplitude).sub_(amplitude).mul_(~mask)


def _sweep_domains(ndom):
    """(n, dx, radius, separation) of the sweep's members: circles across the regimes on 128^2 to
    512^2 grids, twice (forward and backward), and dumbbells; ndom of the 48 evenly spaced."""
    circles = [(128, 0.16, r, 0.0) for r in (5.0, 5.1, 5.2, 5.25, 5.3, 5.35)]
    circles += [(256, 0.08, r, 0.0) for r in (5.4, 5.6, 5.8, 6.4)] + [(512, 0.08, r, 0.0) for r in (7.2, 8.0)]
    bells = [(256, 0.08, r, r * (1.0 + 0.9 * i / 7)) for r in (2.8, math.pi, 3.5) for i in range(8)]
    every = circles + circles + bells
    return [every[i * 48 // ndom] for i in range(ndom)]


def _domain(case, mask, v, dt=0.01):
    d = ttsh.Domain(mask.to(torch.uint8).cpu().numpy(), case["n"], case["dx"], precision=case["precision"], dt=dt, **TABLE1)
    torch.cuda.synchronize()   # v was made on torch's stream
    d.set_velocity_device(v[0].data_ptr(), v[1].data_ptr())
    return d


def _smooth(shape, gen):
    """Band-limited random fields of unit variance over the last two axes (float64)."""
    n = shape[-1]
    f = torch.fft.rfft2(torch.randn(shape, device="cuda", dtype=torch.float64, generator=gen))
    k = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)
    f[..., (k[:, None] ** 2 + k[None, : n // 2 + 1] ** 2) > (n / 8) ** 2] = 0
    f = torch.fft.irfft2(f, s=(n, n))
    return f / f.std(dim=(-2, -1), keepdim=True)


def _fno_inputs(case, seed):
    """Features (omega, v_x, v_y, K) scaled to unit variance, target, and the weights."""
    g = _gen(seed)
    B, n = case["batch"], case["n"]
    x = _smooth((B, 4, n, n), g)
    x[:, 3] = x[:, 3].clamp(0.0, 1.0) * 2.0
    t = _smooth((B, n, n), g)
    return x.permute(0, 2, 3, 1).float().contiguous(), t.float().contiguous(), _weights(case, g)


def _fno_shapes(case):
    m, C = case["modes"], 32
    s = [("Wp", (4, C)), ("bp", (C,))]
    for l in range(case["layers"]):
        s += [("Wr%d" % l, (2 * m, m, C, C)), ("Wi%d" % l, (2 * m, m, C, C)), ("W%d" % l, (C, C)), ("b%d" % l, (C,))]
    return s + [("Wq", (C,)), ("bq", (1,))]


def _weights(case, g):
    """Flat float32 weights: uniform +-1/sqrt(fan-in), spectral ones as after some training."""
    parts = []
    for name, shp in _fno_shapes(case):
        w = torch.rand(shp, device="cuda", dtype=torch.float64, generator=g)
        if name[:2] in ("Wr", "Wi"):
            w = (2.0 * w - 0.5) / 32 ** 2
        elif name[0] == "b":
            w = 0.1 * (2.0 * w - 1.0)
        else:
            w = (2.0 * w - 1.0) / math.sqrt(4 if name == "Wp" else 32)
        parts.append(w.reshape(-1))
    return torch.cat(parts).float()


IN_SCALE, OUT_SCALE = (0.8, 1.1, 1.1, 2.0), 200.0


def _net(case, theta, batch):
    net = ttsh.FNO(n=case["n"], width=32, modes=case["modes"], layers=case["layers"], max_batch=batch, seed=0)
    net.set_params(theta.cpu().numpy())
    return net


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("step", "diag"):
        mask = _mask(case["n"], case["dx"], case["radius"])
        d = _domain(case, mask, _noise(mask, case["amplitude"], _gen(seed)), case["dt"])
        s = dict(case=case, dom=d)
        if kind == "step":
            if case["tuned"]:
                d.autotune(iters=max(20, min(200, int(4e7 // case["n"] ** 2))))
            if case["every"]:
                s["samples"] = -(-case["steps"] // case["every"])
                s["series"] = torch.zeros((s["samples"], 5), device="cuda", dtype=torch.float64)
        torch.cuda.synchronize()
        return s
    if kind == "noalloc":
        n = case["n"]
        mask = _mask(n, case["dx"], case["radius"])
        d = _domain(case, mask, _noise(mask, case["amplitude"], _gen(seed)), case["dt"])
        dt = torch.float32 if case["precision"] == 32 else torch.float64
        K = torch.from_numpy(d.mask()).to("cuda", dt)
        w, v0 = d.spectral_state()
        ne = 2 * w.size
        at = (ne + 3) // 4 * 4   # v^(0) on the next 16-byte boundary behind the spectrum
        state = torch.zeros(at + 2, device="cuda", dtype=dt)
        state[:ne] = torch.view_as_real(torch.from_numpy(w)).reshape(-1).to("cuda", dt)
        state[at:] = torch.from_numpy(v0).to("cuda", dt)
        p = ttsh.ttsh_default_params(n=n, dx=case["dx"], precision=case["precision"], dt=case["dt"], **TABLE1)
        d.close()
        return dict(case=case, K=K, state=state, v0=state.data_ptr() + at * state.element_size(), p=p)
    if kind == "sweep":
        g = _gen(seed)
        doms = []
        for n, dx, r, sep in _sweep_domains(case["ndom"]):
            mask = _mask(n, dx, r, sep)
            doms.append(_domain(dict(case, n=n, dx=dx), mask, _noise(mask, case["amplitude"], g)))
        return dict(case=case, doms=doms, batch=ttsh.Batch(doms))
    if kind in ("fno_forward", "fno_train"):
        x, t, theta = _fno_inputs(case, seed)
        y = torch.zeros_like(t)
        return dict(case=case, net=_net(case, theta, case["batch"]), x=x, t=t, y=y)
    g = _gen(seed)
    mask = _mask(case["n"], case["dx"], case["radius"])
    d = _domain(case, mask, _noise(mask, case["amplitude"], g), case["dt"])
    net = _net(case, _weights(case, g), 1)
    net.set_scales(np.array(IN_SCALE, np.float32), OUT_SCALE)
    return dict(case=case, net=net, dom=d, scratch=torch.zeros(5 * case["n"] ** 2, device="cuda"))


# ---------------------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------------------
def _checkpoint(dom, precision):
    """The state as a user saves it: omega^ and, behind it, the mean flow."""
    w, v0 = dom.spectral_state()
    out = np.empty(w.size + 1, dtype=np.complex64 if precision == 32 else np.complex128)
    out[:-1] = w.reshape(-1)
    out[-1] = complex(v0[0], v0[1])
    return out


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        d = state["dom"]
        if case["every"]:
            d.step_record(case["steps"], case["every"], state["series"].data_ptr(), state["samples"])
            out = {"state": _checkpoint(d, case["precision"])}
            out["series"] = state["series"].float() if case["precision"] == 32 else state["series"].clone()
            return out
        d.step(case["steps"])
        return {"state": _checkpoint(d, case["precision"])}
    if kind == "noalloc":
        ttsh.ttsh_step_noalloc(state["p"], state["K"].data_ptr(), state["state"].data_ptr(), state["v0"], case["steps"])
        return state["state"]
    if kind == "sweep":
        state["batch"].step(case["steps"])
        state["batch"].synchronize()
        return [_checkpoint(d, case["precision"]) for d in state["doms"]]
    if kind == "diag":
        r = state["dom"].diagnostics(nbins=case["nbins"])
        # max_div is left out: it is round-off itself
        out = {"observables": np.array([r[k] for k in ("energy", "enstrophy", "psi", "mean_vx", "mean_vy")])}
        if case["nbins"]:
            out["spectrum"] = r["spectrum"]
        return {k: v.astype(np.float32) if case["precision"] == 32 else v for k, v in out.items()}
    if kind == "fno_forward":
        state["net"].forward(state["x"].data_ptr(), state["y"].data_ptr(), case["batch"])
        return state["y"]
    if kind == "fno_train":
        net, losses = state["net"], []
        for _ in range(case["iters"]):
            loss, _ = net.loss_grad(state["x"].data_ptr(), state["t"].data_ptr(), case["batch"])
            net.adam_step(1e-3)
            losses.append(loss)
        return {"loss": np.array(losses, dtype=np.float32), "weights": net.get_params()}
    state["net"].rollout(state["dom"], case["steps"], state["scratch"].data_ptr(), case["every"])
    return {"state": _checkpoint(state["dom"], 32)}


# ---------------------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------------------
def _step_work(n, precision, steps):
    """Per step: the state read and written, the mask read; three real transforms each way (5 m
    log2 m for m complex points, the columns the 1/2 rule keeps) and the real-space terms."""
    e = 4 if precision == 32 else 8
    H, NK = n // 4 + 1, n // 2 + 1
    flops = 6 * n * 5 * (n / 2) * math.log2(n / 2) + 6 * H * 5 * n * math.log2(n) + 20 * n * n
    return dict(bytes=steps * e * (4 * H * NK + n * n), flops=steps * flops)


def _fno_work(n, modes, layers, batch):
    P, C, J = batch * n * n, 32, 2 * modes
    layer = 2 * P * C * C + 2 * 2 * P * J * C + 2 * 8 * batch * n * J * modes * C + 8 * batch * J * modes * C * C
    weights = layers * (2 * J * modes * C * C + C * C + C)
    return layers * layer + 10 * P * C, weights


def work(case):
    kind, n = case["kind"], case.get("n", 0)
    if kind in ("step", "noalloc"):
        return _step_work(n, case["precision"], case["steps"])
    if kind == "sweep":
        w = [_step_work(m, case["precision"], case["steps"]) for m, _, _, _ in _sweep_domains(case["ndom"])]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    if kind == "diag":
        one = _step_work(n, case["precision"], 1)
        return dict(bytes=(4 if case["precision"] == 32 else 8) * 2 * (n // 4 + 1) * (n // 2 + 1), flops=one["flops"])
    flops, weights = _fno_work(n, case["modes"], case["layers"], case.get("batch", 1))
    if kind == "fno_forward":
        return dict(bytes=4 * 5 * case["batch"] * n * n + 2 * weights, flops=flops)
    if kind == "fno_train":   # inputs, weights, gradients and both moments, once an iteration
        return dict(bytes=case["iters"] * (4 * 5 * case["batch"] * n * n + 4 * 8 * weights), flops=case["iters"] * 3 * flops)
    w, reps = _step_work(n, 32, case["steps"]), case["steps"] // case["every"]
    return dict(bytes=w["bytes"] + reps * (2 * weights + 4 * 5 * n * n), flops=w["flops"] + reps * flops)


# ---------------------------------------------------------------------------------------
# The same results in 64 bits
# ---------------------------------------------------------------------------------------
class _Solver:
    """Pseudospectral integrating-factor Euler steps with torch's FFT in double precision."""

    def __init__(self, n, dx, mask, v, dt):
        self.n, self.dx, self.dt, self.M = n, dx, dt, n // 4
        f64 = dict(device="cuda", dtype=torch.float64)
        self.my = torch.fft.fftfreq(n, 1.0 / n, **f64)[:, None]
        self.mx = torch.arange(n // 2 + 1, **f64)[None, :]
        dk = 2 * math.pi / (n * dx)
        self.kx, self.ky = dk * self.mx, dk * self.my
        m2 = self.mx ** 2 + self.my ** 2
        self.k2 = dk * dk * m2
        self.keep = (m2 <= self.M ** 2) & (m2 > 0)
        self.inv = torch.where(self.keep, 1.0 / self.k2, torch.zeros_like(m2))
        self.decay = torch.where(self.keep, torch.exp((TABLE1["a"] - (1 - self.k2) ** 2) * dt), torch.zeros_like(m2))
        f = torch.fft.rfft2(mask.double(), norm="ortho")
        f[m2 > (n // 8) ** 2] = 0
        self.K = torch.fft.irfft2(f, s=(n, n), norm="ortho") ** 2
        ux, uy = self.fwd(v[0]), self.fwd(v[1])
        self.v0 = torch.stack([ux[0, 0].real, uy[0, 0].real])
        self.w = self.project(1j * (self.kx * uy - self.ky * ux))

    def fwd(self, f):
        return torch.fft.rfft2(f, norm="ortho")

    def back(self, f):
        return torch.fft.irfft2(f, s=(self.n, self.n), norm="ortho")

    def project(self, w):
        w = torch.where(self.keep, w, torch.zeros_like(w))
        w[1:, 0] = 0.5 * (w[1:, 0] + w[1:, 0].flip(0).conj())
        return w

    def fields(self):
        psi = self.w * self.inv
        return self.back(self.w), self.back(1j * self.ky * psi) + self.v0[0] / self.n, self.back(-1j * self.kx * psi) + self.v0[1] / self.n

    def step(self):
        w, vx, vy = self.fields()
        c1 = -TABLE1["b"] * (vx * vx + vy * vy) - TABLE1["gamma_v"] * self.K
        f0 = self.fwd(c1 * vx + TABLE1["lam"] * vy * w)
        f1 = self.fwd(c1 * vy - TABLE1["lam"] * vx * w)
        rhs = 1j * (self.kx * f1 - self.ky * f0) + self.fwd(-TABLE1["gamma_w"] * self.K * w)
        self.w = self.project(self.decay * (self.w + self.dt * rhs))
        self.v0 = math.exp((TABLE1["a"] - 1) * self.dt) * (self.v0 + self.dt * torch.stack([f0[0, 0].real, f1[0, 0].real]))

    def stored(self):
        """omega^ as the library stores it: columns mx = 0..N/4, entries my = 0..N/4, -N/4..-1."""
        return torch.cat([self.w[: self.M + 1, : self.M + 1], self.w[-self.M:, : self.M + 1]]).t().contiguous()

    def checkpoint(self):
        return torch.cat([self.stored().reshape(-1), torch.complex(self.v0[:1], self.v0[1:])])

    def observables(self):
        w, vx, vy = self.fields()
        n, c = self.n, (torch.arange(self.n, device="cuda", dtype=torch.float64) - self.n // 2) * self.dx
        r = torch.sqrt(c[None, :] ** 2 + c[:, None] ** 2)
        vt = torch.where(r > 0, (c[None, :] * vy - c[:, None] * vx).abs() / r.clamp_min(1e-300), torch.zeros_like(r))
        ratio = vt.sum() / torch.sqrt(vx * vx + vy * vy).sum()
        psi = (ratio - 2 / math.pi) / (1 - 2 / math.pi)
        return [float((vx * vx + vy * vy).sum() / (2 * n * n)), float((w * w).sum() / (2 * n * n)), float(psi)]

    def spectrum(self, nbins):
        m = torch.sqrt(self.mx ** 2 + self.my ** 2)
        e = (self.w.real ** 2 + self.w.imag ** 2) * self.inv
        e[0, 0] = (self.v0 ** 2).sum()
        e = e * torch.where(self.mx > 0, 2.0, 1.0)
        s = torch.floor(m + 0.5).long()
        out = torch.zeros(max(nbins, int(s.max()) + 1), device="cuda", dtype=torch.float64)
        out.index_add_(0, s.reshape(-1), e.reshape(-1))
        return (out / (2 * self.n ** 2))[:nbins]


def _parameters(case, theta):
    out, o = {}, 0
    for name, shp in _fno_shapes(case):
        k = math.prod(shp)
        out[name] = theta[o:o + k].reshape(shp)
        o += k
    return out


def _network(case, theta, x):
    """The Fourier neural operator with torch's FFT, in the precision of its arguments."""
    n, m, L = case["n"], case["modes"], case["layers"]
    p = _parameters(case, theta)
    h = x @ p["Wp"] + p["bp"]
    rows = torch.cat([torch.arange(m), torch.arange(n - m, n)]).to(h.device)
    for l in range(L):
        H = torch.fft.rfft2(h, dim=(1, 2))[:, rows][:, :, :m]
        Y = torch.einsum("bykc,ykco->byko", H, torch.complex(p["Wr%d" % l], p["Wi%d" % l]))
        full = torch.zeros((h.shape[0], n, n // 2 + 1, 32), device=h.device, dtype=Y.dtype)
        full = _placed(full, rows, m, Y)
        z = h @ p["W%d" % l] + p["b%d" % l] + torch.fft.irfft2(full, s=(n, n), dim=(1, 2))
        h = torch.nn.functional.gelu(z) if l + 1 < L else z
    return h @ p["Wq"] + p["bq"]


def _placed(full, rows, m, Y):
    full = full.clone()
    full[:, rows[:m], :m] = Y[:, :m]
    full[:, rows[m:], :m] = Y[:, m:]
    return full


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "diag", "noalloc"):
        if case.get("steps", 1) * float(case["n"]) ** 2 > 1.2e10:
            return None
        mask = _mask(case["n"], case["dx"], case["radius"])
        s = _Solver(case["n"], case["dx"], mask, _noise(mask, case["amplitude"], _gen(seed)), case["dt"])
        if kind == "diag":
            o = s.observables() + [float(s.v0[0]) / s.n, float(s.v0[1]) / s.n]
            out = {"observables": np.array(o)}
            if case["nbins"]:
                out["spectrum"] = s.spectrum(case["nbins"]).cpu().numpy()
            return out
        series = []
        for i in range(case["steps"]):
            if case.get("every") and i % case["every"] == 0:
                series.append([float(i)] + s.observables() + [0.0])
            s.step()
        if kind == "noalloc":
            flat = torch.view_as_real(s.stored()).reshape(-1)
            pad = torch.zeros(-flat.numel() % 4, device="cuda", dtype=torch.float64)
            return torch.cat([flat, pad, s.v0])
        out = {"state": s.checkpoint().cpu().numpy()}
        if case["every"]:
            out["series"] = torch.tensor(series, dtype=torch.float64)
        return out
    if kind == "sweep":
        members = _sweep_domains(case["ndom"])
        if case["steps"] * sum(m[0] ** 2 + 2e4 for m in members) > 2e10:
            return None
        g, out = _gen(seed), []
        for n, dx, r, sep in members:
            mask = _mask(n, dx, r, sep)
            s = _Solver(n, dx, mask, _noise(mask, case["amplitude"], g), 0.01)
            for _ in range(case["steps"]):
                s.step()
            out.append(s.checkpoint().cpu().numpy())
        return out
    if kind == "rollout":
        g = _gen(seed)
        mask = _mask(case["n"], case["dx"], case["radius"])
        s = _Solver(case["n"], case["dx"], mask, _noise(mask, case["amplitude"], g), case["dt"])
        theta = _weights(case, g).double()
        scale = torch.tensor(IN_SCALE, dtype=torch.float64, device="cuda")
        for i in range(case["steps"]):
            s.step()
            if (i + 1) % case["every"] == 0:
                x = torch.stack([*s.fields(), s.K], dim=-1)[None] * scale
                s.w = s.w + s.project(s.fwd(_network(case, theta, x)[0] / OUT_SCALE))
        return {"state": s.checkpoint().cpu().numpy()}
    x, t, theta = _fno_inputs(case, seed)
    x, t, theta = x.double(), t.double(), theta.double()
    if kind == "fno_forward":
        return _network(case, theta, x)
    mom, var, losses = torch.zeros_like(theta), torch.zeros_like(theta), []
    for i in range(case["iters"]):
        theta.requires_grad_(True)
        loss = ((_network(case, theta, x) - t) ** 2).mean()
        (grad,) = torch.autograd.grad(loss, theta)
        theta = theta.detach()
        losses.append(float(loss))
        mom = 0.9 * mom + 0.1 * grad
        var = 0.999 * var + 0.001 * grad * grad
        theta = theta - 1e-3 * (mom / (1 - 0.9 ** (i + 1))) / (torch.sqrt(var / (1 - 0.999 ** (i + 1))) + 1e-8)
    return {"loss": np.array(losses), "weights": theta}
