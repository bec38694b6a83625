"""The work that a user of this library has it do, as cases to be timed.

Every case goes through the package's public entry points on plans made beforehand, as a
user's program does.  Grid sizes are the supported ones, from 16 cubed to 512 cubed (a plan of
1024 cubed holds 97 GB, so that three of them do not fit the card), cells of 2 to 4 Mpc/h as in
the configurations of `workloads`, |f_R0| from 1e-6 to 1e-4.

Shell power spectra are reduced from FP32 fields and so good to FP32; the programs here keep
them, and the derivative in ln|f_R0|, in FP32 (`.float()`), as a loss or an emulator's table does.

Two outputs of the library are discontinuous: a position at the edge of the periodic box, and
the gradient of a CIC density where a particle crosses a cell face.  The programs that return
them are the small ones, where no particle of the realisation lies within a rounding of
either; the larger ones return the density, the displacements, and gradients through a
cotangent of the positions.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1909_06282_gb300 as L
import workloads as W

SIZES = (16, 32, 64, 96, 128, 192, 256, 512)
SUPPORTED_BATCH = (32, 64, 96, 128, 192)
N_STEPS = 1024          # growth integration steps of every plan here (the library's default)


# ------------------------------------------------------------------------- cases
def listed():
    return [
        # one small realisation to positions, density and P(k): launches and latency count
        {"name": "fwd_64", "kind": "fwd", "n": 64, "box": 256.0, "fr0": 1e-5, "shells": 32, "pos": True},
        # the throughput workload: 512 cubed, Philox noise to CIC density and P(k)
        {"name": "fwd_512", "kind": "fwd", "n": 512, "box": 1024.0, "fr0": 1e-5, "shells": 32, "pos": False},
        # initial conditions: first- and second-order displacements of a given noise field
        {"name": "ics_256", "kind": "ics", "n": 256, "box": 1024.0, "fr0": 1e-5},
        # one realisation seen at several redshifts: P(k) at five output times
        {"name": "times_128", "kind": "times", "n": 128, "box": 512.0, "fr0": 1e-4, "shells": 32, "times": 5},
        # one step of a field-level fit through autograd: density + P(k) loss, both gradients
        {"name": "train_32", "kind": "train", "n": 32, "box": 128.0, "fr0": 1e-5, "shells": 16},
        # forward and adjoint at the size of the throughput workload: a loss of the positions
        {"name": "grad_512", "kind": "grad", "n": 512, "box": 1024.0, "fr0": 1e-5},
        # the batched configuration: 96 realisations of mixed grids in one plan, graph replayed
        {"name": "batch_96", "kind": "batch", "sizes": "96,128,192", "count": 32, "cell": 4.0, "shells": 32},
        # many small realisations at once (covariances, emulator tables)
        {"name": "batch_small", "kind": "batch", "sizes": "32", "count": 64, "cell": 4.0, "shells": 16},
        # P(k) of a particle set by the interlaced, window-corrected estimator; a radix-3 grid
        {"name": "est_192", "kind": "est", "n": 192, "box": 768.0, "shells": 48, "interlace": True, "deconvolve": True},
        # the transforms by themselves, both directions
        {"name": "fft_256", "kind": "fft", "n": 256, "box": 512.0},
        # one point of a scan over |f_R0|: new growth tables, then the forward map
        {"name": "scan_64", "kind": "scan", "n": 64, "box": 256.0, "fr0": 3e-6, "shells": 32},
    ]


def draw(rng):
    """One more case of the same ranges: the kind, the grid among those its listed case stands
    for, the cell and |f_R0| anywhere between their ends (logarithmically), odd shell counts."""
    kind = rng.choice(("fwd", "ics", "times", "train", "grad", "batch", "est", "fft", "scan"))
    cell = math.exp(rng.uniform(math.log(2.0), math.log(4.0)))
    fr0 = math.exp(rng.uniform(math.log(1e-6), math.log(1e-4)))
    top = {"fwd": 512, "ics": 256, "times": 256, "train": 32, "grad": 512, "est": 256, "fft": 512, "scan": 128}
    if kind == "batch":
        few = sorted(rng.sample(SUPPORTED_BATCH, rng.randint(1, 3)))
        # at most the listed batch's particles
        most = int(32 * (96 ** 3 + 128 ** 3 + 192 ** 3) / sum(n ** 3 for n in few))
        return {"kind": kind, "sizes": ",".join(str(n) for n in few), "count": rng.randint(2, min(48, most)),
                "cell": cell, "shells": rng.randint(5, 40)}
    n = rng.choice([m for m in SIZES if m <= top[kind]])
    c = {"kind": kind, "n": n, "box": n * cell}
    if kind in ("fwd", "ics", "times", "train", "grad", "scan"):
        c["fr0"] = fr0
    if kind in ("fwd", "times", "train", "est", "scan"):
        c["shells"] = rng.randint(5, max(6, n // 2 - 1)) if n <= 128 else rng.randint(5, 128)
    if kind == "fwd":
        c["pos"] = n <= 64
    if kind == "times":
        c["times"] = rng.randint(2, 6)
    if kind == "est":
        c["interlace"], c["deconvolve"] = rng.random() < 0.5, rng.random() < 0.5
    return c


# ------------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 13)


def _noise(n, seed):
    return torch.randn((n, n, n), generator=_gen(seed), device="cuda", dtype=torch.float32)


def _philox_seed(seed):
    return (int(seed) * 0x9E3779B97F4A7C15 + 1) & (2 ** 64 - 1)


def _instance(case, seed):
    return W.Instance(int(case["n"]), float(case["box"]), _philox_seed(seed), W.COSMO.replace(fr0_abs=float(case["fr0"])))


def _batch_instances(case, seed):
    rng = np.random.default_rng(int(seed))
    out = []
    for n in (int(s) for s in case["sizes"].split(",")):
        for _ in range(int(case["count"])):
            fr0 = float(np.exp(rng.uniform(np.log(1e-6), np.log(1e-4))))
            out.append(W.Instance(n, n * float(case["cell"]), int(rng.integers(1, 2 ** 62)), W.COSMO.replace(fr0_abs=fr0)))
    return out


def _out_times(case):
    return [float(a) for a in np.linspace(0.35, 1.0, int(case["times"]))]


def _particles(n, box, seed):
    """Cell corners with a Gaussian jitter of three cells, in the box (`workloads.random_positions`)."""
    i = torch.arange(n, device="cuda", dtype=torch.float64) * (box / n)
    q = torch.stack(torch.meshgrid(i, i, i, indexing="ij"))
    q += torch.randn(q.shape, generator=_gen(seed), device="cuda", dtype=torch.float32) * (3.0 * box / n)
    x = torch.remainder(q, box).float()
    return torch.where(x >= box, torch.zeros_like(x), x).contiguous()


def _train_target(n, box, shells, seed):
    """A clustered target field (log-normal) and a falling target spectrum."""
    g = torch.fft.rfftn(_noise(n, seed + 500009).double())
    m, mz = _modes(n)
    n2 = m[:, None, None] ** 2 + m[None, :, None] ** 2 + mz[None, None, :] ** 2
    f = torch.fft.irfftn(g * torch.exp(-n2 * (2.0 / n) ** 2 * 4.0), s=(n, n, n))
    rho = torch.exp(f / f.std())
    k = (torch.arange(shells, device="cuda", dtype=torch.float64) + 0.5) * (math.pi * n / box / shells)
    return (rho / rho.mean() - 1.0).float(), torch.log(500.0 / (0.1 + k)).float()


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": case}
    if kind == "batch":
        s["stream"] = torch.cuda.Stream()
        with torch.cuda.stream(s["stream"]):
            s["plan"] = L.Plan(_batch_instances(case, seed), n_steps=N_STEPS, stream=s["stream"], graph=True)
    elif kind in ("est", "fft"):
        s["plan"] = L.Plan(W.Instance(int(case["n"]), float(case["box"]), 1, W.COSMO), n_steps=N_STEPS)
    else:
        s["plan"] = L.Plan(_instance(case, seed), n_steps=N_STEPS, keep_state=kind == "train",
                           max_outputs=int(case.get("times", 0)))
    n = int(case.get("n", 0))
    if kind in ("ics", "grad", "train"):
        s["noise"] = _noise(n, seed)
    if kind == "times":
        L.lpt2_set_outputs(s["plan"], _out_times(case))
    if kind == "grad":   # the cotangent of a mean-square loss of positions a few cells off
        s["g_pos"] = torch.randn((3, n, n, n), generator=_gen(seed + 900001), device="cuda", dtype=torch.float32) / n ** 3
    if kind == "train":
        s["noise"].requires_grad_(True)
        s["log_fr0"] = torch.tensor(math.log(float(case["fr0"])), device="cuda", requires_grad=True)
        s["target"], s["target_lnp"] = _train_target(n, float(case["box"]), int(case["shells"]), seed)
    if kind == "est":
        s["pos"] = _particles(n, float(case["box"]), seed)
    if kind == "fft":
        s["field"] = _noise(n, seed)
        s["spec"] = torch.fft.rfftn(_noise(n, seed + 500009))[..., : n // 2].contiguous()
    return s


# ------------------------------------------------------------------------- passes
def run(s):
    kind, case, plan = s["kind"], s["case"], s["plan"]
    if kind == "fwd":
        return _forward(plan, case)
    if kind == "scan":
        L.lpt2_set_fr0(plan, float(case["fr0"]))
        return _forward(plan, case)
    if kind == "ics":
        return L.lpt2_displace(plan, noise=s["noise"], psi1=True, psi2=True, pos=False)
    if kind == "times":
        r = L.lpt2_displace_outputs(plan, pos=False, n_shells=int(case["shells"]))
        return {"pk": r["pk"].float(), "k_mean": r["k_mean"], "n_modes": r["n_modes"]}
    if kind == "train":
        s["noise"].grad = s["log_fr0"].grad = None
        density, pk = L.Displace.apply(s["noise"], s["log_fr0"], plan, int(case["shells"]))
        loss = (density - s["target"]).square().mean() + (torch.log(pk[1:].float()) - s["target_lnp"][1:]).square().sum()
        loss.backward()
        return {"loss": loss.detach(), "g_noise": s["noise"].grad, "g_log_fr0": s["log_fr0"].grad}
    if kind == "grad":
        g_noise, g_log_fr0 = L.lpt2_displace_vjp(plan, noise=s["noise"], g_pos=s["g_pos"])
        return {"g_noise": g_noise, "g_log_fr0": g_log_fr0.float()}
    if kind == "batch":
        with torch.cuda.stream(s["stream"]):
            L.lpt2_displace(plan, psi1=False, psi2=False, pos=False)
            return _summary(L.lpt2_cic_pk(plan, density=True, n_shells=int(case["shells"])))
    if kind == "est":
        return _summary(L.lpt2_cic_pk_est(plan, pos=s["pos"], density=True, n_shells=int(case["shells"]),
                                          deconvolve=bool(case["deconvolve"]), interlace=bool(case["interlace"])))
    if kind == "fft":
        return {"spectrum": L.lpt2_fft_r2c(plan, s["field"]), "field": L.lpt2_fft_c2r(plan, s["spec"])}
    raise ValueError(kind)


def _forward(plan, case):
    out = L.lpt2_displace(plan, psi1=False, psi2=False, pos=bool(case.get("pos", False)))
    out.update(_summary(L.lpt2_cic_pk(plan, density=True, n_shells=int(case["shells"]))))
    return out


def _summary(r):
    return {"density": r["density"], "pk": r["pk"].float(), "k_mean": r["k_mean"], "n_modes": r["n_modes"]}


# ------------------------------------------------------------------------- work
def work(case):
    """Inputs read once and outputs written once; the transforms of real fields at
    2.5 N^3 log2(N^3) operations, 60 per particle deposited or gathered, 200 per noise draw."""
    kind = case["kind"]

    def fft(n, count):
        return 2.5 * n ** 3 * math.log2(float(n) ** 3) * count

    if kind == "batch":
        ns = [int(v) for v in case["sizes"].split(",")]
        c = int(case["count"])
        return {"bytes": c * sum(4.0 * n ** 3 for n in ns), "flops": c * sum(fft(n, 12) + 280.0 * n ** 3 for n in ns)}
    n = int(case["n"])
    v = 4.0 * n ** 3
    if kind in ("fwd", "scan"):
        return {"bytes": v * (4 if case.get("pos") else 1), "flops": fft(n, 12) + 280.0 * n ** 3}
    if kind == "ics":
        return {"bytes": 7 * v, "flops": fft(n, 14) + 20.0 * n ** 3}
    if kind == "times":
        t = int(case["times"])
        return {"bytes": t * 20.0 * int(case["shells"]), "flops": fft(n, 8 + 4 * t) + (220.0 + 60.0 * t) * n ** 3}
    if kind == "train":
        return {"bytes": 4 * v, "flops": fft(n, 12 + 14) + 160.0 * n ** 3}
    if kind == "grad":
        return {"bytes": 5 * v, "flops": fft(n, 8 + 11) + 60.0 * n ** 3}
    if kind == "est":
        g = 2 if case["interlace"] else 1
        return {"bytes": 4 * v, "flops": fft(n, g) + 60.0 * g * n ** 3}
    return {"bytes": 4 * v, "flops": fft(n, 2)}


# ------------------------------------------------------------------------- in 64 bits
# The same maps in float64 torch with library transforms, written from the paper's equations.
H0C = 1.0 / 2997.92458


def _modes(n):
    m = torch.fft.fftfreq(n, d=1.0 / n, device="cuda", dtype=torch.float64)
    return m, torch.arange(n // 2 + 1, device="cuda", dtype=torch.float64)


def _growth(fr0, a_out, tangents=False):
    """D1, D2 (and d/dln|f_R0|) [len(fr0), 512] of the orthogonal triangle by RK4 in ln a."""
    c = W.COSMO
    dev = "cpu" if len(fr0) <= 4 else "cuda"
    k = torch.as_tensor(W.K_MIN * (W.K_MAX / W.K_MIN) ** (np.arange(W.N_K) / (W.N_K - 1.0)), device=dev)[None, :]
    f = torch.as_tensor(np.asarray(fr0, dtype=np.float64), device=dev)[:, None]
    x0 = c.omega_m + 4 * c.omega_l

    def background(s):
        a = math.exp(s)
        om = c.omega_m * a ** -3 / (c.omega_m * a ** -3 + c.omega_l)
        x = c.omega_m * a ** -3 + 4 * c.omega_l
        m2 = 0.5 * H0C ** 2 * x ** 3 / (f * x0 ** 2)
        big = (2.0 / 27.0) * 1.5 * c.omega_m * a ** -3 * H0C ** 2 * 2.25 * H0C ** 2 * x ** 5 / (f ** 2 * x0 ** 4)
        q = k * k / a ** 2
        p, ph = q + m2, 0.5 * q + m2
        mu, muh, b = 1 + q / (3 * p), 1 + 0.5 * q / (3 * ph), big * q / (p * ph * ph)
        mut, muht = q * m2 / (3 * p * p), 0.5 * q * m2 / (3 * ph * ph)
        return 2 - 1.5 * om, 1.5 * om, mu, muh, mu - b, mut, muht, mut - b * (-2 + m2 / p + 2 * m2 / ph)

    def rhs(bg, y):
        damp, cc, mu, muh, br, mut, muht, brt = bg
        d = [y[1], -damp * y[1] + cc * mu * y[0], y[3], -damp * y[3] + cc * muh * y[2],
             y[5], -damp * y[5] + cc * (mu * y[4] - y[2] * y[2] * br)]
        if tangents:
            d += [y[7], -damp * y[7] + cc * (mu * y[6] + mut * y[0]), y[9], -damp * y[9] + cc * (muh * y[8] + muht * y[2]),
                  y[11], -damp * y[11] + cc * (mu * y[10] + mut * y[4] - 2 * y[2] * y[8] * br - y[2] * y[2] * brt)]
        return torch.stack(d)

    def integrate(background, rhs, y, a1):
        s0 = math.log(c.a_init)
        h = (math.log(a1) - s0) / N_STEPS
        for i in range(N_STEPS):
            b0, bm, b1 = background(s0 + i * h), background(s0 + (i + 0.5) * h), background(s0 + (i + 1) * h)
            k1 = rhs(b0, y)
            k2 = rhs(bm, y + 0.5 * h * k1)
            k3 = rhs(bm, y + 0.5 * h * k2)
            y = y + (h / 6) * (k1 + 2 * k2 + 2 * k3 + rhs(b1, y + h * k3))
        return y

    def background_gr(s):
        a3 = math.exp(-3 * s)
        om = c.omega_m * a3 / (c.omega_m * a3 + c.omega_l)
        return 2 - 1.5 * om, 1.5 * om

    y0 = np.array([c.a_init, c.a_init])
    norm = integrate(background_gr, lambda b, y: np.array([y[1], -b[0] * y[1] + b[1] * y[0]]), y0, 1.0)[0]
    one = torch.ones(len(fr0), W.N_K, dtype=torch.float64, device=dev)
    y = torch.stack([c.a_init * one] * 4 + [-3 / 7 * c.a_init ** 2 * one, -6 / 7 * c.a_init ** 2 * one]
                    + ([0 * one] * 6 if tangents else []))
    y = integrate(background, rhs, y, a_out)
    out = [y[0] / norm, y[4] / norm ** 2] + ([y[6] / norm, y[10] / norm ** 2] if tangents else [])
    return [t.cuda() for t in out]


def _transfer(k):
    """Eisenstein & Hu (1998) without wiggles, Eqs. 26 and 28-31, k in h/Mpc (a numpy array or a tensor)."""
    c, lib = W.COSMO, (torch if torch.is_tensor(k) else np)
    wm, wb, fb = c.omega_m * c.h ** 2, c.omega_b * c.h ** 2, c.omega_b / c.omega_m
    s = 44.5 * math.log(9.83 / wm) / math.sqrt(1 + 10 * wb ** 0.75)
    al = 1 - 0.328 * math.log(431 * wm) * fb + 0.38 * math.log(22.3 * wm) * fb * fb
    q = k * (c.t_cmb / 2.7) ** 2 / (c.omega_m * c.h * (al + (1 - al) / (1 + (0.43 * k * c.h * s) ** 4)))
    l0 = lib.log(2 * math.e + 1.8 * q)
    return l0 / (l0 + (14.2 + 731.0 / (1 + 62.5 * q)) * q * q)


def _amplitude():
    lnk = np.linspace(math.log(1e-5), math.log(1e3), 20001)
    k = np.exp(lnk)
    x = 8 * k
    f = k ** (3 + W.COSMO.n_s) * _transfer(k) ** 2 * (3 * (np.sin(x) - x * np.cos(x)) / x ** 3) ** 2 / (2 * math.pi ** 2)
    w = np.ones(len(k))
    w[1:-1:2], w[2:-1:2] = 4, 2
    return W.COSMO.sigma8 ** 2 / ((lnk[1] - lnk[0]) / 3 * np.dot(w, f))


def _philox_noise(n, seed):
    """The white noise of a Philox4x32-10 key: one Box-Muller pair for the cells of an even and the next odd iy."""
    lo32 = 0xFFFFFFFF
    ix, iy, iz = (torch.arange(m, device="cuda", dtype=torch.int64) for m in (n, n // 2, n))
    cell = (ix[:, None, None] * n + 2 * iy[None, :, None]) * n + iz[None, None, :]

    def mul(m, x):   # high and low words of the 64-bit product
        p0, p1 = m * (x & 0xFFFF), m * (x >> 16)
        t = p1 + (p0 >> 16)
        return t >> 16, ((t & 0xFFFF) << 16) | (p0 & 0xFFFF)

    c0, c1, c2, c3 = cell & lo32, cell >> 32, torch.zeros_like(cell), torch.zeros_like(cell)
    k0, k1 = seed & lo32, (seed >> 32) & lo32
    for r in range(10):
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & lo32, (k1 + 0xBB67AE85) & lo32
    u0, u1 = ((c0 >> 8) + 1).double() * 2.0 ** -24, ((c1 >> 8) + 1).double() * 2.0 ** -24
    del c0, c1, c2, c3, h0, l0, h1, l1, cell
    rad = torch.sqrt(-2 * torch.log(u0))
    out = torch.empty((n, n, n), device="cuda", dtype=torch.float64)
    out[:, 0::2] = rad * torch.cos(2 * math.pi * u1)
    out[:, 1::2] = rad * torch.sin(2 * math.pi * u1)
    return out


class _Grid:
    """Wave numbers, the modes that are set to zero, sqrt(P N^3/V) and table lookups of one grid."""

    def __init__(self, n, box):
        self.n, self.box = n, box
        m, mz = _modes(n)
        kf = 2 * math.pi / box
        self.k = [kf * m[:, None, None], kf * m[None, :, None], kf * mz[None, None, :]]
        self.k2 = self.k[0] ** 2 + self.k[1] ** 2 + self.k[2] ** 2
        nyq = m.abs() == n // 2
        self.zero = (nyq[:, None, None] | nyq[None, :, None] | (mz == n // 2)[None, None, :]) | (self.k2 == 0)
        self.k2 = torch.where(self.zero, torch.ones_like(self.k2), self.k2)

    def spectrum_scale(self):
        kk = torch.sqrt(self.k2)
        s = math.sqrt(_amplitude() * self.n ** 3 / self.box ** 3) * kk ** (0.5 * W.COSMO.n_s) * _transfer(kk)
        return torch.where(self.zero, torch.zeros_like(s), s)

    def lookup(self, *tables):
        lo, step = math.log(W.K_MIN), math.log(W.K_MAX / W.K_MIN) / (W.N_K - 1)
        x = ((0.5 * torch.log(self.k2) - lo) / step).clamp(0, W.N_K - 1)
        i = x.long().clamp(max=W.N_K - 2)
        x = x - i
        return [t[i] + x * (t[i + 1] - t[i]) for t in tables]

    def inverse(self, spec):
        return torch.fft.irfftn(spec, s=(self.n,) * 3)

    def derivative(self, spec, *axes):
        for a in axes:
            spec = spec * (1j * self.k[a])
        return self.inverse(spec)

    def potentials(self, noise):
        """delta(k) / k^2, S(k) / k^2 (with the modes set to zero)."""
        first = torch.fft.rfftn(noise) * (self.spectrum_scale() / self.k2)
        xx, yy, zz = (self.derivative(first, a, a) for a in range(3))
        src = xx * yy + (xx + yy) * zz
        del xx, yy, zz
        for a, b in ((0, 1), (0, 2), (1, 2)):
            src = src - self.derivative(first, a, b).square()
        second = torch.fft.rfftn(src) / self.k2
        return first, torch.where(self.zero, torch.zeros_like(second), second)

    def positions(self, potential):
        out = []
        for a in range(3):
            q = torch.arange(self.n, device="cuda", dtype=torch.float64) * (self.box / self.n)
            out.append(self.derivative(potential, a) + q.view([-1 if j == a else 1 for j in range(3)]))
        return torch.stack(out)

    def deposit(self, pos, shift=0.0):
        n = self.n
        u = pos.reshape(3, -1) * (n / self.box) + shift
        i = torch.floor(u)
        d = u - i
        i = torch.remainder(i, n).long()
        rho = torch.zeros(n ** 3, dtype=torch.float64, device="cuda")
        for c in range(8):
            o = (c >> 2, (c >> 1) & 1, c & 1)
            w = torch.ones_like(d[0])
            e = torch.zeros_like(i[0])
            for a in range(3):
                w = w * (d[a] if o[a] else 1 - d[a])
                e = e * n + torch.remainder(i[a] + o[a], n)
            rho = rho.index_add(0, e, w)
        return rho.view(n, n, n) - 1.0

    def shells(self, count):
        m, mz = _modes(self.n)
        n2 = (m[:, None, None] ** 2 + m[None, :, None] ** 2 + mz[None, None, :] ** 2).long()
        big = 4 * count * count * n2
        r = torch.sqrt(big.double()).long()
        r = torch.where((r + 1) ** 2 <= big, r + 1, r)
        r = torch.where(r * r > big, r - 1, r)
        ok = (n2 > 0) & (4 * n2 < self.n ** 2)
        w = torch.where(mz == 0, 1.0, 2.0).double()[None, None, :].expand(n2.shape)
        return (r // self.n)[ok], ok, w[ok], (2 * math.pi / self.box) * torch.sqrt(n2[ok].double())

    def power(self, spec, count, window=None):
        b, ok, w, k = self.shells(count)
        p = (spec.real.square() + spec.imag.square())[ok] * (self.box ** 3 / float(self.n) ** 6)
        if window is not None:
            p = p / window[ok]

        def total(x):
            return torch.zeros(count, dtype=torch.float64, device="cuda").index_add(0, b, x)

        modes = total(w)
        per = modes.clamp(min=1)
        return total(w * p) / per, total(w * k) / per, modes.round().long()

    def summary(self, pos, count):
        rho = self.deposit(pos)
        pk, km, nm = self.power(torch.fft.rfftn(rho), count)
        return {"density": rho, "pk": pk, "k_mean": km, "n_modes": nm}


def _exact_forward(n, box, noise, tables, shells, pos):
    g = _Grid(n, box)
    first, second = g.potentials(noise)
    d1, d2 = g.lookup(*tables)
    x = g.positions(first * d1 - second * d2)
    out = g.summary(x, shells)
    if pos:
        out["pos"] = torch.remainder(x, box)
    return out


def _exact_adjoint(case, seed):
    n, box = int(case["n"]), float(case["box"])
    g = _Grid(n, box)
    d1, d2, t1, t2 = (t[0] for t in _growth([float(case["fr0"])], 1.0, tangents=True))
    noise = _noise(n, seed).double().requires_grad_(True)
    theta = torch.zeros((), dtype=torch.float64, device="cuda", requires_grad=True)
    first, second = g.potentials(noise)
    d1, d2, t1, t2 = g.lookup(d1, d2, t1, t2)
    x = g.positions(first * (d1 + theta * t1) - second * (d2 + theta * t2))
    if case["kind"] == "grad":
        cot = torch.randn((3, n, n, n), generator=_gen(seed + 900001), device="cuda", dtype=torch.float32) / n ** 3
        loss = (cot.double() * x).sum()
    else:
        target, lnp = _train_target(n, box, int(case["shells"]), seed)
        r = g.summary(x, int(case["shells"]))
        loss = (r["density"] - target.double()).square().mean() + (torch.log(r["pk"][1:]) - lnp.double()[1:]).square().sum()
    loss.backward()
    out = {"g_noise": noise.grad, "g_log_fr0": theta.grad}
    return out if case["kind"] == "grad" else {"loss": loss.detach(), **out}


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        insts = _batch_instances(case, seed)
        d1, d2 = _growth([i.cosmo.fr0_abs for i in insts], 1.0)
        got = [_exact_forward(i.n, i.box, _philox_noise(i.n, i.seed), (d1[j], d2[j]), int(case["shells"]), False)
               for j, i in enumerate(insts)]
        out = {k: torch.stack([r[k] for r in got]) for k in ("pk", "k_mean", "n_modes")}
        out["density"] = torch.cat([r["density"].reshape(-1) for r in got])
        if len(insts) == 1:
            out = {k: v[0] if k != "density" else got[0]["density"] for k, v in out.items()}
        return out
    n, box = int(case["n"]), float(case["box"])
    if kind in ("fwd", "scan"):
        t = [v[0] for v in _growth([float(case["fr0"])], 1.0)]
        return _exact_forward(n, box, _philox_noise(n, _philox_seed(seed)), t, int(case["shells"]), bool(case.get("pos", False)))
    if kind == "ics":
        g = _Grid(n, box)
        first, second = g.potentials(_noise(n, seed).double())
        d1, d2 = g.lookup(*[v[0] for v in _growth([float(case["fr0"])], 1.0)])
        first, second = first * d1, -second * d2
        return {"psi1": torch.stack([g.derivative(first, a) for a in range(3)]),
                "psi2": torch.stack([g.derivative(second, a) for a in range(3)])}
    if kind == "times":
        g = _Grid(n, box)
        first, second = g.potentials(_philox_noise(n, _philox_seed(seed)))
        got = []
        for a in _out_times(case):
            d1, d2 = g.lookup(*[v[0] for v in _growth([float(case["fr0"])], a)])
            got.append(g.summary(g.positions(first * d1 - second * d2), int(case["shells"])))
        return {"pk": torch.stack([r["pk"] for r in got]), "k_mean": got[0]["k_mean"], "n_modes": got[0]["n_modes"]}
    if kind in ("train", "grad"):
        return _exact_adjoint(case, seed)
    if kind == "est":
        g = _Grid(n, box)
        pos = _particles(n, box, seed).double()
        rho = g.deposit(pos)
        spec = torch.fft.rfftn(rho)
        m, mz = _modes(n)
        if case["interlace"]:
            phase = (m[:, None, None] + m[None, :, None] + mz[None, None, :]) * (math.pi / n)
            spec = 0.5 * (spec + torch.fft.rfftn(g.deposit(pos, 0.5)) * torch.polar(torch.ones_like(phase), phase))
        win = None
        if case["deconvolve"]:
            sx, sz = torch.sinc(m / n) ** 4, torch.sinc(mz / n) ** 4
            win = sx[:, None, None] * sx[None, :, None] * sz[None, None, :]
        pk, km, nm = g.power(spec, int(case["shells"]), win)
        return {"density": rho, "pk": pk, "k_mean": km, "n_modes": nm}
    if kind == "fft":
        spec = torch.fft.rfftn(_noise(n, seed + 500009))[..., : n // 2].to(torch.complex128)
        spec = torch.cat([spec, torch.zeros_like(spec[..., :1])], -1)
        return {"spectrum": torch.fft.rfftn(_noise(n, seed).double())[..., : n // 2].contiguous(),
                "field": torch.fft.irfftn(spec, s=(n, n, n)) * float(n) ** 3}
    return None
