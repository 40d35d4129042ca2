"""Performance cases of the library: what a program that uses it spends its time on.

Every case is one electron-phonon system (or a batch of them) with the structure of the paper's
workloads: tight-binding bands inside an energy window, acoustic and optical phonon branches on
commensurate k/q grids, log-normal couplings and occupations out of equilibrium.  ``prepare``
builds the channel list and the device handle that a program keeps; ``run`` is one call (or one
forward and backward pass) through the public entry points.  Inputs follow from the seed alone:
the couplings, the occupations and their random part.

Kinds of pass:
  collision   one collision integral I[f] (Eq. 2)
  rates       the scattering rates 1/tau
  rk4         a few RK4 steps of the rt-BTE (a program advances f in such runs between outputs)
  transport   the whole iterative transport solve (weights at f0, then iterations to 1e-10)
  batch       RK4 steps of many small systems at once
  adjoint     loss gradient of an RK4 trajectory in f0 and in every coupling
"""
import math
import random

import numpy as np
import torch

import paper_2511_03683_gb300 as pb
from paper_2511_03683_gb300 import autograd as pa

HBAR = 0.6582119569  # eV fs
KB = 8.617333262e-5  # eV / K
BANDS = (0.0, 0.2, 1.1, 1.3)  # band offsets, eV
DT = 1.0  # fs


def listed():
    return [
        # the smallest calls: one collision integral on the 8^3 full Brillouin zone (1024 states),
        # where the launches and the host path are most of the time
        dict(name="collision-8", kind="collision", variant="ff", n1=8, n2=8, n3=8, bands=2, modes=3, window=0.0,
             sigma=0.005, T=300.0),
        # time stepping of a coarse grid, as in convergence studies: 20 dependent steps
        dict(name="rk4-16", kind="rk4", variant="ff", n1=16, n2=16, n3=16, bands=4, modes=6, window=0.3, sigma=0.008,
             T=300.0, steps=20),
        # an ordinary single call on an odd grid
        dict(name="collision-35", kind="collision", variant="ff", n1=35, n2=35, n3=35, bands=4, modes=6, window=0.3,
             sigma=0.008, T=300.0),
        # rates for a lifetime plot: uneven grid, three bands, low temperature
        dict(name="rates-29", kind="rates", variant="ff", n1=30, n2=29, n3=27, bands=3, modes=6, window=0.3, sigma=0.008,
             T=150.0),
        # the headline workload: RK4 on the 40^3 grid, FP64-accurate
        dict(name="rk4-40", kind="rk4", variant="ff", n1=40, n2=40, n3=40, bands=4, modes=6, window=0.3, sigma=0.008,
             T=300.0, steps=10),
        # the other half of the headline: the transport solve on the same grid
        dict(name="transport-40", kind="transport", variant="ff", n1=40, n2=40, n3=40, bands=4, modes=6, window=0.3,
             sigma=0.008, T=300.0),
        # the reduced-precision form for long runs: FP32 pair coefficients
        dict(name="rk4-c32-36", kind="rk4", variant="c32", n1=36, n2=36, n3=36, bands=4, modes=6, window=0.3,
             sigma=0.008, T=300.0, steps=4),
        # couplings kept as data (FP16 |g|^2, per-channel arithmetic): where they change between runs
        dict(name="collision-h16-28", kind="collision", variant="h16", n1=28, n2=28, n3=28, bands=4, modes=6,
             window=0.3, sigma=0.008, T=300.0),
        # the paper's cutoffs (delta at 6 sigma, |g|^2 >= 1e-5 eV^2): rows that miss most partners
        dict(name="rk4-cut-32", kind="rk4", variant="ff", n1=32, n2=32, n3=32, bands=4, modes=6, window=0.3,
             sigma=0.008, T=300.0, steps=10, nsigma=6.0, g2min=1e-5),
        # many uneven systems together: the FP64-accurate batch and the default FP32 one
        dict(name="batch-ff", kind="batch", precision="ff", count=16, nmin=16, nmax=26, draw=1, steps=5),
        dict(name="batch-fp32", kind="batch", precision="fp32", count=16, nmin=16, nmax=24, draw=2, steps=5),
        # fitting: gradient of a carrier-energy loss through 20 steps, all couplings among the parameters
        dict(name="adjoint-24", kind="adjoint", variant="ff", n1=24, n2=24, n3=24, bands=4, modes=6, window=0.3,
             sigma=0.008, T=300.0, steps=20),
    ]


def draw(rng):
    kind = rng.choice(["collision", "collision", "rates", "rk4", "rk4", "rk4", "transport", "transport", "batch",
                       "adjoint"])
    if kind == "batch":
        nmin = rng.randint(12, 18)
        return dict(kind="batch", precision=rng.choice(["ff", "c32", "fp32"]), count=rng.randint(3, 14), nmin=nmin,
                    nmax=rng.randint(nmin, 24), draw=rng.randint(3, 1 << 20), steps=rng.randint(1, 6))
    top = 22 if kind == "adjoint" else 34
    n = round(math.exp(rng.uniform(math.log(9 if kind == "collision" else 12), math.log(top))))
    dims = [n, n, n]
    if rng.random() < 0.4:
        dims = [max(6, n + rng.randint(-2, 1)) for _ in range(3)]
    # (the FP32 pair coefficients are the form for time stepping)
    variants = {"collision": ["ff", "ff", "ff", "g32", "h16", "f64"], "rates": ["ff", "ff", "g32"],
                "rk4": ["ff", "ff", "ff", "c32", "g32"], "transport": ["ff", "ff", "f64"], "adjoint": ["ff", "ff", "g32"]}
    c = dict(kind=kind, variant=rng.choice(variants[kind]), n1=dims[0], n2=dims[1], n3=dims[2],
             bands=rng.randint(2, 4), modes=rng.randint(3, 6), window=round(rng.uniform(0.25, 0.32), 3),
             sigma=round(rng.uniform(0.005, 0.012), 4), T=round(rng.uniform(100.0, 500.0), 1))
    if kind in ("rk4", "adjoint"):
        c["steps"] = rng.randint(1, 10) if c["variant"] == "ff" else rng.randint(1, 3)
    if kind in ("collision", "rk4") and c["variant"] == "ff" and rng.random() < 0.3:
        c["nsigma"], c["g2min"] = round(rng.uniform(4.0, 8.0), 1), 10.0 ** rng.uniform(-6.0, -4.5)
    return c


# ------------------------------------------------------------------ the model


class Model:
    """One system: bands, velocities, phonons and window on the full grid, and its window states."""

    def __init__(self, c):
        self.nk = nk = (c["n1"], c["n2"], c["n3"])
        self.nb, self.nm, self.T, self.sigma = c["bands"], c["modes"], c["T"], c["sigma"]
        t = 0.3
        j = np.stack(np.meshgrid(*[np.arange(n) for n in nk], indexing="ij"), axis=-1).reshape(-1, 3)
        fold = [np.minimum(j[:, i], (nk[i] - j[:, i]) % nk[i]) for i in range(3)]
        sign = [np.where(j[:, i] > nk[i] // 2, -1.0, 1.0) for i in range(3)]
        cosine = np.sort(np.stack([1.0 - np.cos(2 * np.pi * fold[i] / nk[i]) for i in range(3)], axis=1), axis=1)
        sine = np.stack([np.where((fold[i] == 0) | (2 * fold[i] == nk[i]), 0.0, sign[i] * np.sin(2 * np.pi * fold[i] / nk[i]))
                         for i in range(3)], axis=1)
        half = np.sort(np.stack([np.sin(np.pi * fold[i] / nk[i]) ** 2 for i in range(3)], axis=1), axis=1)
        full = c["window"] <= 0.0  # the full zone: the small two-band system
        offs = np.array([0.0, 0.5] if full else BANDS[:self.nb])
        self.eps = offs[None, :] + (2 * t * ((cosine[:, 0] + cosine[:, 1]) + cosine[:, 2]))[:, None]
        self.vel = np.repeat((2 * t / HBAR * sine)[:, None, :], self.nb, axis=1)
        s = np.sqrt(((half[:, 0] + half[:, 1]) + half[:, 2]) / 3.0)
        if full:
            self.omega = np.stack([(10.0 + 5.0 * v + 5.0 * s) * 1e-3 for v in range(self.nm)], axis=1)
            self.win = None
        else:
            br = [15e-3 * s, 20e-3 * s, 25e-3 * s] + [np.full_like(s, w) for w in (35e-3, 47.5e-3, 60e-3)]
            self.omega = np.stack(br[:self.nm], axis=1)
            self.win = np.stack([offs - 1.0, offs + c["window"]], axis=1)
        inside = np.ones(self.eps.shape, bool) if full else \
            (self.eps >= self.win[None, :, 0]) & (self.eps <= self.win[None, :, 1])
        self.ids = np.flatnonzero(inside.reshape(-1)).astype(np.int64)  # window states, ascending full-grid id
        self.e = self.eps.reshape(-1)[self.ids]
        self.v = self.vel.reshape(-1, 3)[self.ids]
        self.j = j[self.ids // self.nb]
        self.ns = len(self.ids)
        self.nsigma, self.g2min = c.get("nsigma", 0.0), c.get("g2min", 0.0)

    def couplings(self, seed):
        """|g|^2 of every (state, partner, branch) on the GPU, [ns, ns, modes] float64: log-normal,
        exp(-7 + Z) eV^2, with Z from a hash that is symmetric under exchange of the two states and
        under the symmetries of the grid (inversion; the axes' permutations where they are equal)."""
        r = np.random.default_rng([seed, 1])
        dev = "cuda"
        tables, key = {}, torch.zeros((self.ns, self.ns), dtype=torch.int64, device=dev)

        def table(n):
            if n not in tables:
                a = torch.tensor(r.integers(-(1 << 62), 1 << 62, (n, n)), device=dev)
                neg = (-torch.arange(n, device=dev)) % n
                a = a + a[neg][:, neg]
                tables[n] = a + a.T
            return tables[n]

        for i in range(3):
            ji = torch.tensor(self.j[:, i], device=dev)
            key += table(self.nk[i])[ji][:, ji]
        hb = torch.tensor(r.integers(-(1 << 62), 1 << 62, self.nb), device=dev)[torch.tensor(self.ids % self.nb, device=dev)]
        key += hb[:, None] + hb[None, :]
        hm = r.integers(-(1 << 62), 1 << 62, self.nm)
        g2 = torch.empty((self.ns, self.ns, self.nm), dtype=torch.float64, device=dev)
        shift = lambda h, n: (h >> n) & ((1 << (64 - n)) - 1)  # noqa: E731 - logical shift
        for nu in range(self.nm):
            h = key + int(hm[nu])
            h = (h ^ shift(h, 30)) * -4658895280553007687
            h = (h ^ shift(h, 27)) * -7723592293110705685
            u = (shift(h ^ shift(h, 31), 11).double() + 0.5) * 2.0 ** -53
            g2[:, :, nu] = torch.exp(torch.special.ndtri(u) - 7.0)
        return g2

    def channels(self, g2):
        """The channel list (host), its couplings looked up in the table g2."""
        host = g2.cpu().numpy().reshape(self.ns, self.ns * self.nm)
        pos = np.full(self.eps.size, -1, np.int32)
        pos[self.ids] = np.arange(self.ns, dtype=np.int32)
        nm = np.int32(self.nm)
        return pb.Channels.build(self.nk, self.nb, self.nm, self.eps, self.omega, self.T, self.sigma,
                                 lambda s, p, nu: host[pos[s[0]]].take(pos[p] * nm + nu) if len(s) else np.empty(0),
                                 vel=self.vel, win=self.win, g2_min=self.g2min, delta_nsigma=self.nsigma)

    def occupations(self, seed, centre=0.3):
        """A hot population ``centre`` above the lowest window energy with a random part per state."""
        r = np.random.default_rng([seed, 2])
        amp, c0, width = 0.1 * r.uniform(0.8, 1.2), centre * r.uniform(0.9, 1.1), 0.05 * r.uniform(0.9, 1.2)
        hot = amp * np.exp(-((self.e - self.e.min() - c0) ** 2) / (2 * width * width))
        return hot * r.uniform(0.7, 1.3, self.ns) + 1e-3 * r.uniform(0.0, 1.0, self.ns)

    def fermi(self, seed):
        mu = self.e.min() - 0.2 * np.random.default_rng([seed, 3]).uniform(0.8, 1.2)
        return 1.0 / (np.exp((self.e - mu) / (KB * self.T)) + 1.0)

    def coupled(self):
        """Ordered state pairs within reach of a phonon: |difference| <= max energy + 15 widths of
        the delta function (beyond, the Gaussian is below every FP32 number), or the list's own cutoff."""
        es = np.sort(self.e)
        cut = float(self.omega.max()) + (min(self.nsigma, 15.0) if self.nsigma > 0 else 15.0) * self.sigma
        return int((np.searchsorted(es, es + cut, side="right") - np.searchsorted(es, es - cut)).sum())


def batch_models(c):
    """The systems of a batch: grids, bands, modes, temperatures and excitation energies."""
    r = random.Random(c["draw"])
    got = []
    for _ in range(c["count"]):
        n = r.randint(c["nmin"], c["nmax"])
        m = Model(dict(n1=n, n2=n, n3=n, bands=r.randint(2, 4), modes=r.randint(3, 6), window=0.3, sigma=0.008,
                       T=r.uniform(100.0, 500.0)))
        got.append((m, r.uniform(0.1, 0.5)))
    return got


def cuda(a):
    return torch.tensor(a, dtype=torch.float64, device="cuda")


# ------------------------------------------------------------------ prepare and run


def prepare(case, seed):
    c, st = case, {"case": case}
    if c["kind"] == "batch":
        ms = batch_models(c)
        chs = [m.channels(m.couplings(seed + 1000 * i)) for i, (m, _) in enumerate(ms)]
        st["dev"] = pb.Batch(chs, precision=c["precision"])
        st["f"] = cuda(np.concatenate([m.occupations(seed + 1000 * i, e) for i, (m, e) in enumerate(ms)]))
        return st
    m = Model(c)
    ch = m.channels(m.couplings(seed))
    kind = c["kind"]
    st["dev"] = pb.Device(ch, variant=c["variant"], transport=kind == "transport", adjoint=kind == "adjoint")
    if kind == "transport":
        st["f"], st["vel"] = cuda(m.fermi(seed)), cuda(m.v)
    else:
        st["f"] = cuda(m.occupations(seed))
    if kind in ("collision", "rates"):
        st["out"] = torch.empty_like(st["f"])
    if kind == "transport":
        st["out"] = torch.empty_like(st["vel"])
    if kind == "adjoint":
        st["f"].requires_grad_(True)
        st["g2"] = pa.g2_tensor(ch).requires_grad_(True)
        st["eps"] = cuda(m.e)
    return st


def run(st):
    c, dev, kind = st["case"], st["dev"], st["case"]["kind"]
    if kind == "collision":
        return dev.collision(st["f"], out=st["out"])
    if kind == "rates":
        return dev.rates(st["f"], out=st["out"])
    if kind in ("rk4", "batch"):
        return dev.rk4(st["f"], DT, c["steps"])
    if kind == "transport":
        F, iters, _, _ = dev.transport(st["f"], st["vel"], tol=1e-10, maxit=200, out=st["out"])
        return F, iters
    st["f"].grad = st["g2"].grad = None
    f = pa.trajectory(dev, st["f"], st["g2"], DT, c["steps"], 10)
    (st["eps"] * f).sum().backward()
    return f.detach(), st["f"].grad, st["g2"].grad


# ------------------------------------------------------------------ work


def work(case):
    """A sweep is a product of the coupled pairs' coefficients with a vector, and the next sweep
    needs the result of this one, so every sweep reads each coefficient once: P_in and P_out of an
    unordered pair (they serve both directions) in the storage type, or one weight per ordered pair
    in transport, or each |g|^2 where the couplings are the data.  Flops: a multiply-add per
    coefficient and direction; about 20 operations per channel for the per-channel forms."""
    c = case
    if c["kind"] == "batch":
        ms = [m for m, _ in batch_models(c)]
        pairs, ns = sum(m.coupled() for m in ms), sum(m.ns for m in ms)
        chans = sum(m.coupled() * m.nm for m in ms)
        form, sweeps = {"ff": "ff", "c32": "c32", "fp32": "g32"}[c["precision"]], 4 * c["steps"]
    else:
        m = Model(c)
        pairs, ns, chans = m.coupled(), m.ns, m.coupled() * m.nm
        form = c["variant"]
        sweeps = 4 * c["steps"] if "steps" in c else 1
    per_channel = form in ("g32", "h16")
    sweep_bytes = chans * (4 if form == "g32" else 2) / 2 if per_channel else pairs * (8 if form == "c32" else 16) / 2
    sweep_flops = 20 * chans if per_channel else 4 * pairs
    if c["kind"] == "transport":
        it = 21  # iterations to 1e-10 on the windowed grids
        return {"bytes": pairs * 8 * (it + 2) + 8 * 7 * ns, "flops": pairs * (6 * it + 4)}
    if c["kind"] == "adjoint":  # forward, recomputed stages and the reverse sweeps; the |g|^2 gradient once
        return {"bytes": 4 * sweeps * sweep_bytes + 24 * chans, "flops": 5 * sweeps * sweep_flops + 4 * chans}
    return {"bytes": sweeps * sweep_bytes + 16 * ns, "flops": sweeps * sweep_flops}


# ------------------------------------------------------------------ the same in 64 bits


def matrices(m, g2):
    """K_in, K_out [ns, ns, modes] of Eq. 2 without |g|^2 (zero where the list holds no channel), and
    which (pair, branch) slots the list holds."""
    e = cuda(m.e)
    x = e[:, None] - e[None, :]
    j = torch.tensor(m.j, device="cuda")
    iq = torch.zeros((m.ns, m.ns), dtype=torch.int64, device="cuda")
    for i in range(3):
        iq = iq * m.nk[i] + (j[None, :, i] - j[:, None, i]) % m.nk[i]
    om = cuda(m.omega)
    kin, kout = torch.empty_like(g2), torch.empty_like(g2)
    has = torch.empty(g2.shape, dtype=torch.bool, device="cuda")
    norm = 1.0 / (math.sqrt(2 * math.pi) * m.sigma)
    for nu in range(m.nm):
        w = om[:, nu][iq]
        ok = w > 0
        if m.nsigma > 0:
            ok &= torch.minimum((x + w).abs(), (x - w).abs()) <= m.nsigma * m.sigma
        if m.g2min > 0:
            ok &= g2[:, :, nu] >= m.g2min
        N = 1.0 / torch.expm1(torch.where(ok, w, 1.0) / (KB * m.T))
        ga = norm * torch.exp(-(x + w) ** 2 / (2 * m.sigma ** 2))
        ge = norm * torch.exp(-(x - w) ** 2 / (2 * m.sigma ** 2))
        kin[:, :, nu] = torch.where(ok, ga * (N + 1) + ge * N, 0.0)
        kout[:, :, nu] = torch.where(ok, ga * N + ge * (N + 1), 0.0)
        has[:, :, nu] = ok
    return kin, kout, has


def exact_system(m, g2, c, seed, centre=0.3):
    pref = 2 * math.pi / (HBAR * m.nk[0] * m.nk[1] * m.nk[2])
    kin, kout, has = matrices(m, g2)
    kind = c["kind"]
    if kind != "adjoint":
        g2, (pin, pout) = None, [(k * g2).sum(-1) for k in (kin, kout)]
        del kin, kout, has

    def rhs(f, pin, pout):
        return pref * ((1.0 - f) * (pin @ f) - f * (pout @ (1.0 - f)))

    def steps(f, pin, pout):
        for _ in range(c["steps"]):
            k1 = rhs(f, pin, pout)
            k2 = rhs(f + 0.5 * DT * k1, pin, pout)
            k3 = rhs(f + 0.5 * DT * k2, pin, pout)
            k4 = rhs(f + DT * k3, pin, pout)
            f = f + DT / 6 * (k1 + 2 * k2 + 2 * k3 + k4)
        return f

    if kind == "transport":
        f0, v = cuda(m.fermi(seed)), cuda(m.v)
        W = pref * (pin * f0[None, :] + pout * (1.0 - f0)[None, :])
        rate = W.sum(1)
        tau = torch.where(rate > 0, 1.0 / rate, 0.0)[:, None]
        F, it = tau * v, 0
        while it < 200:
            new = tau * (v + W @ F)
            res = float((new - F).abs().max() / new.abs().max())
            F, it = new, it + 1
            if not res > 1e-10:
                break
        return F, it
    f = cuda(m.occupations(seed, centre))
    if kind == "collision":
        return rhs(f, pin, pout)
    if kind == "rates":
        return pref * (pin @ f + pout @ (1.0 - f))
    if kind in ("rk4", "batch"):
        return steps(f, pin, pout)
    pin, pout = (kin * g2).sum(-1).requires_grad_(True), (kout * g2).sum(-1).requires_grad_(True)
    f.requires_grad_(True)
    end = steps(f, pin, pout)
    (cuda(m.e) * end).sum().backward()
    grad = (pin.grad[:, :, None] * kin + pout.grad[:, :, None] * kout)[has]
    return end.detach(), f.grad, grad


def exact(case, seed):
    if case["kind"] == "batch":
        return torch.cat([exact_system(m, m.couplings(seed + 1000 * i), case, seed + 1000 * i, e)
                          for i, (m, e) in enumerate(batch_models(case))])
    m = Model(case)
    return exact_system(m, m.couplings(seed), case, seed)
