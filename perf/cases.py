"""The work that users of the package have it do, as measurable cases.

Every case goes through the package's public entry points (``fill``,
``Context``, ``MPREnergy``, ``sample_energy_noalloc``) on synthetic fields of
the kinds that the repository's workloads are made of: Gaussian, lognormal and
gamma-copula random fields with uniform random gaps, solid rectangles or both.
A case is a dict of plain values:

    kind    fill | estimate_T | sweep | open | checkpoint | energy_grad | sample_energy
    images  number of images; one image is ly x lx, several have square sides
            drawn log-uniformly from [lo, hi] by the case's own `layout` number
    field, ell, frac, block, rects   the field and its gaps
    chains, n_equil, n_meas, sweeps, warm, phase, T, q, model, record   the run

The inputs are made on the GPU from the seed alone.
"""
import math
import random

import numpy as np
import torch

import paper_1710_03038_gb300 as mpr

TWO_PI = 2.0 * math.pi
SEED = 0x2545F4914F6CDD1D   # seed of the random stream (the package's default)


# ------------------------------------------------------------------- cases

def listed():
    return [
        # a small field as in the paper's tables (64^2, a third missing): the whole
        # gap fill in one call, where launches and latency count
        dict(name="fill_64", kind="fill", images=1, ly=64, lx=64, field="grf", ell=8.0, frac=0.33,
             chains=10, n_equil=200, n_meas=100),
        # a batch of ragged maps filled in one call (satellite tiles, well logs)
        dict(name="fill_ragged_batch", kind="fill", images=8, lo=96, hi=512, layout=5, field="lognormal",
             ell=12.0, frac=0.4, rects=2, chains=16, n_equil=50, n_meas=100),
        # the temperature by specific energy matching, for one map larger than the
        # lattices it runs on (256^2, 16 chains)
        dict(name="temperature_1024", kind="estimate_T", images=1, ly=1024, lx=1024, field="lognormal",
             ell=16.0, frac=0.4, chains=4),
        # equilibration of many realisations of a mid-sized map, half missing
        # (100 chains: whole groups of 32 and 4 left over), then the states
        dict(name="equil_1024_r100", kind="sweep", phase="equil", images=1, ly=1024, lx=1024,
             field="lognormal", ell=20.0, frac=0.5, chains=100, warm=0, sweeps=20, T=0.01),
        # the sampling sweeps of a large map and the prediction with its spread: the
        # bulk of every job
        dict(name="measure_4096_r32", kind="sweep", phase="measure", images=1, ly=4096, lx=4096,
             field="lognormal", ell=16.0, frac=0.4, chains=32, warm=5, sweeps=20, T=0.003),
        # a map with a large solid hole (cloud cover, a swath gap) and sparse gaps
        dict(name="equil_hole_2048_r32", kind="sweep", phase="equil", images=1, ly=2048, lx=2048,
             field="gamma", ell=64.0, frac=0.2, block=512, chains=32, warm=0, sweeps=12, T=0.02),
        # sampling of a ragged batch with rectangles, 16 realisations each
        dict(name="measure_ragged_batch", kind="sweep", phase="measure", images=16, lo=128, hi=1024,
             layout=7, field="grf", ell=15.0, frac=0.45, rects=3, chains=16, warm=5, sweeps=25, T=0.05),
        # the Gaussian (GMRF) variant on a small odd-sized map, energies recorded
        dict(name="gmrf_251x173_r16", kind="sweep", phase="measure", images=1, ly=251, lx=173,
             field="grf", ell=10.0, frac=0.4, chains=16, warm=4, sweeps=16, T=0.05, model="gmrf",
             record=True),
        # setting a job up: map, tables, hot start, sample energy; its first states
        dict(name="open_2048_r32", kind="open", images=1, ly=2048, lx=2048, field="lognormal", ell=16.0,
             frac=0.4, chains=32),
        # resume and save: states and running sums in and out, energies of the chains
        dict(name="checkpoint_1000x777_r24", kind="checkpoint", images=1, ly=1000, lx=777, field="grf",
             ell=12.0, frac=0.5, chains=24),
        # the energy as a differentiable function, forward and backward
        dict(name="energy_grad_12x509x383", kind="energy_grad", images=12, ly=509, lx=383, q=0.5),
        # sample energies of two maps where nothing may be allocated
        dict(name="sample_energy_pair", kind="sample_energy", images=2, lo=300, hi=1400, layout=3,
             field="lognormal", ell=16.0, frac=0.4, q=0.5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the listed ranges: any kind, sizes log-uniform, odd sides as often as even."""
    kind = rng.choice(["fill", "estimate_T", "sweep", "sweep", "sweep", "open", "checkpoint",
                       "energy_grad", "sample_energy"])
    field = rng.choice(["grf", "lognormal", "gamma"])
    ell = round(rng.uniform(5.0, 40.0), 1)
    frac = round(rng.uniform(0.2, 0.66), 3)
    if kind == "fill":
        side = _log_int(rng, 32, 400)
        return dict(kind="fill", images=1, ly=side, lx=_log_int(rng, max(32, side // 2), min(400, 2 * side)),
                    field=field, ell=ell, frac=frac, chains=rng.choice([8, 10, 16, 20, 32]),
                    n_equil=rng.randint(40, 200), n_meas=rng.randint(50, 100))
    if kind == "estimate_T":
        side = _log_int(rng, 96, 2048)
        return dict(kind="estimate_T", images=1, ly=side, lx=_log_int(rng, 96, 2048), field=field, ell=ell,
                    frac=frac, chains=rng.choice([2, 4, 8]))
    if kind == "sweep":
        # gap sites x chains x sweeps stay below the largest listed case's
        phase = rng.choice(["equil", "measure"])
        sweeps = rng.randint(8, 25)
        common = dict(kind="sweep", phase=phase, field=field, ell=ell, frac=frac,
                      warm=5 if phase == "measure" else 0, sweeps=sweeps,
                      T=round(math.exp(rng.uniform(math.log(0.003), math.log(0.3))), 4),
                      q=rng.choice([0.5, 0.5, 0.5, 0.35]),
                      model=rng.choice(["mpr", "mpr", "mpr", "gmrf"]), record=rng.random() < 0.3)
        if rng.random() < 0.3:
            lo = _log_int(rng, 64, 256)
            return dict(common, images=rng.randint(2, 16), lo=lo, hi=_log_int(rng, lo + 32, 1024),
                        layout=rng.randint(0, 999), rects=rng.randint(0, 4),
                        chains=rng.choice([4, 10, 16, 32]))
        side = _log_int(rng, 64, 2400)
        return dict(common, images=1, ly=side, lx=_log_int(rng, max(64, side // 2), min(2400, 2 * side)),
                    block=side // 4 if rng.random() < 0.3 else 0,
                    chains=rng.choice([7, 16, 32, 32, 48, 100] if side < 1100 else [16, 30, 32]))
    if kind == "open":
        return dict(kind="open", images=1, ly=_log_int(rng, 64, 2400), lx=_log_int(rng, 64, 2400),
                    field=field, ell=ell, frac=frac, chains=rng.choice([8, 10, 16, 32]))
    if kind == "checkpoint":
        return dict(kind="checkpoint", images=1, ly=_log_int(rng, 64, 1500), lx=_log_int(rng, 64, 1500),
                    field=field, ell=ell, frac=frac, chains=rng.choice([6, 10, 16, 24, 32]))
    if kind == "energy_grad":
        return dict(kind="energy_grad", images=rng.randint(1, 40), ly=_log_int(rng, 32, 700),
                    lx=_log_int(rng, 32, 700), q=rng.choice([0.5, 0.35]))
    lo = _log_int(rng, 64, 700)
    return dict(kind="sample_energy", images=rng.randint(1, 6), lo=lo, hi=_log_int(rng, lo + 32, 2048),
                layout=rng.randint(0, 999), field=field, ell=ell, frac=frac, q=0.5)


def _shapes(case):
    n = case["images"]
    if "ly" in case:
        return [(case["ly"], case["lx"])] * n
    rng = random.Random(case["layout"])
    sides = [_log_int(rng, case["lo"], case["hi"]) for _ in range(n)]
    return [(s, s) for s in sides]


def _params(case):
    return mpr.Params(q=case.get("q", 0.5), model=case.get("model", "mpr"), seed=SEED)


# ------------------------------------------------------------------ inputs

def _field(shape, kind, ell, gen):
    """A random field with exponential covariance (circulant embedding) and the
    marginal `kind`, float32 on the GPU."""
    ly, lx = shape
    my, mx = 2 * ly, 2 * lx
    dy = torch.arange(my, device="cuda").float()
    dx = torch.arange(mx, device="cuda").float()
    dy, dx = torch.minimum(dy, my - dy), torch.minimum(dx, mx - dx)
    cov = torch.exp(-torch.sqrt(dy[:, None] ** 2 + dx[None, :] ** 2) / ell)
    amp = torch.sqrt(torch.fft.fft2(cov).real.clamp_(min=0.0) / (my * mx))
    del cov
    w = torch.complex(torch.randn(my, mx, device="cuda", generator=gen),
                      torch.randn(my, mx, device="cuda", generator=gen))
    y = torch.fft.fft2(w * amp).real[:ly, :lx].contiguous()
    if kind == "lognormal":
        return torch.exp(y)
    if kind == "gamma":
        # gamma(2, 10) by the Wilson-Hilferty cube of a normal variable
        return 20.0 * (1.0 - 1.0 / 18.0 + y / math.sqrt(18.0)).clamp_(min=0.02) ** 3
    return 50.0 + 10.0 * y


def _images(case, seed):
    """Values and gap masks (uint8, 1 = missing) of the case's images."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    rng = random.Random(int(seed))
    zs, gs = [], []
    for ly, lx in _shapes(case):
        z = _field((ly, lx), case["field"], case["ell"], gen)
        g = torch.rand(ly, lx, device="cuda", generator=gen) < case["frac"]
        b = case.get("block", 0)
        if b:
            y0, x0 = rng.randint(0, max(0, ly - b)), rng.randint(0, max(0, lx - b))
            g[y0:y0 + b, x0:x0 + b] = True
        for _ in range(case.get("rects", 0)):
            h, w = rng.randint(ly // 16 + 1, ly // 5 + 1), rng.randint(lx // 16 + 1, lx // 5 + 1)
            y0, x0 = rng.randint(0, ly - h), rng.randint(0, lx - w)
            g[y0:y0 + h, x0:x0 + w] = True
        zs.append(z)
        gs.append(g.to(torch.uint8))
    return zs, gs


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "energy_grad":
        gen = torch.Generator(device="cuda").manual_seed(int(seed))
        phi = TWO_PI * torch.rand(case["images"], case["ly"], case["lx"], device="cuda", generator=gen)
        st["phi"] = phi.requires_grad_(True)
        st["J"] = torch.tensor(1.25, dtype=torch.float64, device="cuda", requires_grad=True)
        st["weights"] = torch.randn(case["images"], dtype=torch.float64, device="cuda", generator=gen)
        return st
    zs, gs = _images(case, seed)
    if kind == "sample_energy":
        st["z"] = torch.cat([z.reshape(-1) for z in zs])
        st["gap"] = torch.cat([g.reshape(-1) for g in gs])
        st["shapes"] = _shapes(case)
        n = case["images"]
        st["out"] = dict(e_s=torch.empty(n, dtype=torch.float64, device="cuda"),
                         n_sp=torch.empty(n, dtype=torch.int64, device="cuda"),
                         zmin=torch.empty(n, dtype=torch.float32, device="cuda"),
                         zmax=torch.empty(n, dtype=torch.float32, device="cuda"))
        return st
    st["z"], st["gap"] = zs, gs
    if kind in ("fill", "open"):
        return st
    # a running job: its context lives on a stream of its own
    st["stream"] = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(st["stream"]):
        st["ctx"] = mpr.Context(zs, gs, chains=case["chains"], params=_params(case))
        if kind == "sweep":
            st["ctx"].set_T(case["T"])
            st["ctx"].sweep(case["warm"], "equil")
    if kind == "checkpoint":
        st.update(_saved(case, seed, gs))
    torch.cuda.synchronize()
    return st


def _saved(case, seed, gs):
    """Saved states and running sums of 40 sampling sweeps."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed) + 7)
    R = case["chains"]
    states, sums, sums2 = [], [], []
    for g in gs:
        mean = 0.2 + 0.9 * TWO_PI * torch.rand(g.shape, device="cuda", generator=gen)
        states.append((mean + 0.2 * torch.randn(R, *g.shape, device="cuda", generator=gen)).remainder(6.28))
        m = mean.double() * 40 * R
        sums.append(m)
        sums2.append(m * mean.double() * 1.01)
    return dict(states=states, sums=sums, sums2=sums2, terms=40 * R)


# --------------------------------------------------------------------- run

def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "fill":
        (z_hat, z_std), ctx = mpr.fill(st["z"], st["gap"], case["chains"], case["n_equil"], case["n_meas"],
                                       params=_params(case), std=True)
        ctx.close()
        return dict(z_hat=z_hat, z_std=z_std)
    if kind == "open":
        ctx = mpr.Context(st["z"], st["gap"], chains=case["chains"], params=_params(case))
        out = dict(info=ctx.image_info(), state=ctx.get_state())
        ctx.close()
        return out
    if kind == "energy_grad":
        H = mpr.MPREnergy.apply(st["phi"], st["J"], case["q"])
        g_phi, g_J = torch.autograd.grad((H * st["weights"]).sum(), (st["phi"], st["J"]))
        return dict(H=H.detach(), g_phi=g_phi, g_J=g_J)
    if kind == "sample_energy":
        return mpr.sample_energy_noalloc(st["z"], st["gap"], q=case["q"], out=st["out"], shapes=st["shapes"])
    ctx = st["ctx"]
    with torch.cuda.stream(st["stream"]):
        if kind == "estimate_T":
            return dict(T=ctx.estimate_T())
        if kind == "checkpoint":
            ctx.set_state(st["states"])
            ctx.set_accumulators(st["sums"], st["sums2"], st["terms"])
            s1, s2, n = ctx.accumulators()
            return dict(state=ctx.get_state(), sums=s1, sums2=s2, terms=n, energy=ctx.energy())
        ctx.sweep(case["sweeps"], case["phase"], record_energy=case.get("record", False))
        out = {}
        if case["phase"] == "measure":
            out["z_hat"], out["z_std"] = ctx.predict(std=True)
        else:
            out["state"] = ctx.get_state()
        if case.get("record", False):
            out["chains"] = {k: v for k, v in ctx.chain_info().items() if k != "a"}
        return out


# -------------------------------------------------------------------- work

# Arithmetic of one gap site-update as written in the method: the local field (8
# additions), its angle and length, the reflection, the proposal, the energy
# difference and its exponential, and half a random block (integer multiplies and
# exclusive-ors, counted as operations).
UPDATE_FLOPS = 100.0


def _gap_sites(case):
    n = sum(h * w for h, w in _shapes(case))
    f = case["frac"]
    extra = (1.0 - f) * min(case.get("block", 0) ** 2, n) + 0.01 * case.get("rects", 0) * n * (1.0 - f)
    return n, f * n + extra


def work(case):
    kind = case["kind"]
    if kind == "energy_grad":
        n = case["images"] * case["ly"] * case["lx"]
        return dict(bytes=12.0 * n, flops=60.0 * n)
    n, p = _gap_sites(case)
    R = case.get("chains", 0)
    if kind == "sample_energy":
        return dict(bytes=5.0 * n, flops=40.0 * n)
    if kind == "open":
        return dict(bytes=5.0 * n + 4.0 * n * R, flops=40.0 * n + 25.0 * p * R)
    if kind == "checkpoint":
        return dict(bytes=8.0 * n * R + 32.0 * n, flops=40.0 * n * R)
    # lattices of the temperature estimate: 16 chains, 40 + 4 x (40 + 40) sweeps of
    # both colours, every site free, read and written once a sweep
    t_sites = 360.0 * 16 * sum(min(256, max(h, w)) ** 2 for h, w in _shapes(case))
    if kind == "estimate_T":
        return dict(bytes=8.0 * t_sites, flops=UPDATE_FLOPS * t_sites)
    # a sweep reads the samples once and reads and writes every gap angle once
    sweeps = case["n_equil"] + case["n_meas"] if kind == "fill" else case["sweeps"]
    b, f = sweeps * (8.0 * p * R + 4.0 * n), sweeps * UPDATE_FLOPS * p * R
    if kind == "fill":
        return dict(bytes=b + 8.0 * t_sites + 13.0 * n, flops=f + UPDATE_FLOPS * t_sites)
    out = 4.0 * n * R if case["phase"] == "equil" else 8.0 * n
    return dict(bytes=b + out, flops=f)


# ------------------------------------------------------------------- exact

M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors that hold 32-bit words."""
    k0, k1 = SEED & M32, SEED >> 32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57   # modulo 2^64: both halves are exact
        c0, c1, c2, c3 = (((p1 >> 32) & M32) ^ c1 ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c3 ^ k1, p0 & M32)
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c0, c1, c2, c3


class _Grid64:
    """One image's field in 64 bits: mapped samples, gap sites by colour, neighbours."""

    def __init__(self, z, gap, index):
        self.ly, self.lx = z.shape
        g = gap.reshape(-1) != 0
        z = z.double().reshape(-1)
        self.zmin, self.zmax = float(z[~g].min()), float(z[~g].max())
        self.z, self.gap, self.index = z, g, index
        self.phi = torch.where(g, torch.zeros_like(z), TWO_PI * (z - self.zmin) / (self.zmax - self.zmin))
        self.colours = []
        for c in (0, 1):
            i = torch.nonzero(g).reshape(-1)
            y, x = i // self.lx, i % self.lx
            i = i[(x + y) % 2 == c]
            y, x = i // self.lx, i % self.lx
            has = torch.stack([y > 0, y + 1 < self.ly, x > 0, x + 1 < self.lx])
            nb = torch.stack([i - self.lx, i + self.lx, i - 1, i + 1])
            self.colours.append((i, torch.where(has, nb, i.expand(4, -1)), has.double(), (y << 16) | (x >> 1)))

    def uniforms(self, c, sweep, first, n):
        """(u, r) of colour c's sites in the realisations first .. first + n - 1 (first even)."""
        pos = self.colours[c][3]
        pairs = torch.arange(first // 2, (first + n + 1) // 2, device=pos.device)[:, None]
        w = _philox(pos[None, :].expand(len(pairs), -1), torch.full_like(pos, sweep)[None, :],
                    pairs.expand(-1, len(pos)), torch.full_like(pos, self.index | (c << 31))[None, :])
        both = [torch.stack([a, b], 1).reshape(-1, len(pos))[:n] for a, b in ((w[0], w[2]), (w[1], w[3]))]
        return [(b >> 8).double() * 2.0 ** -24 for b in both]

    def hot(self, first, n):
        s = self.phi.expand(n, -1).clone()
        for c in (0, 1):
            s[:, self.colours[c][0]] = TWO_PI * self.uniforms(c, M32, first, n)[0]
        return s

    def update(self, s, c, sweep, first, a, T, q, model):
        """Alg. 1 at every gap site of colour c of the chains s; returns the accepted counts."""
        i, nb, has, _ = self.colours[c]
        phi, v = s[:, i], s[:, nb]                      # [n, S], [n, 4, S]
        u, r = self.uniforms(c, sweep, first, len(s))
        alpha = (TWO_PI / a)[:, None]
        if model == "gmrf":
            m = (v * has).sum(1) / has.sum(0)
            t = 2.0 * m - phi
            phi1 = torch.where((t >= 0) & (t < TWO_PI), t, phi)
            phi2 = (phi1 + alpha * (u - 0.5)).remainder(TWO_PI)
            dH = has.sum(0) * (phi2 - phi1) * (phi2 + phi1 - 2.0 * m) / (2.0 * math.pi ** 2)
        else:
            C, S = (torch.cos(q * v) * has).sum(1), (torch.sin(q * v) * has).sum(1)
            field = torch.sqrt(C * C + S * S) > 1e-6    # a shorter field vanishes
            t = (2.0 * torch.atan2(S, C) - q * phi).remainder(TWO_PI)
            phi1 = torch.where(field & (t < TWO_PI * q), t / q, phi)
            phi2 = (phi1 + alpha * (u - 0.5)).remainder(TWO_PI)
            # -J [cos(q phi'' - Psi) - cos(q phi' - Psi)] R as a product: no cancellation
            x, h = q * phi1, 0.5 * q * (phi2 - phi1)
            dH = 2.0 * torch.sin(h) * (C * torch.sin(x + h) - S * torch.cos(x + h)) * field
        ok = r < torch.exp((-dH / T).clamp(max=0.0))
        s[:, i] = torch.where(ok, phi2, phi1)
        return ok.sum(1)

    def energy(self, s, q=0.5, model="mpr"):
        """H per bond of every chain."""
        p = s.reshape(len(s), self.ly, self.lx)
        e = (lambda d: d * d / (2.0 * math.pi ** 2) - 1.0) if model == "gmrf" else (lambda d: -torch.cos(q * d))
        H = e(p[:, 1:] - p[:, :-1]).sum((1, 2)) + e(p[:, :, 1:] - p[:, :, :-1]).sum((1, 2))
        return H / (self.ly * (self.lx - 1) + self.lx * (self.ly - 1))

    def sample_energy(self, q=0.5, model="mpr"):
        """(mean bond energy, number) of the sample pairs."""
        p, ok = self.phi.reshape(self.ly, self.lx), ~self.gap.reshape(self.ly, self.lx)
        e = (lambda d: d * d / (2.0 * math.pi ** 2) - 1.0) if model == "gmrf" else (lambda d: -torch.cos(q * d))
        down, right = ok[1:] & ok[:-1], ok[:, 1:] & ok[:, :-1]
        n = int(down.sum() + right.sum())
        tot = e(p[1:] - p[:-1])[down].sum() + e(p[:, 1:] - p[:, :-1])[right].sum()
        return float(tot) / n, n


def _exact_sweeps(case, seed):
    n_sites, p = _gap_sites(case)
    total = case["warm"] + case["sweeps"]
    if total > 30 or total * p * case["chains"] > 6e9:   # too slow in 64 bits
        return None
    R, T, model, q = case["chains"], case["T"], case.get("model", "mpr"), case.get("q", 0.5)
    measure = case["phase"] == "measure"
    out = dict(z_hat=[], z_std=[]) if measure else dict(state=[])
    accepted, e_last = [], []
    for k, (z, g) in enumerate(zip(*_images(case, seed))):
        G = _Grid64(z, g, k)
        s1 = torch.zeros_like(G.z)
        s2 = torch.zeros_like(G.z)
        states = []
        chunk = max(2, 2 * int(3e7 // max(1, G.z.numel())))
        for first in range(0, R, chunk):
            n = min(chunk, R - first)
            s = G.hot(first, n)
            a = torch.ones(n, dtype=torch.float64, device="cuda")
            for i in range(total):
                acc = sum(G.update(s, c, i, first, a, T, q, model) for c in (0, 1))
                if i < case["warm"] or not measure:
                    low = acc.double() < 0.3 * float(G.gap.sum())
                    a = torch.where(low, torch.full_like(a, float(np.float32(1.0 + (i + 1) / 3.0))), a)
                else:
                    s1 += s.sum(0)
                    s2 += (s * s).sum(0)
            accepted.append(acc)
            e_last.append(G.energy(s, q, model))
            if not measure:
                states.append(s.float())   # compared at 32 bits: halves the memory
            del s
        if measure:
            m, scale = s1 / (R * case["sweeps"]), (G.zmax - G.zmin) / TWO_PI
            sd = torch.sqrt((s2 / (R * case["sweeps"]) - m * m).clamp(min=0.0)) * scale
            out["z_hat"].append(torch.where(G.gap, G.zmin + scale * m, G.z).reshape(G.ly, G.lx))
            out["z_std"].append(torch.where(G.gap, sd, torch.zeros_like(sd)).reshape(G.ly, G.lx))
        else:
            out["state"].append(torch.cat(states).reshape(R, G.ly, G.lx))
    if case.get("record", False):
        out["chains"] = dict(e_last=torch.cat(e_last).reshape(-1, R), accepted=None)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("fill", "estimate_T"):
        # hundreds of sweeps whose decisions feed the temperature and one another: two
        # arithmetics part ways, and only distributions agree
        return None
    if kind == "sweep":
        return _exact_sweeps(case, seed)
    if kind == "energy_grad":
        st = prepare(case, seed)
        p, q, w = st["phi"].detach().double(), case["q"], st["weights"][:, None, None]
        J = float(st["J"])
        dv, dh = q * (p[:, 1:] - p[:, :-1]), q * (p[:, :, 1:] - p[:, :, :-1])
        B = torch.cos(dv).sum((1, 2)) + torch.cos(dh).sum((1, 2))
        t = torch.zeros_like(p)
        t[:, 1:] += torch.sin(dv)
        t[:, :-1] -= torch.sin(dv)
        t[:, :, 1:] += torch.sin(dh)
        t[:, :, :-1] -= torch.sin(dh)
        return dict(H=-J * B, g_phi=J * q * w * t, g_J=-(st["weights"] * B).sum())
    grids = [_Grid64(z, g, k) for k, (z, g) in enumerate(zip(*_images(case, seed)))]
    if kind in ("open", "sample_energy"):
        e = [G.sample_energy(case.get("q", 0.5)) for G in grids]
        info = dict(e_s=np.array([v for v, _ in e]), n_sp=np.array([n for _, n in e]),
                    zmin=np.array([G.zmin for G in grids]), zmax=np.array([G.zmax for G in grids]))
        if kind == "sample_energy":
            return info
        info["n_gap"] = np.array([int(G.gap.sum()) for G in grids])
        R = case["chains"]
        return dict(info=info, state=[torch.cat([G.hot(k, 2) for k in range(0, R, 2)])
                                      .reshape(R, G.ly, G.lx) for G in grids])
    G, s = grids[0], _saved(case, seed, _images(case, seed)[1])
    g = G.gap.reshape(G.ly, G.lx)
    state = torch.where(g, s["states"][0].double(), G.phi.reshape(G.ly, G.lx))
    zero = torch.zeros_like(s["sums"][0])
    return dict(state=[state], sums=[torch.where(g, s["sums"][0], zero)],
                sums2=[torch.where(g, s["sums2"][0], zero)], terms=s["terms"],
                energy=G.energy(state.reshape(case["chains"], -1))[None, :])
