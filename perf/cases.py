"""The work that programs built on this library have it do, as measurable cases.

A case is a dict of plain values.  `kind` names the entry points it goes through:

  lattice   the production loop of one simulation (Sim): some leapfrog steps,
            the observables of the network, and a map of one plane of the state
            (the whole state while the lattice is small)
  resume    a checkpoint restart: the whole state is loaded, stepped and read back
  ensemble  ah_batch_run_ex over lattices of uneven size, era, s and seed
  serve     a burst of requests to the continuous-batching Server
  buffers   ah_observables_noalloc on a state in the caller's own device buffers

Lattices use dx = 0.5, dt = 0.1, lambda0 = 2, e0 = 1, sigma = 1 throughout (the
library's defaults).  `start` is "random" (the random-phase state at tau = 1, which
the library makes from the seed) or "network" (a smooth field with strings at its
zeros, weak Pi, theta and E: what a run looks like after its strings have formed).
Single lattices with s = 1 are large enough that repeated passes stay inside the
stretch of a(tau) in which the leapfrog is stable.
"""
import math
import random
import time

import numpy as np
import torch

import paper_1809_00995_gb300 as ah

RAD, MAT = 1, 2
DX, DT = 0.5, 0.1
WHOLE = 64          # sides up to this are read back whole, larger ones as a map
MAP = 256           # largest side of a map of one z plane
SMALL_MAP = 64      # map of a lattice of an ensemble or of a served request
SIZES = (64, 96, 128, 192, 256)
SERVE_SIZES, SERVE_WEIGHTS = (64, 128, 192, 256, 384), (0.3, 0.3, 0.2, 0.15, 0.05)


def _lattice(name, N, **kw):
    c = {"kind": "lattice", "N": N, "fp64": False, "two_step": False, "wrap": False, "era": RAD, "s": 0.0,
         "steps": 20, "start": "random"}
    if name:
        c["name"] = name
    c.update(kw)
    return c


def listed():
    return [
        # the smallest configuration: 32^3 in FP64, diagnostics every 10 steps; a trial run,
        # a check of new parameters
        _lattice("lattice32_fp64", 32, fp64=True, steps=10),
        # a small FP32 lattice with frequent diagnostics: parameter scans, teaching runs
        _lattice("lattice64", 64, steps=10),
        # an odd side with compact link phases in the matter era
        _lattice("lattice125_wrap", 125, era=MAT, wrap=True),
        # the 256^3 configuration, diagnostics every 20 steps, once its strings have formed
        _lattice("lattice256_network", 256, start="network"),
        # the same configuration in FP64 from the initial state
        _lattice("lattice256_fp64", 256, fp64=True),
        # the paper's production cadence: 512^3, diagnostics every 5 steps
        _lattice("lattice512_diag5", 512, steps=5),
        # two steps per pass, true equations of motion (s = 1), radiation era, ragged side
        _lattice("lattice381_two_step", 381, two_step=True, s=1.0, steps=50),
        # the headline configuration: 1024^3, matter era, s = 1, diagnostics every 50 steps
        _lattice("lattice1024_two_step", 1024, two_step=True, era=MAT, s=1.0, steps=50),
        # an ensemble of uneven lattices, as for the averages over seeds, eras and s
        {"name": "ensemble16", "kind": "ensemble", "count": 16, "pick": 100, "steps": 40, "diag_every": 20},
        # requests that arrive together at the server
        {"name": "serve12", "kind": "serve", "count": 12, "pick": 7, "steps": 40},
        # diagnostics inside a host framework that owns the device memory
        {"name": "buffers200", "kind": "buffers", "N": 200, "start": "network"},
        # restart from a checkpoint, ten steps, new checkpoint
        {"name": "resume80", "kind": "resume", "N": 80, "steps": 10},
    ]


def _log_int(rng, lo, hi):
    return min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49))))))


def draw(rng):
    kind = rng.choice(("fp32", "fp32", "fp32", "fp64", "two_step", "two_step", "ensemble", "serve", "buffers",
                       "resume"))
    if kind == "fp32":
        N = _log_int(rng, 24, 640)
        start = "network" if N <= 300 and rng.random() < 0.5 else "random"
        return _lattice(None, N, era=rng.choice((RAD, MAT)), wrap=rng.random() < 0.3, steps=rng.choice((5, 10, 20)),
                        start=start)
    if kind == "fp64":
        N = _log_int(rng, 16, 256)
        return _lattice(None, N, fp64=True, era=rng.choice((RAD, MAT)), steps=rng.choice((5, 10, 20)),
                        start=rng.choice(("random", "network")))
    if kind == "two_step":
        N = _log_int(rng, 64, 800)
        s = 1.0 if N >= 256 and rng.random() < 0.6 else 0.0
        era = MAT if s == 1.0 and N >= 512 else RAD
        return _lattice(None, N, two_step=True, era=era, s=s, wrap=rng.random() < 0.2, steps=rng.choice((10, 20, 50)),
                        start="network" if N <= 300 and rng.random() < 0.5 else "random")
    if kind == "ensemble":
        return {"kind": "ensemble", "count": rng.randint(4, 24), "pick": rng.randrange(1 << 20),
                "steps": rng.choice((20, 30, 40)), "diag_every": rng.choice((0, 10, 20))}
    if kind == "serve":
        return {"kind": "serve", "count": rng.randint(4, 16), "pick": rng.randrange(1 << 20),
                "steps": rng.choice((20, 30, 40))}
    if kind == "buffers":
        return {"kind": "buffers", "N": _log_int(rng, 48, 400), "start": rng.choice(("random", "network"))}
    return {"kind": "resume", "N": _log_int(rng, 24, 128), "steps": rng.choice((5, 10, 20))}


# ---- what each case runs on ------------------------------------------------------------
def _members(case):
    """(N, era, s) of the lattices of an ensemble or of a burst of requests."""
    r = random.Random(case["pick"])
    out = []
    for _ in range(case["count"]):
        N = r.choice(SIZES) if case["kind"] == "ensemble" else r.choices(SERVE_SIZES, SERVE_WEIGHTS)[0]
        out.append((N, r.choice((RAD, MAT)), float(r.choice((0, 1)))))
    return out


def _member_configs(case, seed):
    cfgs = []
    for k, (N, era, s) in enumerate(_members(case)):
        c = ah.config(N, era=era, s=s, seed=1000 * seed + k, diag_every=case.get("diag_every", 0))
        c.tau_ref = N * DX / 2.0
        c.tau_end = c.tau0 + case["steps"] * c.dt
        cfgs.append(c)
    return cfgs


def _start_step(N):
    return int(N * DX / 4.0 / DT)           # half of the run


def _network(N, seed):
    """A (10, N, N, N) state (float32, on the GPU) with strings at the zeros of a
    smooth complex Gaussian field, and smooth weak Pi, theta and E."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) * 2 + 1)
    k = torch.fft.fftfreq(N, device="cuda", dtype=torch.float64) * 2 * math.pi
    ks = k * k
    k2 = ks[:, None, None] + ks[None, :, None] + ks[None, None, :]

    def smooth(length):
        z = torch.randn((N, N, N), generator=g, device="cuda", dtype=torch.complex128)
        z = torch.fft.ifftn(torch.fft.fftn(z) * torch.exp(-0.5 * length ** 2 * k2))
        return z / z.abs().square().mean().sqrt()

    f = torch.empty((10, N, N, N), dtype=torch.float32, device="cuda")
    psi = smooth(4.0)
    phi = psi / psi.abs().clamp_min(1e-30) * torch.tanh(psi.abs() / 0.4)
    pi = 0.15 * smooth(3.0)
    a, b, c = smooth(4.0), smooth(4.0), smooth(4.0)
    for i, x in enumerate((phi.real, phi.imag, pi.real, pi.imag, 0.2 * a.real, 0.2 * a.imag, 0.2 * b.real,
                           0.02 * b.imag, 0.02 * c.real, 0.02 * c.imag)):
        f[i] = x
    return f


def _phases(N, seed):
    """The random-phase state of Sec. 2 (u from Philox-4x32-10), float64 on the GPU."""
    m32 = 0xFFFFFFFF
    idx = torch.arange(N ** 3, dtype=torch.int64, device="cuda")
    c = [torch.zeros_like(idx), torch.zeros_like(idx), idx & m32, idx >> 32]
    k0, k1 = seed & m32, (seed >> 32) & m32
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & m32) ^ c[1] ^ k0, p1 & m32, ((p0 >> 32) & m32) ^ c[3] ^ k1, p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    u = ((c[0] << 21) + (c[1] >> 11)).double() * 2.0 ** -53
    f = torch.zeros((10, N, N, N), dtype=torch.float64, device="cuda")
    f[0] = torch.cos(2 * math.pi * u).view(N, N, N)
    f[1] = torch.sin(2 * math.pi * u).view(N, N, N)
    return f


def _window(N, small=False):
    if N <= WHOLE and not small:
        return (0, 0, 0, N, N, N)
    m = min(N, SMALL_MAP if small else MAP)
    return (N // 3, N - m // 2, N // 2, m, m, 1)     # crosses the periodic boundary in y


def prepare(case, seed):
    kind = case["kind"]
    if kind == "lattice":
        flags = (ah.AH_FLAG_TWO_STEP if case["two_step"] else 0) | (ah.AH_FLAG_WRAP_THETA if case["wrap"] else 0)
        sim = ah.Sim(case["N"], precision=ah.AH_FP64 if case["fp64"] else ah.AH_FP32, era=case["era"], s=case["s"],
                     seed=seed, flags=flags)
        if case["start"] == "network":
            sim.set_fields(_network(case["N"], seed).cpu().numpy(), _start_step(case["N"]))
        return {"case": case, "sim": sim}
    if kind == "resume":
        return {"case": case, "sim": ah.Sim(case["N"], seed=seed), "step": _start_step(case["N"]),
                "fields": _network(case["N"], seed).double().cpu().numpy()}
    if kind == "buffers":
        f = _network(case["N"], seed) if case["start"] == "network" else _phases(case["N"], seed).float()
        return {"case": case, "fields": [x.clone() for x in f], "cfg": ah.config(case["N"], seed=seed),
                "step": _start_step(case["N"]) if case["start"] == "network" else 0,
                "sums": torch.empty(26, dtype=torch.float64, device="cuda")}
    cfgs = _member_configs(case, seed)
    wins = [_window(c.N, True) for c in cfgs]
    if kind == "ensemble":
        return {"case": case, "cfgs": cfgs, "windows": [(i,) + w for i, w in enumerate(wins)]}
    return {"case": case, "cfgs": cfgs, "windows": wins, "server": ah.Server(int(150e9), 64)}


# ---- one pass ---------------------------------------------------------------------------
def _row(o):
    """What a run writes to its log for one set of observables."""
    n = float(o["n_sites"])
    return [o["tau"], o["a"], o["sums"][1] / n, o["sums"][0] / n, o["v2_V"], o["xi_W"], o["max_abs_theta"]]


def _observed(obs, real):
    return {"row": np.array([_row(o) for o in obs], dtype=real), "sums": np.array([o["sums"] for o in obs], dtype=real)}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "lattice":
        sim = state["sim"]
        real = np.float64 if case["fp64"] else np.float32      # results in the precision of the state
        sim.step(case["steps"])
        out = _observed([sim.observables()], real)
        fields = torch.from_numpy(sim.fields(*_window(case["N"])))
        out["fields"] = fields if case["fp64"] else fields.float()
        return out
    if kind == "resume":
        sim = state["sim"]
        sim.set_fields(state["fields"], state["step"])
        sim.step(case["steps"])
        return {"fields": torch.from_numpy(sim.fields()).float()}
    if kind == "buffers":
        d = state["sums"]
        ah.ah_observables_noalloc([x.data_ptr() for x in state["fields"]], case["N"], state["cfg"], state["step"],
                                  d.data_ptr(), torch.cuda.current_stream().cuda_stream)
        return {"sums": d[:18].float(), "counts": d[18:].view(torch.int64).clone()}
    if kind == "ensemble":
        series, _, maps = ah.ah_batch_run_ex(state["cfgs"], state["windows"])
        out = _observed([o for s in series for o in s], np.float32)
    else:
        srv = state["server"]
        reqs = [srv.submit_ex(c, [w]) for c, w in zip(state["cfgs"], state["windows"])]
        done = {}
        while len(done) < len(reqs):
            for i, (rid, _) in enumerate(reqs):
                if i not in done:
                    got = srv.poll(rid)
                    if got is not None:
                        done[i] = got[0]
            if len(done) < len(reqs):
                time.sleep(1e-4)
        out = _observed([done[i] for i in range(len(reqs))], np.float32)
        maps = [bufs[0] for _, bufs in reqs]
    out["maps"] = np.stack(maps).astype(np.float32)
    return out


# ---- what a pass cannot do without ------------------------------------------------------
FLOPS_STEP, FLOPS_DIAG = 330, 300       # multiplies and adds per site of the equations as written


def work(case):
    """One read and one write of the ten-component state per leapfrog step (the two-step
    pass may halve that), one read per set of observables."""
    kind = case["kind"]
    if kind in ("lattice", "resume"):
        n, b = case["N"] ** 3, 8 if case.get("fp64") else 4
        diags = 1 if kind == "lattice" else 0
        host = 160 * n if kind == "resume" else 0       # the checkpoints, FP64 on the host
        return {"bytes": n * b * (20 * case["steps"] + 10 * diags) + host,
                "flops": n * (FLOPS_STEP * case["steps"] + FLOPS_DIAG * diags)}
    if kind == "buffers":
        return {"bytes": 40 * case["N"] ** 3, "flops": FLOPS_DIAG * case["N"] ** 3}
    n = sum(N ** 3 for N, _, _ in _members(case))
    diags = len(_stops(case)) if kind == "ensemble" else 1
    return {"bytes": n * (80 * case["steps"] + 40 * diags), "flops": n * (FLOPS_STEP * case["steps"] + FLOPS_DIAG * diags)}


def _stops(case):
    """Steps at which an ensemble reports observables."""
    d, n = case["diag_every"], case["steps"]
    return sorted({0, n} | (set(range(0, n, d)) if d > 0 else set()))


# ---- the same in 64 bits with plain torch -----------------------------------------------
class _Model:
    """Leapfrog and observables of Sec. 2 in float64, arrays indexed [z, y, x]."""

    def __init__(self, N, era, s, wrap=False):
        self.era, self.s, self.wrap, self.ref = era, s, wrap, N * DX / 2.0
        self.e0, self.lam0, self.sig2 = 1.0, 2.0, 1.0

    def a(self, t):
        return (t / self.ref) ** self.era

    def e(self, t):
        return self.e0 * self.a(t) ** (self.s - 1.0)

    @staticmethod
    def up(x, d):
        return torch.roll(x, -1, 2 - d)

    @staticmethod
    def down(x, d):
        return torch.roll(x, 1, 2 - d)

    def sines(self, th):
        return {(i, j): th[i] + self.up(th[j], i) - self.up(th[i], j) - th[j] for i, j in ((0, 1), (0, 2), (1, 2))}

    def load(self, f):
        self.phi, self.pi = torch.complex(f[0], f[1]), torch.complex(f[2], f[3])
        self.th, self.E = [f[4].clone(), f[5].clone(), f[6].clone()], [f[7].clone(), f[8].clone(), f[9].clone()]

    def step(self, n):
        t = 1.0 + n * DT
        an, am, ap = self.a(t), self.a(t - DT / 2), self.a(t + DT / 2)
        en, em, ep = self.e(t), self.e(t - DT / 2), self.e(t + DT / 2)
        lam = self.lam0 * an ** (2.0 * (self.s - 1.0))
        phi = self.phi
        lap = -6.0 * phi
        cur = []
        for d in range(3):
            u = torch.polar(torch.ones_like(self.th[d]), self.th[d])
            w = u * self.up(phi, d)
            lap += w
            lap += self.down(u.conj() * phi, d)
            cur.append(w.real * phi.imag - w.imag * phi.real)
        pot = DT * (an * an / ap) ** 2 * lam * 0.5 * (phi.real ** 2 + phi.imag ** 2 - self.sig2)
        self.pi = (am / ap) ** 2 * self.pi - pot * phi + DT / DX ** 2 * (an / ap) ** 2 * lap
        p = {q: torch.sin(x) for q, x in self.sines(self.th).items()}
        curl = [p[0, 1] - self.down(p[0, 1], 1) + p[0, 2] - self.down(p[0, 2], 2),
                self.down(p[0, 1], 0) - p[0, 1] + p[1, 2] - self.down(p[1, 2], 2),
                self.down(p[0, 2], 0) - p[0, 2] + self.down(p[1, 2], 1) - p[1, 2]]
        for d in range(3):
            self.E[d] = ((ep / em) ** 2 * self.E[d] + 2.0 * DT * an * an * ep * ep * cur[d]
                         - DT / DX ** 2 * (ep / en) ** 2 * curl[d])
            self.th[d] = self.th[d] + DT * self.E[d]
            if self.wrap:
                k = torch.round(self.th[d] / (2 * math.pi)) * (self.th[d].abs() > math.pi)
                self.th[d] = self.th[d] - 2 * math.pi * k
        self.phi = phi + DT * self.pi

    def observe(self, n):
        t = 1.0 + n * DT
        a, am = self.a(t), self.a(t - DT / 2)
        e2a2, lam = (self.e(t) * a) ** 2, self.lam0 * a ** (2.0 * (self.s - 1.0))
        phi, pi = self.phi, self.pi
        K = pi.real ** 2 + pi.imag ** 2
        U = [torch.polar(torch.ones_like(x), x) for x in self.th]
        z = [phi.conj() * U[d] * self.up(phi, d) for d in range(3)]
        G2 = sum((U[d] * self.up(phi, d) - phi).abs().square() for d in range(3)) / DX ** 2
        V = a * a * lam / 4.0 * (phi.real ** 2 + phi.imag ** 2 - self.sig2) ** 2
        El = sum(x * x for x in self.E) / (2.0 * e2a2 * DX ** 2)
        xi = self.sines(self.th)
        B = sum(2.0 * torch.sin(0.5 * x) ** 2 for x in xi.values()) / (e2a2 * DX ** 4)
        L, rho = K - G2 - V + El - B, K + G2 + V + El + B
        p = K - G2 / 3.0 - V + (El + B) / 3.0
        g1 = sum(self.E[d] - self.down(self.E[d], d) for d in range(3)) / self.e(t - DT / 2) ** 2
        g2 = 2.0 * DX ** 2 * am * am * (phi.real * pi.imag - phi.imag * pi.real)
        G, gs = g1 + g2, g1.abs() + g2.abs()
        sums = [x.sum().item() for x in (L, rho, p, K, G2, V, El, B, K * V, G2 * V, K * L, G2 * L, p * L, rho * L,
                                         G * G, gs * gs)]
        counts = [[], [], 0]
        for i, j in ((0, 1), (0, 2), (1, 2)):
            z2, z3 = self.up(z[j], i), self.up(z[i], j)
            tot = z[i].angle() + z2.angle() - z3.angle() - z[j].angle() - (z[i] * z2 * z3.conj() * z[j].conj()).angle()
            w = torch.round(tot / (2 * math.pi))
            counts[0].append(int(w.abs().sum().item()))
            counts[1].append(int(w.sum().item()))
            counts[2] += int((w != 0).sum().item())
        nsites, tmax = phi.numel(), max(x.abs().max().item() for x in self.th)
        rv = sums[8] / sums[9] if sums[9] else math.nan
        xi_w = math.sqrt(nsites * DX ** 3 / (math.pi / 6.0 * DX * sum(counts[0]))) if sum(counts[0]) else math.inf
        row = [t, a, sums[1] / nsites, sums[0] / nsites, 2.0 * rv / (1.0 + rv), xi_w, tmax]
        return {"row": row, "sums": sums, "gmax": G.abs().max().item(), "tmax": tmax}

    def window(self, w):
        x0, y0, z0, nx, ny, nz = w
        N = self.phi.shape[0]
        ix = [torch.arange(o, o + m, device="cuda") % N for o, m in ((z0, nz), (y0, ny), (x0, nx))]
        comps = [self.phi.real, self.phi.imag, self.pi.real, self.pi.imag] + self.th + self.E
        return torch.stack([c[ix[0]][:, ix[1]][:, :, ix[2]] for c in comps]).cpu().numpy()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("ensemble", "serve"):
        rows, sums, maps = [], [], []
        for k, (N, era, s) in enumerate(_members(case)):
            m = _Model(N, era, s)
            m.load(_phases(N, 1000 * seed + k))
            stops = _stops(case) if kind == "ensemble" else [case["steps"]]
            for n in range(case["steps"] + 1):
                if n in stops:
                    o = m.observe(n)
                    rows.append(o["row"])
                    sums.append(o["sums"])
                if n < case["steps"]:
                    m.step(n)
            maps.append(m.window(_window(N, True)))
        return {"row": np.array(rows), "sums": np.array(sums), "maps": np.stack(maps)}
    N = case["N"]
    if kind == "lattice" and N ** 3 * case["steps"] > 700 ** 3 * 10:
        return None                                     # too long
    m = _Model(N, case.get("era", RAD), case.get("s", 0.0), case.get("wrap", False))
    network = kind == "resume" or case["start"] == "network"
    n0 = _start_step(N) if network else 0
    f = _network(N, seed).double() if network else _phases(N, seed)
    if kind == "buffers":
        m.load(f.float().double())
        o = m.observe(n0)
        return {"sums": np.array(o["sums"] + [o["gmax"], o["tmax"]]), "counts": None}
    m.load(f)
    del f
    for n in range(n0, n0 + case["steps"]):
        m.step(n)
    if kind == "resume":
        return {"fields": m.window((0, 0, 0, N, N, N))}
    o = m.observe(n0 + case["steps"])
    return {"row": np.array([o["row"]]), "sums": np.array([o["sums"]]), "fields": m.window(_window(N))}
