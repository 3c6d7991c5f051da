"""The work that programs have this library do, as cases to be timed and compared.

Every case goes through the Python binding, as a user's program does, on
inputs that a seed fixes: material maps with seeded draws where the workload
has them (sigma_n of the metal, a random substrate, random boxes), a seeded
random state of the fields, the workload's sources and probes.

Kinds of a case ("kind"):
  step    K steps of one grid, then the integer-level fields and the probes'
          spectra: a stretch of a run between two read-outs.
  watch   K steps, then the watchdog's statistics of every field: the loop of
          a monitored long run (no field leaves the device).
  batch   K steps of many resonator variants at once, then their fields.
  adjoint objective and gradients of a probe's power by the discrete adjoint,
          from the state at rest (the grid is kept between calls).
  design  the same through the autograd function, as an optimiser's iteration
          calls it: new maps in, a scalar and two gradients out.
  fp64    K steps of the FP64 stepper, fields read back to the host.
"""
import functools
import math

import numpy as np
import torch

from paper_2305_13419_gb300 import adjoint as tfa
from paper_2305_13419_gb300 import twofluid as tf
from paper_2305_13419_gb300 import workloads as W

# A 1 V/m source gives objectives near 1e-34 (the DFT carries dt); its
# gradients would be subnormal FP32 numbers.  They scale with the amplitude's
# square: sources of 1e12 V/m keep them in FP32's normal range.
ADJOINT_AMP = 1e12


def listed():
    return [
        # the 1-D columns of the reflection study (4480 cells, Mur walls): tiny
        # steps by the thousand, where what a step costs is its launch
        {"name": "column-reflection", "kind": "step", "geom": "column", "nx": 1, "ny": 1, "nz": 4480, "steps": 400},
        # the quasi-1-D slab of the reflection / skin-depth study
        {"name": "slab", "kind": "step", "geom": "slab", "nx": 4, "ny": 4, "nz": 2048, "steps": 400},
        # a small resonator, the size of a quick look or of a parameter sweep's member
        {"name": "cpw-small", "kind": "step", "geom": "cpw", "template": "small", "nx": 128, "ny": 64, "nz": 40,
         "steps": 200},
        # the same grid stepped in short calls by a program that looks at the fields in between
        {"name": "cpw-small-call", "kind": "step", "geom": "cpw", "template": "small", "nx": 128, "ny": 64, "nz": 40,
         "steps": 3},
        # a box of odd sizes whose material varies from cell to cell (mu too), three kinds of boundary
        {"name": "box-mixed", "kind": "step", "geom": "box", "nx": 189, "ny": 131, "nz": 75, "bcx": "periodic",
         "bcy": "pec", "bcz": "cpml", "mu": True, "edge_rule": 0, "theta": 0.5, "steps": 50},
        # a monitored run of the 256 x 128 x 64 resonator
        {"name": "cpw-watch", "kind": "watch", "geom": "cpw", "template": "half", "nx": 256, "ny": 128, "nz": 64,
         "steps": 64},
        # the resonator at its ordinary size
        {"name": "cpw", "kind": "step", "geom": "cpw", "template": "full", "nx": 512, "ny": 256, "nz": 128,
         "steps": 50},
        # the largest single grid of the benchmark
        {"name": "cpw-large", "kind": "step", "geom": "cpw", "template": "large", "nx": 1024, "ny": 512, "nz": 256,
         "steps": 24},
        # resonator variants of uneven sizes stepped together
        {"name": "batch", "kind": "batch", "count": 16, "small": 96, "large": 160, "variant": 3, "steps": 64},
        # the gradient of a probe's power on the 256 x 128 x 64 resonator with a random substrate
        {"name": "adjoint", "kind": "adjoint", "geom": "cpw", "template": "half", "nx": 256, "ny": 128, "nz": 64,
         "steps": 128, "segment": 64},
        # an optimiser's iteration on a small resonator, set-up included
        {"name": "design", "kind": "design", "geom": "cpw", "template": "scaled", "nx": 96, "ny": 64, "nz": 48,
         "steps": 96, "segment": 32},
        # the FP64 stepper beside the FP32 path (the precision study)
        {"name": "fp64", "kind": "fp64", "geom": "cpw", "template": "small", "nx": 128, "ny": 64, "nz": 40,
         "steps": 64},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["watch", "batch", "adjoint", "design", "fp64"])
    if kind == "batch":
        small = rng.randint(64, 112)
        return {"kind": kind, "count": _log(rng, 2, 24), "small": small, "large": small + rng.randint(16, 48),
                "variant": rng.randint(0, 10 ** 6), "steps": rng.randint(8, 80)}
    if kind in ("adjoint", "design", "fp64"):
        n = (_log(rng, 72, 220), _log(rng, 56, 120), _log(rng, 44, 72))
        c = {"kind": kind, "geom": "cpw", "template": "scaled", "nx": n[0], "ny": n[1], "nz": n[2],
             "steps": rng.randint(24, 120)}
        if kind != "fp64":
            c["segment"] = rng.randint(12, 70)
        return c
    geom = rng.choice(["column", "slab", "cpw", "cpw", "box", "box"])
    c = {"kind": kind, "geom": geom}
    if geom == "column":
        c.update(nx=1, ny=1, nz=_log(rng, 600, 9000))
    elif geom == "slab":
        nxy = rng.randint(1, 9)
        c.update(nx=nxy, ny=nxy, nz=_log(rng, 400, 4096))
    elif geom == "cpw":
        c.update(template="scaled", nx=_log(rng, 80, 900), ny=_log(rng, 56, 400), nz=_log(rng, 44, 200))
    else:
        kinds = ["periodic", "pec", "cpml"]
        c.update(nx=_log(rng, 20, 300), ny=_log(rng, 17, 200), nz=_log(rng, 19, 150), bcx=rng.choice(kinds),
                 bcy=rng.choice(kinds), bcz=rng.choice(kinds + ["mur"]), mu=rng.random() < 0.4,
                 edge_rule=rng.randint(0, 1), theta=rng.choice([0.5, 1.0]))
    cells = c["nx"] * c["ny"] * c["nz"]
    # longer stretches on smaller grids, none longer than the large grid's work
    c["steps"] = max(2, min(_log(rng, 3, 500), int(1.6e9 / cells)))
    return c


# ------------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=None)
def _workload(key):
    """The workload of a case: geometry, boundaries, sources, probes.  Its
    sigma map is 1 on metal cells here; the draws are made per seed."""
    c = dict(key)
    n = (c["nx"], c["ny"], c["nz"])
    geom = c["geom"]
    if geom == "column":
        z_if = max(40, n[2] * 350 // 4480)
        return W.reflection_column(1.0, nz=n[2], z_if=z_if, z_probe=z_if - 10, nsteps=c["steps"])
    if geom == "slab":
        nz = n[2]
        z = nz // 2
        return W.slab("mur", nxy=n[0], nz=nz, z_sc=z, probes_z=(z - nz // 6, z, z + 8, z + 16), z_src=nz // 10,
                      nsteps=c["steps"], sigma_sc=1.0)
    if geom == "box":
        return W.random_box(n=n, bc=(c["bcx"], c["bcy"], c["bcz"]), theta=c["theta"])
    t = c["template"]
    if t == "large":
        return W.cpw_large(sigma_override=1.0)
    if t == "full":
        return W.cpw(sigma_override=1.0)
    if t == "half":
        return W.cpw_adjoint(sigma_override=1.0)
    if t == "small":
        return W.cpw_small(n=n, sigma_override=1.0)
    return _scaled(n, 8, 6)


def _scaled(n, strip, gap, lam=3.0):
    """The 512 x 256 x 128 resonator scaled to a grid, as the batch's members are."""
    m = min(n)
    pml, margin = max(6, round(12 * m / 128)), max(2, round(4 * m / 128))
    free = n[1] - 2 * (pml + margin)
    while strip + 2 * gap > free - 4:
        strip, gap = max(4, strip - 2), max(2, gap - 2)
    return W.cpw(n=n, pml=pml, margin=margin, substrate_cells=max(8, round(32 * n[2] / 128)),
                 film_cells=max(2, round(4 * n[2] / 128)), strip_w=strip, gap_w=gap, lam_cells=lam, sigma_override=1.0)


@functools.lru_cache(maxsize=None)
def _members(key):
    """The batch's workloads: every axis of every member from three sizes,
    strip, gap and London depth drawn, all fixed by the case."""
    c = dict(key)
    rng = np.random.Generator(np.random.PCG64(W.BASE_SEED + c["variant"]))
    sizes = (c["small"], (c["small"] + c["large"]) // 2, c["large"])
    out = []
    for _ in range(c["count"]):
        n = tuple(int(rng.choice(sizes)) for _ in range(3))
        out.append(_scaled(n, int(rng.integers(4, 17)), int(rng.integers(4, 17)), float(rng.uniform(2.0, 6.0))))
    return out


def _key(case):
    return tuple(sorted((k, v) for k, v in case.items() if k != "name"))


def _maps(w, gen, case):
    """The four material maps on the GPU, float32: what the seed draws is drawn here."""
    def dev(a):
        return torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()

    def rnd(lo, hi):
        return torch.rand(w.eps_r.shape, generator=gen, device="cuda") * (hi - lo) + lo

    if case.get("geom") == "box":
        sc = torch.rand(w.eps_r.shape, generator=gen, device="cuda") < 0.5
        return [rnd(1.0, 4.0), rnd(1.0, 2.0) if case["mu"] else torch.ones_like(sc, dtype=torch.float32),
                torch.where(sc, rnd(30e-9, 60e-9), 0.0), rnd(0.0, 1e6)]
    eps, sig = dev(w.eps_r), dev(w.sigma)
    if case["kind"] in ("adjoint", "design"):   # a substrate drawn per cell
        eps = torch.where(eps > 1.0, rnd(10.0, 13.0), eps)
    return [eps, torch.ones_like(eps), dev(w.lambda_L), sig.mul_(rnd(0.0, 1e6))]


def _state(w, gen, off_walls=False):
    """A random state of all nine components, of the fields' usual magnitudes.
    off_walls: E and B off the walls and no Js, for the FP64 stepper, which
    takes a state as it is given (the FP32 path zeroes what the grid holds at
    zero)."""
    N = w.storage_dims()
    out = [(torch.rand((N[2], N[1], N[0]), generator=gen, device="cuda") * 2 - 1) * W.FIELD_SCALE[c] for c in range(9)]
    if off_walls:
        for c, a in enumerate(out):
            keep = torch.zeros_like(a)
            keep[1:-2, 1:-2, 1:-2] = 1.0 if c < 6 else 0.0
            a.mul_(keep)
    return out


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(1000003 * (int(seed) + 1))


def _probes(w):
    if w.probes:
        return w.probes
    f = W.C0 / (40 * w.d[2])   # boxes: one probe off the walls, a few frequencies
    return [W.Probe(comp=0, p=tuple(x // 2 for x in w.n), freqs=np.linspace(0.5 * f, 2.0 * f, 16))]


def _sources(w, case):
    amp = ADJOINT_AMP if case["kind"] in ("adjoint", "design") else 1.0
    return [(s.comp, s.lo, s.hi, s.amp * amp, s.kind, s.f, s.t0, s.tw) for s in w.sources]


def _edge_rule(case):
    return case.get("edge_rule", 0)


def _grid(w, maps, case, cls=tf.Grid):
    g = cls(w.n, w.d, w.theta, w.bc, w.cpml, dt=w.dt, courant=w.courant, edge_rule=_edge_rule(case))
    g.set_materials(*maps)
    for s in _sources(w, case):
        g.add_source(*s)
    for p in _probes(w):
        g.add_probe(p.comp, p.p, p.freqs, p.n0)
    return g


# ------------------------------------------------------------- prepare, run
def prepare(case, seed):
    gen = _gen(seed)
    kind = case["kind"]
    if kind == "batch":
        ws = _members(_key(case))
        grids = []
        for w in ws:
            g = _grid(w, _maps(w, gen, case), case)
            for c, a in enumerate(_state(w, gen)):
                g.set_field(c, a)
            grids.append(g)
        n = [math.prod(g.shape) for g in grids]
        return {"case": case, "grids": grids, "n": n, "out": torch.empty((9, sum(n)), device="cuda")}
    w = _workload(_key(case))
    maps = _maps(w, gen, case)
    if kind == "design":
        import copy
        w = copy.copy(w)
        w.sigma = maps[3].cpu().numpy()
        w.sources = [W.Source(comp=s[0], lo=s[1], hi=s[2], amp=s[3], kind=s[4], f=s[5], t0=s[6], tw=s[7])
                     for s in _sources(w, case)]
        return {"case": case, "w": w, "eps": maps[0].requires_grad_(), "lam": maps[2].requires_grad_()}
    if kind == "fp64":
        g = _grid(w, [m.cpu().numpy() for m in maps], case, tf.Grid64)
        for c, a in enumerate(_state(w, gen, off_walls=True)):
            g.set_field(c, a.cpu().numpy())
        return {"case": case, "g": g}
    g = _grid(w, maps, case)
    if kind == "adjoint":   # the state at rest, to start every call from
        rest = torch.empty(g.checkpoint_size(), dtype=torch.uint8, device="cuda")
        g.save_checkpoint(rest)
        return {"case": case, "g": g, "rest": rest}
    for c, a in enumerate(_state(w, gen)):
        g.set_field(c, a)
    out = None
    if kind == "step":
        out = [torch.empty(g.shape, dtype=torch.float32, device="cuda") for _ in range(9)]
    return {"case": case, "g": g, "out": out}


def run(state):
    case = state["case"]
    kind, steps = case["kind"], case["steps"]
    if kind == "batch":
        tf.batch_run(state["grids"], steps)
        o = 0
        for g, n in zip(state["grids"], state["n"]):
            for c in range(9):
                g.field(c, out=state["out"][c, o:o + n])
            o += n
        return {"fields": [state["out"][c] for c in range(9)],
                "spectra": np.concatenate([g.probe_dft(p) for g in state["grids"] for p in range(2)])}
    if kind == "design":
        eps, lam = state["eps"], state["lam"]
        eps.grad = lam.grad = None
        J = tfa.probe_power(eps, lam, state["w"], steps, probe=1, freq_index=0, segment=case["segment"])
        J.backward()
        return {"J": J, "grad_eps": eps.grad, "grad_lambda": lam.grad}
    g = state["g"]
    if kind == "adjoint":
        g.load_checkpoint(state["rest"])
        J, ge, gl = g.adjoint(steps, probe=1, freq_index=0, segment=case["segment"])
        return {"J": J, "grad_eps": ge, "grad_lambda": gl}
    g.step(steps)
    if kind == "watch":
        st = [g.field_stats(c) for c in range(9)]
        return {"sumsq": [s[0] for s in st], "maxabs": [s[1] for s in st], "nonfinite": [s[2] for s in st]}
    if kind == "fp64":
        return {"fields": [g.field(c) for c in range(9)], "spectra": [g.probe_dft(p) for p in range(len(g.freqs))]}
    return {"fields": [g.field(c, out=state["out"][c]) for c in range(9)],
            "spectra": [g.probe_dft(p) for p in range(len(g.freqs))]}


# --------------------------------------------------------------------- work
def _cells(case):
    if case["kind"] == "batch":
        return sum(w.ncells for w in _members(_key(case)))
    return case["nx"] * case["ny"] * case["nz"]


def work(case):
    """A step reads and writes E and B of every cell once (48 bytes in FP32)
    and takes about 45 operations; the CPML layers, Js and the maps come on
    top and are not counted.  Read-outs: every field read and written once.
    An adjoint step: a forward step, and the adjoint state and the gradient
    sums read and written once."""
    n, k, kind = _cells(case), case["steps"], case["kind"]
    if kind == "fp64":
        return {"bytes": 96 * n * k + 2 * 72 * n, "flops": 70 * n * k}
    if kind in ("adjoint", "design"):
        return {"bytes": (48 + 48 + 96) * n * k, "flops": 140 * n * k}
    return {"bytes": 48 * n * k + (36 if kind == "watch" else 72) * n, "flops": 45 * n * k}


# -------------------------------------------------- the same in 64 bits, plain
class _Plain:
    """The two-fluid Yee scheme in float64 torch, sub-step by sub-step on the
    integer-level state, every operation on whole arrays: E on edges, B on
    faces, Js on edges; forward differences of E and backward ones of H by
    rolled copies (what wraps at a wall is masked), Roden-Gedney CPML, a soft
    source, first-order Mur on z, probe sums.  Differentiable in eps_r and
    lambda_L."""

    def __init__(self, w, maps, case):
        self.n, self.N = w.n, w.storage_dims()
        self.per = [b == "periodic" for b in w.bc]
        self.mur = w.bc[2] == "mur"
        self.d = w.d
        self.dt = w.dt or w.courant / (W.C0 * math.sqrt(sum(1.0 / x ** 2 for x in w.d)))
        dt = self.dt
        dd = dict(dtype=torch.float64, device="cuda")
        shape = (self.N[2], self.N[1], self.N[0])
        pos = [torch.arange(self.N[a], device="cuda") for a in range(3)]
        view = [(1, 1, -1), (1, -1, 1), (-1, 1, 1)]

        def mask(halves, mur_wall=False):
            m = torch.ones(shape, dtype=torch.bool, device="cuda")
            for a in range(3):
                if self.per[a]:
                    continue
                ok = pos[a] < self.n[a]
                if not halves[a]:
                    ok = ok & (pos[a] >= 1)
                    if mur_wall and a == 2:
                        ok = (pos[a] == 0) | (pos[a] == self.n[a])
                m &= ok.view(view[a])
            return m

        self.mE = [mask([a == c for a in range(3)]) for c in range(3)]
        self.mB = [mask([a != c for a in range(3)]) for c in range(3)]
        self.wall = [mask([a == c for a in range(3)], True) for c in range(2)] if self.mur else None
        eps, mu, lam, sig = (m.double() for m in maps)
        sc = (lam > 0) & torch.isfinite(lam)
        kap = torch.where(sc, 1.0 / (torch.where(sc, lam, 1.0) ** 2 * W.MU0 * mu), 0.0)

        def grid(x):   # a cell map on the storage points
            for a in range(3):
                if not self.per[a]:
                    x = torch.cat([x, x.narrow(2 - a, self.n[a] - 1, 1)], dim=2 - a)
            return x

        def back(x, a):
            return torch.roll(x, 1, 2 - a)

        def four(x, c):   # sum over the cells that share edge c
            b1, b2 = (c + 1) % 3, (c + 2) % 3
            x = x + back(x, b1)
            return x + back(x, b2)

        def edge(x, c):
            if _edge_rule(case):
                return four(x, c) / 4
            cnt = four((x > 0).to(torch.float64), c)
            return torch.where(cnt > 0, four(x, c) / cnt.clamp(min=1.0), 0.0)

        geps, gmu, gkap, gsig = grid(eps), grid(mu), grid(kap), grid(sig)
        self.ca, self.cb, self.kap = [], [], []
        for c in range(3):
            e = W.EPS0 * four(geps, c) / 4
            s = edge(gsig, c) * dt / e
            den = 1 + w.theta * s
            self.ca.append((1 - (1 - w.theta) * s) / den)
            self.cb.append(dt / e / den)
            self.kap.append(torch.where(self.mE[c], edge(gkap, c), 0.0))
        self.imu = [2.0 / (W.MU0 * (gmu + back(gmu, c))) for c in range(3)]
        self.prof = {}
        self.slab = {}
        for a in range(3):
            if w.bc[a] != "cpml":
                continue
            cp = w.cpml[a]
            L, n = cp.ncells, self.n[a]
            for half in (0, 1):
                x = pos[a].to(torch.float64) + 0.5 * half
                rho = torch.where(x < L, (L - x) / L, torch.where(x > n - L, (x - (n - L)) / L, 0.0)).clamp(min=0.0)
                s, al = cp.sigma_max * rho ** cp.order, cp.alpha_max * (1 - rho)
                b = torch.exp(-(s + al) * dt / W.EPS0)
                cc = torch.where(s + al > 0, s * (b - 1) / torch.where(s + al > 0, s + al, 1.0), 0.0)
                on = rho > 0
                self.prof[a, half] = (torch.where(on, b, 0.0).view(view[a]), torch.where(on, cc, 0.0).view(view[a]))
            self.slab[a] = ((pos[a] < L) | (pos[a] >= n - L)).view(view[a])
        self.zero = torch.zeros(shape, **dd)

    def start(self, state):
        E = [torch.where(self.mE[c] | self.wall[c] if self.mur and c < 2 else self.mE[c], state[c].double(), 0.0)
             for c in range(3)]
        B = [torch.where(self.mB[c], state[3 + c].double(), 0.0) for c in range(3)]
        J = [torch.where(self.kap[c] > 0, state[6 + c].double(), 0.0) for c in range(3)]
        pb = {(c, a): self.zero for a in self.slab for c in range(3) if c != a}
        pe = dict(pb)
        S = E, B, J, pb, pe
        return E, B, J, self._psi_b(S), pe

    def _dE(self, E, e, a):
        return (torch.roll(E[e], -1, 2 - a) - E[e]) / self.d[a]

    def _dH(self, H, h, a):
        return (H[h] - torch.roll(H[h], 1, 2 - a)) / self.d[a]

    @staticmethod
    def _sg(c, a):
        return 1.0 if (a - c) % 3 == 1 else -1.0

    def _psi_b(self, S):
        E, _, _, pb, _ = S
        new = {}
        for (c, a), p in pb.items():
            b, cc = self.prof[a, 1]
            new[c, a] = torch.where(self.slab[a] & self.mB[c], b * p + cc * self._dE(E, 3 - c - a, a), 0.0)
        return new

    def _half_b(self, S):
        E, B, _, pb, _ = S
        out = []
        for c in range(3):
            r = 0.0
            for a in range(3):
                if a != c:
                    v = self._dE(E, 3 - c - a, a)
                    if (c, a) in pb:
                        v = v + pb[c, a]
                    r = r + self._sg(c, a) * v
            out.append(torch.where(self.mB[c], B[c] - 0.5 * self.dt * r, B[c]))
        return out

    def step(self, S, level, sources):
        E, B, J, pb, pe = S
        dt = self.dt
        B = self._half_b(S)
        J = [J[c] + 0.5 * dt * self.kap[c] * E[c] for c in range(3)]
        H = [B[c] * self.imu[c] for c in range(3)]
        new_pe = {}
        En = []
        for c in range(3):
            r = 0.0
            for a in range(3):
                if a == c:
                    continue
                v = self._dH(H, 3 - c - a, a)
                if (c, a) in pe:
                    b, cc = self.prof[a, 0]
                    new_pe[c, a] = torch.where(self.slab[a] & self.mE[c], b * pe[c, a] + cc * v, 0.0)
                    v = v + new_pe[c, a]
                r = r + self._sg(c, a) * v
            En.append(torch.where(self.mE[c], self.ca[c] * E[c] + self.cb[c] * (r - J[c]), E[c]))
        t = (level + 1) * dt
        for comp, lo, hi, amp, kind, f, t0, tw in sources:
            env = math.exp(-(t - t0) ** 2 / (2 * tw * tw)) if kind != W.SRC_SIN else 1.0
            s = env * (math.sin(2 * math.pi * f * t) if kind != W.SRC_GAUSS else 1.0)
            box = torch.zeros_like(self.zero)
            box[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]] = amp * s
            En[comp] = En[comp] + torch.where(self.mE[comp], box, 0.0)
        if self.mur:
            M = (W.C0 * dt - self.d[2]) / (W.C0 * dt + self.d[2])
            nz = self.n[2]
            for c in range(2):
                e = En[c].clone()
                for kw, ki in ((0, 1), (nz, nz - 1)):
                    v = E[c][ki] + M * (En[c][ki] - E[c][kw])
                    e[kw] = torch.where(self.wall[c][kw], v, E[c][kw])
                En[c] = e
        J = [J[c] + 0.5 * dt * self.kap[c] * En[c] for c in range(3)]
        S = En, B, J, pb, new_pe
        pb = self._psi_b(S)
        S = En, B, J, pb, new_pe
        return En, self._half_b(S), J, pb, new_pe

    def phases(self, p, level):
        ang = [2 * math.pi * math.fmod(float(f) * self.dt * level, 1.0) for f in p.freqs]
        return self.dt * np.exp(-1j * np.asarray(ang))

    def run(self, S, steps, sources, probes):
        X = [np.zeros(len(p.freqs), np.complex128) for p in probes]
        for n in range(steps):
            s = torch.stack([S[0][p.comp][p.p[2], p.p[1], p.p[0]] for p in probes]).tolist()
            for x, p, v in zip(X, probes, s):
                if n >= p.n0:
                    x += v * self.phases(p, n)
            S = self.step(S, n, sources)
        return list(S[0]) + list(S[1]) + list(S[2]), X


def _plain_adjoint(w, maps, case):
    from torch.utils.checkpoint import checkpoint
    eps = maps[0].double().requires_grad_()
    lam = maps[2].double().requires_grad_()
    g = _Plain(w, [eps, maps[1], lam, maps[3]], case)
    p = _probes(w)[1]
    src = _sources(w, case)
    S = g.start([g.zero] * 9)
    names = sorted(S[3])

    def flat(S):
        return [*S[0], *S[1], *S[2], *(S[3][k] for k in names), *(S[4][k] for k in names)]

    def block(n0, n1, *v):
        m = len(names)
        S = list(v[:3]), list(v[3:6]), list(v[6:9]), dict(zip(names, v[9:9 + m])), dict(zip(names, v[9 + m:]))
        X = torch.zeros(2, dtype=torch.float64, device="cuda")
        for n in range(n0, n1):
            if n >= p.n0:
                ph = g.phases(p, n)[0]
                s = S[0][p.comp][p.p[2], p.p[1], p.p[0]]
                X = X + torch.stack([s * ph.real, s * ph.imag])
            S = g.step(S, n, src)
        return (X, *flat(S))

    v, X = flat(S), 0.0
    for n0 in range(0, case["steps"], 8):
        x, *v = checkpoint(block, n0, min(n0 + 8, case["steps"]), *v, use_reentrant=False)
        X = X + x
    J = (X * X).sum()
    J.backward()
    return {"J": J.detach() if case["kind"] == "design" else float(J.detach()), "grad_eps": eps.grad,
            "grad_lambda": torch.where(maps[2] > 0, lam.grad, 0.0)}


def exact(case, seed):
    kind = case["kind"]
    gen = _gen(seed)
    if kind == "batch":
        fields, spectra = [[] for _ in range(9)], []
        for w in _members(_key(case)):
            maps = _maps(w, gen, case)
            state = _state(w, gen)
            g = _Plain(w, maps, case)
            f, X = g.run(g.start(state), case["steps"], _sources(w, case), _probes(w))
            for c in range(9):
                fields[c].append(f[c].reshape(-1))
            spectra += X
        return {"fields": [torch.cat(f) for f in fields], "spectra": np.concatenate(spectra)}
    w = _workload(_key(case))
    maps = _maps(w, gen, case)
    if kind in ("adjoint", "design"):
        return _plain_adjoint(w, maps, case)
    g = _Plain(w, maps, case)
    with torch.no_grad():
        f, X = g.run(g.start(_state(w, gen, kind == "fp64")), case["steps"], _sources(w, case), _probes(w))
    if kind == "watch":   # the statistics are of the half-level B and Js that the state holds: E alone has a value here
        sq = [float((f[c] ** 2).sum()) for c in range(3)]
        return {"sumsq": sq + [None] * 6, "maxabs": [float(f[c].abs().max()) for c in range(3)] + [None] * 6,
                "nonfinite": [None] * 9}
    return {"fields": f, "spectra": X}
