"""What this framework is used for, as cases that can be timed and checked.

A user of the framework runs gradient evaluations: the density goes in, a forward and an adjoint FDTD run
follow, the objective and dF/drho come out, hundreds of times per optimisation, with the density filter and
its chain rule around each.  The cases are such evaluations over the grid sizes of the configurations, the
serving stream, the paper's own setup and the precision study, the paper's time-domain mode, and the filter.
Only the number of time steps is smaller than in a real run (1000-18 000), so that a pass takes a fraction
of a second; a step's work does not depend on it.  The grid spacing and the pulse lengths follow the window,
so that source, objective and adjoint pulses lie inside it.

`exact` is a plain torch FP64 version of the same discrete method: whole-array operations, no code of the
package.
"""
import math

import numpy as np
import torch

import paper_2305_00234_gb300 as lib

C0 = 299792458.0
MU0 = 1.25663706212e-6
EPS0 = 1.0 / (MU0 * C0 * C0)


def _grad(name, n, cpml, steps, design, poles, nf=1, *, precision=32, source="dipole", layout=0, buffers="device",
          density="uniform", material="metal", dx=20e-9, courant=0.99 / math.sqrt(3.0)):
    return {"name": name, "kind": "gradient", "nx": n[0], "ny": n[1], "nz": n[2], "cpml": cpml, "steps": steps,
            "dnx": design[0], "dny": design[1], "dnz": design[2], "gapx": 2, "gapy": 2, "gapz": 2, "poles1": poles[0],
            "poles2": poles[1], "nf": nf, "precision": precision, "source": source, "layout": layout,
            "buffers": buffers, "density": density, "material": material, "dx": dx, "courant": courant}


def listed():
    return [
        # the smallest problem, in the all-FP64 build: parity checks and finite-difference studies
        _grad("fp64_32", (32, 32, 32), 8, 1000, (16, 16, 16), (0, 2), precision=64, dx=20e-9),
        # smallest grid of the serving stream, host density in, host gradient out; odd design extents
        _grad("serve_48", (48, 48, 48), 8, 1500, (21, 25, 28), (0, 1), buffers="host"),
        # the differentiation workload through torch.autograd
        _grad("autograd_64", (64, 64, 64), 8, 1200, (32, 32, 32), (0, 2), buffers="autograd"),
        # nothing even or aligned: odd x rows (no TMA, no cell pairs), two dispersive materials, two frequencies
        _grad("ragged_odd", (75, 61, 83), 9, 800, (31, 27, 37), (2, 2), 2),
        # middle and largest grids of the serving stream
        _grad("serve_128", (128, 128, 128), 8, 700, (56, 64, 72), (0, 4)),
        _grad("serve_192", (192, 192, 192), 8, 500, (96, 84, 108), (0, 3)),
        # the headline benchmark's grid, plane wave through a TF/SF plane, smooth density, three pole pairs and three
        # frequencies; a dielectric, so that the wave reaches the gap within the window
        _grad("plane_256", (256, 256, 256), 12, 600, (128, 128, 128), (0, 3), 3, source="plane", density="smooth",
              material="dielectric"),
        # the paper's own setup: 100 x 25 x 100 design, 6 x 25 x 6 gap (x and y exchanged), 20-cell CPML, gold in
        # air, one density per E sample, dt = dx / (2 c0), eight frequencies for the broadband objective
        dict(_grad("paper_gold", (96, 170, 170), 20, 1000, (25, 100, 100), (0, 3), 8, source="plane", layout=1,
                   density="smooth", material="gold", dx=10e-9, courant=0.5), gapx=25, gapy=6, gapz=6),
        # the precision study's grid: the largest state, six poles per component, anisotropic eps_inf
        _grad("study_512", (512, 512, 384), 16, 160, (256, 256, 192), (2, 4), 3, density="smooth"),
        # the paper's time-domain objective and history gradient by checkpoint-recompute (energies of 1e-50 J: FP64)
        dict(_grad("time_domain_52", (52, 48, 44), 4, 500, (16, 16, 16), (0, 2), precision=64), kind="paper_mode"),
        # cone filter, projection and chain rule around every gradient: the paper's 12-cell radius with a
        # steep projection on the headline design box, and a small radius on the paper's design box
        {"name": "filter_128", "kind": "filter", "nx": 128, "ny": 128, "nz": 128, "R": 12.0, "beta": 20.0, "eta": 0.5},
        {"name": "filter_paper", "kind": "filter", "nx": 25, "ny": 100, "nz": 100, "R": 3.5, "beta": 8.0, "eta": 0.5},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    u = rng.random()
    if u < 0.2:
        n = [int(_log(rng, 9, 161)) for _ in range(3)]
        return {"kind": "filter", "nx": n[0], "ny": n[1], "nz": n[2], "R": round(rng.uniform(1.2, 12.0), 2),
                "beta": round(_log(rng, 0.5, 20.0), 3), "eta": round(rng.uniform(0.3, 0.7), 3)}
    paper_mode = u < 0.3
    edge = _log(rng, 32, 72 if paper_mode else 300)
    n = [int(edge)] * 3 if rng.random() < 0.5 else [max(32, min(320, int(edge * rng.uniform(0.7, 1.4)))) for _ in range(3)]
    if rng.random() < 0.5:
        n = [v // 4 * 4 for v in n]
    cells = n[0] * n[1] * n[2]
    precision = 64 if paper_mode or (cells <= 72 ** 3 and rng.random() < 0.2) else 32
    steps = max(200, int(min(_log(rng, 300, 1200), (4.0e8 if precision == 64 else 6.0e9) / cells)))
    plane = n[0] <= 150 and not paper_mode and rng.random() < 0.4
    if plane:                                     # the wave crosses half the grid, partly in a dielectric
        steps = max(steps, 4 * n[0])
    cpml = min(rng.choice([6, 8, 9, 12, 16, 20]), min(n) // 5 - 1)
    design = [max(5, int(rng.uniform(0.4, 0.58) * v)) for v in n]
    case = _grad("", n, cpml, steps, design, (rng.randint(0, 2), rng.randint(1, 4)), rng.choice([1, 1, 2, 3, 5]),
                 precision=precision, source="plane" if plane else "dipole",
                 material="dielectric" if plane else rng.choice(["metal", "metal", "gold"]),
                 layout=0 if paper_mode else rng.choice([0, 0, 0, 1]), buffers=rng.choice(["device", "device", "host", "autograd"]),
                 density=rng.choice(["uniform", "smooth"]))
    del case["name"]
    if case["material"] == "gold":
        case.update(poles1=0, poles2=3)
    if paper_mode:
        case.update(kind="paper_mode", buffers="device")
    return case


# ---- inputs -------------------------------------------------------------------------------------------------

def _box(case, key):
    b = []
    for a, n in zip("xyz", (case["nx"], case["ny"], case["nz"])):
        d = case[key + a]
        b += [(n - d) // 2, (n - d) // 2 + d]
    return b


def _metal(rng, pairs):
    """Drude-like metal of the visible range: a Drude pole and (pairs - 1) passive Lorentz pairs."""
    wp, gam = rng.uniform(1.0e16, 1.4e16), rng.uniform(1e14, 6e14)
    poles = [(complex(-gam, 0.0), complex(-wp * wp / (2.0 * gam), 0.0))] + [_lorentz(rng, 3e15, 7e15, 0.3, 3.0)
                                                                        for _ in range(pairs - 1)]
    return {"eps_inf": [1.0] * 3, "sigma": [EPS0 * wp * wp / gam] * 3, "poles": [poles] * 3}


def _lorentz(rng, nu0, nu1, de0, de1):
    g, nu, de = rng.uniform(1e14, 1e15), rng.uniform(nu0, nu1), rng.uniform(de0, de1)
    return complex(-g, nu), complex(0.0, -de * (nu * nu + g * g) / (2.0 * nu))


def _dielectric(rng, pairs, eps_inf):
    """Resonances in the ultraviolet: transparent and dispersive in the visible."""
    return {"eps_inf": list(eps_inf), "sigma": [0.0] * 3,
            "poles": [[_lorentz(rng, 5e15, 8e15, 0.2, 1.0) for _ in range(pairs)]] * 3}


def _vacuum():
    return {"eps_inf": [1.0] * 3, "sigma": [0.0] * 3, "poles": [[], [], []]}


def _setup(case, seed):
    """Grid description and materials of a case: what a user's script builds on the host."""
    rng = np.random.default_rng(seed)
    n, M = (case["nx"], case["ny"], case["nz"]), case["steps"]
    T = M * case["courant"] * case["dx"] / C0
    tau = min(0.1 * T, 2.2e-15)                   # pulses of 8 tau in the first 80% of the window
    nf = case["nf"]
    # objective frequencies across the visible, further apart than the window resolves
    f = [C0 / 600e-9] if nf == 1 else np.linspace(C0 / 1000e-9, C0 / 350e-9, nf).tolist() if nf > 3 else \
        [C0 / w for w in (400e-9, 600e-9, 900e-9)[:nf]]
    plane = case["source"] == "plane"
    desc = {"nx": n[0], "ny": n[1], "nz": n[2], "dx": case["dx"], "courant": case["courant"], "n_steps": M,
            "cpml": [case["cpml"]] * 6, "cpml_m": 3.0, "cpml_sigma_scale": 1.0, "cpml_kappa_max": 1.0,
            "cpml_a_max": 0.05, "precision": case["precision"], "design_box": _box(case, "dn"),
            "gap_box": _box(case, "gap"), "freqs_hz": f, "freq_weights": [1.0] * nf, "src_kind": int(plane),
            "src_comp": 2, "src_pos": [case["cpml"] + 2, 0, 0] if plane else [v // 2 for v in n],
            "src_f0": C0 / 600e-9, "src_fwhm_hz": math.sqrt(2.0 * math.log(2.0)) / (math.pi * tau),
            "src_t0": 3.0 * tau, "src_amp": float(rng.uniform(0.5, 2.0)), "adj_tau": tau,
            "density_layout": case["layout"]}
    m1 = _vacuum()
    if case["poles1"]:
        m1 = _dielectric(rng, case["poles1"], (11.7, 11.7, 12.1))
    if case["material"] == "dielectric":
        m2 = _dielectric(rng, case["poles2"], (2.5, 2.5, 2.7))
    elif case["material"] == "metal":
        m2 = _metal(rng, case["poles2"])
    else:                                         # gold of the paper's Table 1
        m2 = {"eps_inf": [2.31] * 3, "sigma": [1.21e7] * 3,
              "poles": [[(-1.28e14 + 0j, -6.85e17 + 0j), (-6.36e14 - 3.89e15j, 2.06e15 + 8.70e14j),
                         (-2.96e15 - 6.12e15j, 1.60e13 + 1.47e16j)]] * 3}
    gamma = 5e4 if case["layout"] == 1 or case["kind"] == "paper_mode" else 0.0
    return desc, _vacuum(), m1, m2, gamma


def _smooth(x):
    for _ in range(2):
        x = torch.nn.functional.avg_pool3d(torch.nn.functional.pad(x[None, None], (3,) * 6, mode="replicate"), 7, 1)[0, 0]
    return (x - x.min()) / (x.max() - x.min())


def _density(case, seed, dtype):
    """Density on the design box (layout 1: one value per E sample, the three components' sets concatenated)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    l1 = case["layout"]
    nz, ny, nx = case["dnz"], case["dny"], case["dnx"]
    x = torch.rand((nz + l1, ny + l1, nx + l1), generator=g, device="cuda", dtype=torch.float32)
    if case["density"] == "smooth":
        x = _smooth(x)
    if l1:
        x = torch.cat([x[:, :, :nx].reshape(-1), x[:, :ny].reshape(-1), x[:nz].reshape(-1)])
    return x.to(dtype).contiguous()


def prepare(case, seed):
    if case["kind"] == "filter":
        g = torch.Generator(device="cuda").manual_seed(seed)
        shape = (case["nz"], case["ny"], case["nx"])
        rho = torch.rand(shape, generator=g, device="cuda")
        for _ in range(4):                        # nearly binary features a few voxels wide, as designs become
            rho = _smooth(rho)
        rho = torch.sigmoid(20.0 * (rho - 0.5))
        return {"case": case, "rho": rho.requires_grad_(), "g": torch.randn(shape, generator=g, device="cuda")}
    desc, bg, m1, m2, gamma = _setup(case, seed)
    dtype = torch.float64 if case["precision"] == 64 else torch.float32
    p = lib.Problem(desc, bg, m1, m2, gamma, stream=torch.cuda.current_stream().cuda_stream)
    rho = _density(case, seed, dtype)
    s = {"case": case, "problem": p, "rho": rho}
    if case["buffers"] == "host":
        s["rho"] = rho.cpu().numpy()
        s["out"] = np.empty_like(s["rho"])
    elif case["buffers"] == "autograd":
        rho.requires_grad_()
    else:
        s["out"] = torch.empty_like(rho)
    return s


def run(state):
    case, rho = state["case"], state["rho"]
    if case["kind"] == "filter":
        rho.grad = None
        rho_b = lib.FilterProject.apply(rho, case["R"], case["beta"], case["eta"])
        rho_b.backward(state["g"])
        return {"rho_b": rho_b.detach(), "grad": rho.grad}
    p = state["problem"]
    if case["kind"] == "paper_mode":
        p.set_density(rho)
        F = p.paper_forward()
        return {"F": np.float64(F), "grad": p.paper_gradient(state["out"], pole_pairing=1)}
    if case["buffers"] == "autograd":
        rho.grad = None
        F = lib.objective(rho, p)
        F.backward()
        return {"F": F.item(), "grad": rho.grad}
    p.set_density(rho)
    F, _ = p.forward()
    p.adjoint()
    return {"F": F, "grad": p.gradient(state["out"])}


def work(case):
    """Filter: arrays in and out; rows of the sphere at the same distance from the axis summed once, then one short
    correlation per distance.  Runs: the state (E, H, psi, pole currents) read and written once per time step, the
    density read, the DFTs written once at the end, the gradient written."""
    if case["kind"] == "filter":
        nv, R = case["nx"] * case["ny"] * case["nz"], case["R"]
        n = math.ceil(R) - 1
        rows = [y * y + z * z for y in range(-n, n + 1) for z in range(-n, n + 1) if y * y + z * z < R * R]
        taps = sum(2 * (2 * math.floor(math.sqrt(R * R - q)) + 1) for q in set(rows))
        return {"bytes": 24 * nv, "flops": 2 * nv * (len(rows) + taps)}
    ts = case["precision"] // 8
    n = (case["nx"], case["ny"], case["nz"])
    N, nd = n[0] * n[1] * n[2], case["dnx"] * case["dny"] * case["dnz"]
    P = 3 * (case["poles1"] + case["poles2"])
    slab = sum(N // v * 2 * case["cpml"] for v in n)
    runs = 3 if case["kind"] == "paper_mode" else 2
    step = 12 * N * ts + 8 * slab * ts + nd * ts * (4 * P + (3 if case["layout"] else 1))
    end = nd * (2 * 48 * case["nf"] + 2 * ts)
    flops = 36 * N + 20 * slab + nd * (20 * P + 12 + 12 * case["nf"])
    return {"bytes": float(runs * case["steps"] * step + end), "flops": float(runs * case["steps"] * flops)}


# ---- the same discrete method in plain FP64 torch -----------------------------------------------------------

def _view(v, axis):
    return v.reshape([-1 if a == axis else 1 for a in range(3)])


class _Run:
    """One FDTD run (forward or adjoint).  Arrays (nz, ny, nx); component c and derivative direction a count x, y, z."""

    def __init__(self, desc, bg, m1, m2, gamma, rho, case):
        d = self.d = desc
        self.dev = "cuda"
        self.n = (d["nx"], d["ny"], d["nz"])
        self.shape = self.n[::-1]
        self.dx, self.dt, self.M = d["dx"], d["courant"] * d["dx"] / C0, d["n_steps"]
        self.zero = lambda *s: torch.zeros(*s, dtype=torch.float64, device=self.dev)
        self.E, self.H = [self.zero(self.shape) for _ in range(3)], [self.zero(self.shape) for _ in range(3)]
        self.curl, self.tmp = self.zero(self.shape), self.zero(self.shape)
        self.pml = {}
        for a in range(3):
            lo, hi, n = d["cpml"][2 * a], d["cpml"][2 * a + 1], self.n[a]
            for sl in (slice(0, lo), slice(n - hi, n)):
                if sl.stop > sl.start:
                    for half in (0, 1):
                        self.pml.setdefault((a, half), []).append((sl, self.profile(a, sl, half)))
        self.psi = {}
        b = d["design_box"]
        l1 = case["layout"]
        self.wb = [b[0], b[1] + l1, b[2], b[3] + l1, b[4], b[5] + l1]
        w = self.wb
        self.box = (slice(w[4], w[5]), slice(w[2], w[3]), slice(w[0], w[1]))
        self.bshape = (w[5] - w[4], w[3] - w[2], w[1] - w[0])
        g = d["gap_box"]
        self.gap = tuple(slice(g[2 * a] - w[2 * a], g[2 * a + 1] - w[2 * a]) for a in (2, 1, 0))
        self.sb = tuple(slice(g[2 * a], g[2 * a + 1]) for a in (2, 1, 0))
        ex = [b[2 * a + 1] - b[2 * a] for a in range(3)]
        self.sets = [tuple(slice(0, ex[a] + (l1 if a != c else 0)) for a in (2, 1, 0)) for c in range(3)]
        self.rho, self.mask, off = [], [], 0
        for c in range(3):
            r, m = self.zero(self.bshape), torch.zeros(self.bshape, dtype=torch.bool, device=self.dev)
            sizes = [s.stop for s in self.sets[c]]
            cnt = sizes[0] * sizes[1] * sizes[2]
            r[self.sets[c]] = (rho[off:off + cnt] if l1 else rho).reshape(sizes)
            off += cnt
            m[self.sets[c]] = True
            m[self.gap] = False
            self.rho.append(r)
            self.mask.append(m)
        self.mats(bg, m1, m2, gamma)
        self.Q = [torch.zeros((len(self.al[c]),) + self.bshape, dtype=torch.complex128, device=self.dev) for c in range(3)]
        w_ = 2 * math.pi * torch.tensor(d["freqs_hz"], dtype=torch.float64, device=self.dev) * self.dt
        ang = w_[:, None] * torch.arange(1, self.M + 1, dtype=torch.float64, device=self.dev)
        self.ph = torch.cat([torch.cos(ang), -torch.sin(ang)])               # (2F, M)
        self.acc = None

    def profile(self, a, sl, half):
        d, n = self.d, self.n[a]
        lo, hi = d["cpml"][2 * a], d["cpml"][2 * a + 1]
        u = np.arange(sl.start, sl.stop) + 0.5 * half
        dep = np.where(u < lo, (lo - u) / max(lo, 1), np.where(u > n - hi, (u - (n - hi)) / max(hi, 1), 0.0))
        m = d["cpml_m"]
        sig = d["cpml_sigma_scale"] * 0.8 * (m + 1) / (MU0 * C0 * self.dx) * dep ** m
        kap = 1.0 + (d["cpml_kappa_max"] - 1.0) * dep ** m
        al = np.where(dep > 0, d["cpml_a_max"] * (1 - dep), 0.0)
        b = np.exp(-(sig / kap + al) * self.dt / EPS0)
        with np.errstate(invalid="ignore", divide="ignore"):
            c = np.where(sig > 0, sig * (b - 1) / (sig * kap + kap * kap * al), 0.0)
        return tuple(_view(torch.tensor(v, device=self.dev), 2 - a) for v in (1 / kap, b, c))

    def mats(self, bg, m1, m2, gamma):
        dt = self.dt
        self.ca, self.cb, self.al, self.be, self.D, self.N, self.kap = [], [], [], [], [], [], []
        for c in range(3):
            base, s = EPS0 * bg["eps_inf"][c] / dt, 0.5 * bg["sigma"][c]
            self.ca.append((base - s) / (base + s))
            self.cb.append(1.0 / (base + s))
            al, be, DN = [], [], []
            for m in (m1, m2):
                a = np.array([p[0] for p in m["poles"][c]], dtype=complex)
                r = np.array([p[1] for p in m["poles"][c]], dtype=complex)
                beta = EPS0 * r * np.expm1(a * dt) / (2 * a)
                al.append(np.expm1(a * dt))
                be.append(beta)
                e, s = EPS0 * m["eps_inf"][c] / dt, 0.5 * m["sigma"][c] + 2 / dt * beta.real.sum()
                DN.append((e + s, e - s))
            rho = self.rho[c]
            gm = 0.5 * gamma * rho * (1 - rho)
            self.D.append(DN[0][0] + rho * (DN[1][0] - DN[0][0]) + gm)
            self.N.append(DN[0][1] + rho * (DN[1][1] - DN[0][1]) - gm)
            self.kap.append((len(al[0]), 1 - rho, rho))
            self.al.append(np.concatenate(al))
            self.be.append(np.concatenate(be))

    def diff(self, src, a, half, key):
        """d along direction a (forward for half 1: E -> H; backward for 0) times dx, CPML-stretched, in self.tmp."""
        ax, t = 2 - a, self.tmp
        n = src.shape[ax]
        if half:
            torch.sub(src.narrow(ax, 1, n - 1), src.narrow(ax, 0, n - 1), out=t.narrow(ax, 0, n - 1))
            torch.neg(src.narrow(ax, n - 1, 1), out=t.narrow(ax, n - 1, 1))
        else:
            torch.sub(src.narrow(ax, 1, n - 1), src.narrow(ax, 0, n - 1), out=t.narrow(ax, 1, n - 1))
            t.narrow(ax, 0, 1).copy_(src.narrow(ax, 0, 1))
        yield t
        for i, (sl, (kinv, b, c)) in enumerate(self.pml.get((a, half), [])):
            v = t.narrow(ax, sl.start, sl.stop - sl.start)
            psi = self.psi.setdefault((key, i), torch.zeros_like(v))
            psi.mul_(b).addcmul_(v, c.expand_as(v))
            v.mul_(kinv).add_(psi)
        yield t

    def run(self, drive, einc=None, hinc=None):
        """drive(n): list of (component, index, value) added to curl H at step n.  Returns the DFT (F, 3, box)."""
        i0 = self.d["src_pos"][0] if einc is not None else None
        ch, K = self.dt / MU0 / self.dx, 16
        ring = self.zero((K, 3) + self.bshape)
        self.acc = self.zero((self.ph.shape[0], ring[0].numel()))
        for n in range(self.M):
            for c in range(3):
                u, v = (c + 1) % 3, (c + 2) % 3
                for src, a, sign in ((self.E[v], u, -ch), (self.E[u], v, ch)):
                    st = self.diff(src, a, 1, ("H", c, a))
                    t = next(st)
                    if i0 is not None and c == 1 and a == 0:
                        t[:, :, i0 - 1] -= einc[n]
                    next(st)
                    self.H[c].add_(t, alpha=sign)
            terms = drive(n)
            for c in range(3):
                u, v = (c + 1) % 3, (c + 2) % 3
                for k, (src, a) in enumerate(((self.H[v], u), (self.H[u], v))):
                    st = self.diff(src, a, 0, ("E", c, a))
                    t = next(st)
                    if i0 is not None and c == 2 and a == 0:
                        t[:, :, i0] -= hinc[n]
                    next(st)
                    if k == 0:
                        self.curl.copy_(t)
                    else:
                        self.curl.sub_(t)
                self.curl.mul_(1.0 / self.dx)
                for cc, idx, val in terms:
                    if cc == c:
                        self.curl[idx] += val
                E = self.E[c]
                old, cur = E[self.box].clone(), self.curl[self.box]
                E.mul_(self.ca[c]).add_(self.curl, alpha=self.cb[c])
                sq, Q = 0.0, self.Q[c]
                nk, k1, k2 = self.kap[c]
                for p in range(len(self.al[c])):
                    g = 2 / self.dt * self.al[c][p]
                    sq = sq + (k1 if p < nk else k2) * (g.real * Q[p].real - g.imag * Q[p].imag)
                new = (self.N[c] * old + cur - sq) / self.D[c]
                es = new + old
                for p in range(len(self.al[c])):
                    Q[p].mul_(1 + complex(self.al[c][p])).add_(es, alpha=complex(self.be[c][p]))
                E[self.box] = torch.where(self.mask[c], new, E[self.box])
                for a in range(3):
                    if a != c:
                        E.narrow(2 - a, 0, 1).zero_()
                ring[n % K, c] = E[self.box]
            if n % K == K - 1 or n == self.M - 1:
                cnt = n % K + 1
                self.acc += self.ph[:, n + 1 - cnt:n + 1] @ ring[:cnt].reshape(cnt, -1)
            yield n
        F = self.ph.shape[0] // 2
        self.dft = torch.complex(self.acc[:F], self.acc[F:]).reshape((F, 3) + self.bshape)


def _pulse(d, t):
    tau = math.sqrt(2 * math.log(2)) / (math.pi * d["src_fwhm_hz"])
    x = t - d["src_t0"]
    return math.exp(-x * x / (2 * tau * tau)) * math.sin(2 * math.pi * d["src_f0"] * x)


def _incident(d, dt):
    """E and H of the one-sided TF/SF plane wave at its plane: a 1-D Yee line in vacuum, hard-driven at node 0."""
    M, off = d["n_steps"], 2
    L = off + math.ceil(0.6 * M) + 16
    e, h, ei, hi = np.zeros(L), np.zeros(L), np.zeros(M), np.zeros(M)
    ce = dt / (EPS0 * d["dx"])
    e[0] = d["src_amp"] * _pulse(d, 0.0)
    for n in range(M):
        ei[n] = e[off]
        h += dt / (MU0 * d["dx"]) * (np.append(e[1:], 0.0) - e)
        hi[n] = h[off - 1]
        e[1:] += ce * (h[1:] - h[:-1])
        e[0] = d["src_amp"] * _pulse(d, (n + 1) * dt)
    return ei, hi


def _forward(desc, bg, m1, m2, gamma, rho, case):
    f = _Run(desc, bg, m1, m2, gamma, rho, case)
    if desc["src_kind"] == 1:
        ei, hi = _incident(desc, f.dt)
        return f, f.run(lambda n: [], ei, hi)
    i, j, k = desc["src_pos"]
    amp = desc["src_amp"] * EPS0 / f.dt
    return f, f.run(lambda n: [(desc["src_comp"], (k, j, i), amp * _pulse(desc, (n + 0.5) * f.dt))])


def _exact_gradient(case, seed):
    desc, bg, m1, m2, gamma = _setup(case, seed)
    rho = _density(case, seed, torch.float64 if case["precision"] == 64 else torch.float32).double()
    f, steps = _forward(desc, bg, m1, m2, gamma, rho, case)
    for _ in steps:
        pass
    fw, F, dt, M = f.dft, len(desc["freqs_hz"]), f.dt, desc["n_steps"]
    gapd = fw[(slice(None), slice(None)) + f.gap]
    obj = float((gapd.abs() ** 2).sum())
    w = 2 * math.pi * np.array(desc["freqs_hz"])
    x = (np.arange(M) + 0.5) * dt - 4 * desc["adj_tau"]
    env = np.exp(-x * x / (2 * desc["adj_tau"] ** 2))
    basis = np.stack([g(wf * x) * env for wf in w for g in (np.cos, np.sin)])            # (2F, M)
    spec = basis @ np.exp(-1j * np.outer(np.arange(M) * dt, w))                              # (2F, F)
    A = np.stack([spec.real.T, spec.imag.T], 1).reshape(2 * F, 2 * F)
    rhs = torch.stack([gapd.real, -gapd.imag], 1).reshape(2 * F, -1).cpu().numpy()
    drive = torch.tensor(basis.T @ np.linalg.solve(A, rhs), device="cuda").reshape((M, 3) + gapd.shape[2:])
    adj = _Run(desc, bg, m1, m2, gamma, rho, case)
    for _ in adj.run(lambda n: [(c, adj.sb, drive[n, c]) for c in range(3)]):
        pass
    z, parts = np.exp(1j * w * dt), []
    for c in range(3):
        h = [[be * (z + 1) / (z - 1 - al) + np.conj(be) * (z + 1) / (z - 1 - np.conj(al))
              for al, be in zip(f.al[c], f.be[c])]][0]
        P1 = f.kap[c][0]
        ps = sum(h[P1:], 0 * z) - sum(h[:P1], 0 * z)
        dA = (EPS0 * (m2["eps_inf"][c] - m1["eps_inf"][c]) * (z - 1) + (m2["sigma"][c] - m1["sigma"][c]) * dt * (z + 1) / 2 +
              (z - 1) * ps) / dt
        dB = gamma * (z + 1) / 2
        G = 0.0
        for q in range(F):
            dY = complex(dA[q]) + (1 - 2 * f.rho[c]) * complex(dB[q])
            G = G - 2 * (dY * fw[q, c] * adj.dft[q, c]).real
        parts.append(torch.where(f.mask[c], G, torch.zeros_like(G)))
    grad = torch.cat([p[s].reshape(-1) for p, s in zip(parts, f.sets)]) if case["layout"] else parts[0] + parts[1] + parts[2]
    return {"F": obj, "grad": grad}


def _exact_paper(case, seed):
    """The time-domain energy of the gap and its gradient from stored histories, the pole term paired with the
    adjoint level before."""
    desc, bg, m1, m2, gamma = _setup(case, seed)
    rho = _density(case, seed, torch.float64)
    M = desc["n_steps"]
    f, steps = _forward(desc, bg, m1, m2, gamma, rho, case)
    he, hq = f.zero((M + 1, 3) + f.bshape), f.zero((M, 3) + f.bshape)

    def poles(c):
        k = f.kap[c][0]
        return f.Q[c][k:].real.sum(0) - f.Q[c][:k].real.sum(0)

    before = [poles(c) for c in range(3)]
    for n in steps:
        for c in range(3):
            he[n + 1, c] = f.E[c][f.box]
            now = poles(c)
            hq[n, c] = now - before[c]
            before[c] = now
    gh = he[(slice(None), slice(None)) + f.gap]
    obj = np.float64(0.5 * EPS0 * desc["dx"] ** 3 * f.dt * float((gh ** 2).sum()))
    adj = _Run(desc, bg, m1, m2, gamma, rho, case)
    G, am = f.zero(f.bshape), [f.zero(f.bshape) for _ in range(3)]
    for m in adj.run(lambda n: [(c, adj.sb, EPS0 * gh[M - n - 1, c]) for c in range(3)]):
        L = M - 1 - m
        for c in range(3):
            ap = adj.E[c][f.box]
            e = he[L, c]
            ds = m2["sigma"][c] - m1["sigma"][c] + (1 - 2 * rho) * gamma
            G += -EPS0 * (m2["eps_inf"][c] - m1["eps_inf"][c]) * e * (ap - am[c]) - ds * f.dt * e * 0.5 * (ap + am[c]) \
                - 2 * hq[L, c] * am[c]
            am[c] = ap.clone()
    G[f.gap] = 0.0
    return {"F": obj, "grad": G * desc["dx"] ** 3}


def _exact_filter(case, seed):
    s = prepare(case, seed)
    rho, gb = s["rho"].detach().double(), s["g"].double()
    R, beta, eta = case["R"], case["beta"], case["eta"]
    n = math.ceil(R) - 1
    q = torch.arange(-n, n + 1, dtype=torch.float64, device="cuda")
    w = (R - torch.sqrt(q[:, None, None] ** 2 + q[:, None] ** 2 + q ** 2)).clamp_min(0.0)
    size = [v + 2 * n for v in rho.shape]
    spec = torch.fft.rfftn(w, size)

    def cone(x):
        y = torch.fft.irfftn(torch.fft.rfftn(x, size) * spec, size)
        return y[n:n + x.shape[0], n:n + x.shape[1], n:n + x.shape[2]]

    W = cone(torch.ones_like(rho))
    t = cone(rho) / W
    den = math.tanh(beta * eta) + math.tanh(beta * (1 - eta))
    th = torch.tanh(beta * (t - eta))
    return {"rho_b": (math.tanh(beta * eta) + th) / den, "grad": cone(gb * beta * (1 - th * th) / den / W)}


def exact(case, seed):
    if case["kind"] == "filter":
        return _exact_filter(case, seed)
    return _exact_paper(case, seed) if case["kind"] == "paper_mode" else _exact_gradient(case, seed)
