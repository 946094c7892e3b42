"""What a user of the PIC library has it do, as measurable cases.

Every case goes through the public entry points (``Sim`` / ``Batch`` of the binding and the
C ABI's device-side reads), over the range the library serves: both precision families,
power-of-two, 7-smooth and prime z lengths, radial grids from 48 to 1024 nodes, one to three
modes, finite and infinite stencil order, sorted every cycle or every few, with and without
the moving window.  ``exact`` restates the method in plain 64-bit torch.

Kinds:
  cycle      a running simulation: ``cycles`` full PIC cycles, then a dump of the state (E, B,
             rho^n and the particles by id), with the beam's quality when ``diag`` is set
  particles  a driver that hands in a particle set, sorts it, pushes it with its current
             deposit and deposits rho (the stage calls of a program with its own field solver)
  field      the field solver by itself: ``cycles`` field steps on given sources
  scan       independent simulations of uneven size advanced by one captured graph
  setup      a new handle: Bessel zeros, Hankel matrices and their pseudo-inverses, tables
"""
import ctypes
import math

import numpy as np
import torch

from paper_1611_05712_gb300 import binding as bd
from paper_1611_05712_gb300 import workloads as W

FORMS = {"fp64": bd.PIC_FP64, "tf32x3": bd.PIC_MIXED_TF32X3, "bf16x6": bd.PIC_MIXED_BF16X6}
CELL = 0.05e-6


def _case(kind, form, Nz, Nr, Nm, order, **more):
    c = {"kind": kind, "form": form, "Nz": Nz, "Nr": Nr, "Nm": Nm, "order": order, "density": 1e24, "ppz": 1,
         "ppr": 1, "ppt": 1, "beam": 20000, "cdt": 1.0, "cycles": 1, "sort_every": 1, "window": False, "diag": False}
    c.update(more)
    return c


def listed():
    wake = {"density": 1e23, "ppt": 2, "beam": 300000}
    dense = {"density": 1e23, "ppz": 2, "ppr": 2, "ppt": 3}
    return [
        # the small plasma + beam run: 36 k particles, where launches and latency count
        dict(_case("cycle", "fp64", 256, 64, 2, 0, cycles=10), name="small_cycle_fp64"),
        # the beam-driven wakefield the headline metric is quoted on, plain FP64
        dict(_case("cycle", "fp64", 2048, 256, 2, 32, cycles=4, sort_every=4, diag=True, **wake), name="wake_cycle_fp64"),
        # an FP64 member of an order / resolution scan: uneven z length, wide radial grid
        dict(_case("cycle", "fp64", 1800, 400, 2, 16, cdt=0.5, cycles=1), name="uneven_cycle_fp64"),
        # the same wakefield in the mixed form, as the long production runs use it
        dict(_case("cycle", "tf32x3", 2048, 256, 2, 32, cycles=8, sort_every=4, diag=True, **wake), name="wake_cycle_tf32"),
        # ... and following the beam in the moving window, BF16 split, sorted every cycle
        dict(_case("cycle", "bf16x6", 2048, 256, 2, 64, cycles=8, window=True, **wake), name="window_cycle_bf16"),
        # the large single run: about 100 M particles
        dict(_case("cycle", "tf32x3", 8192, 1024, 3, 32, cycles=2, **dict(dense, beam=2000000)), name="large_cycle_tf32"),
        # eight uneven simulations of a parameter scan in one captured graph
        dict(_case("scan", "tf32x3", 0, 0, 0, 0, cycles=2, members=8, base=4000), name="scan_graph_tf32"),
        # the particle stages alone, crowded cells (12 per cell, three modes), FP64
        dict(_case("particles", "fp64", 1024, 128, 3, 32, **dict(dense, beam=31250)), name="dense_particles_fp64"),
        # ... and in the mixed form on an odd-sized single-mode grid
        dict(_case("particles", "bf16x6", 3125, 176, 1, 32, **dict(dense, ppt=1)), name="odd_particles_bf16"),
        # the field solver alone: FP64, ragged sizes
        dict(_case("field", "fp64", 1323, 144, 3, 48, cycles=2), name="ragged_field_fp64"),
        # ... mixed form, the upper end of the scan's grids
        dict(_case("field", "tf32x3", 3600, 448, 2, 0, cycles=4), name="scan_field_tf32"),
        # a new scan member's handle
        dict(_case("setup", "tf32x3", 1000, 240, 2, 32), name="scan_setup"),
    ]


def _between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _length(rng, form, lo, hi):
    """A z length: mostly 7-smooth (a quarter of them powers of two), now and then any integer."""
    n = _between(rng, lo, hi)
    u = rng.random()
    if u < 0.25:
        return 1 << (n.bit_length() - 1)
    if u < 0.35:
        return min(n, 2048 if form == "fp64" else 4096)
    while not W._is_7_smooth(n):
        n -= 1
    return n


def draw(rng):
    kind = rng.choice(["cycle", "cycle", "particles", "field", "field", "setup"])
    form = rng.choice(["fp64", "tf32x3", "bf16x6"])
    lo, hi = (400, 3000) if kind == "setup" else (200, 4096)
    Nr = _between(rng, 48, 420 if kind == "setup" or form == "fp64" else 640)
    Nz = _length(rng, form, lo, hi)
    Nm = rng.choice([1, 2, 2, 3])
    order = rng.choice([8, 16, 24, 32, 48, 64, 0])
    more = {"cdt": rng.choice([0.5, 1.0]), "beam": _between(rng, 5000, 200000)}
    if kind == "cycle":
        more.update(cycles=rng.choice([1, 2, 4]), sort_every=rng.choice([1, 4]), ppt=rng.choice([1, 2]),
                    density=rng.choice([1e23, 1e24]))
    elif kind == "particles":
        more.update(ppz=rng.choice([1, 2]), ppt=rng.choice([1, 2, 3]), density=rng.choice([1e23, 1e24]))
    elif kind == "field":
        more.update(cycles=rng.choice([1, 2, 4]))
    return _case(kind, form, Nz, Nr, Nm, order, **more)


# ---------------------------------------------------------------------------- inputs
def _workload(c):
    return W.Workload("case", c["Nz"], c["Nr"], c["Nm"], CELL, CELL, c["cdt"] * CELL / W.C_LIGHT, c["order"], c["density"],
                      (c["ppz"], c["ppr"], c["ppt"]))


def _particles(c, seed):
    """Uniform cold plasma on sub-cell positions with a random azimuth per ring, and a warm
    Gaussian electron beam (0.1 % energy spread, about 0.5 mm mrad) inside the box.  Returns
    the arrays on the GPU, the number of plasma particles and the beam's Lorentz factor."""
    g = torch.Generator("cuda").manual_seed(int(seed))
    f8 = {"dtype": torch.float64, "device": "cuda"}
    Nz, Nr, pz, pr, pt, n = c["Nz"], c["Nr"], c["ppz"], c["ppr"], c["ppt"], c["beam"]
    nz, nr = Nz * pz, Nr * pr
    z = ((torch.arange(nz, **f8) + 0.5) * (CELL / pz)).view(-1, 1, 1)
    r = ((torch.arange(nr, **f8) + 0.5) * (CELL / pr)).view(1, -1, 1)
    th = 2 * math.pi * (torch.rand((nz, nr, 1), generator=g, **f8) + torch.arange(pt, **f8) / pt)
    flat = lambda a: a.expand(nz, nr, pt).reshape(-1)  # noqa: E731
    plasma = {"x": flat(r * torch.cos(th)), "y": flat(r * torch.sin(th)), "z": flat(z),
              "w": flat(c["density"] * 2 * math.pi * r * (CELL / pr) * (CELL / pz) / pt)}
    n_plasma = nz * nr * pt
    sr, sz, gamma = min(3e-6, Nr * CELL / 8), min(6e-6, Nz * CELL / 16), 1000.0
    a = torch.randn((6, n), generator=g, **f8).clamp_(-3.5, 3.5)
    gam = gamma * (1 + 1e-3 * a[3])
    kick = 0.5e-6 / sr * W.C_LIGHT
    beam = {"x": sr * a[0], "y": sr * a[1], "z": 0.6 * Nz * CELL + sz * a[2], "ux": kick * a[4], "uy": kick * a[5],
            "uz": W.C_LIGHT * torch.sqrt(gam * gam - 1), "w": torch.full((n,), 3e7 / n, **f8)}
    zero = torch.zeros(n_plasma, **f8)
    P = {k: torch.cat([plasma.get(k, zero), beam[k]]) for k in bd.SOA}
    P["id"] = torch.arange(n_plasma + n, dtype=torch.int32, device="cuda")
    return P, n_plasma, gamma


def _members(c):
    """The sizes of a scan's simulations (the scan workload's own distribution)."""
    for k in range(c["members"]):
        w = W.scan_member(k, base_seed=c["base"])
        yield dict(c, kind="cycle", Nz=w.Nz, Nr=w.Nr, Nm=w.Nm, order=w.order_p,
                   cdt=round(w.dt * W.C_LIGHT / CELL, 3))


def _sim(c, P, n_plasma, gamma, stream=None):
    n = len(P["x"])
    s = bd.Sim.from_workload(_workload(c), P, n_plasma, [(n_plasma, n, gamma)], precision=FORMS[c["form"]],
                             capacity=n + (n_plasma // 4 if c["window"] else 0), stream=stream)
    s.set_sort_interval(c["sort_every"])
    if c["window"]:
        s.window_setup(n_plasma, period=1 if c["cdt"] == 1.0 else 2, n_reserve=n_plasma // 4)
    s.sync()
    return s


class _State:
    pass


def prepare(case, seed):
    st = _State()
    st.case = c = dict(case)
    if c["kind"] == "setup":
        w = _workload(c)
        dr = CELL * (1 + 1e-3 * (seed % 97))   # a resolution scan: another radial cell per member
        st.cfg = bd.make_config(w.Nz, w.Nr, w.Nm, w.dz, dr, w.dt, w.order_p, True, FORMS[c["form"]], 1000)
        return st
    if c["kind"] == "scan":
        st.sims = []
        for k, m in enumerate(_members(c)):
            P, npl, gamma = _particles(m, seed * 1000 + k)
            torch.cuda.synchronize()
            st.sims.append(_sim(m, P, npl, gamma, torch.cuda.Stream()))
        st.batch = bd.Batch(st.sims, cycles=c["cycles"])
        return st
    P, npl, gamma = _particles(c, seed)
    st.beam = (npl, len(P["x"]))
    st.sim = _sim(c, P, npl, gamma)
    if c["kind"] == "particles":
        st.P = P
    if c["kind"] == "field":
        st.sim.deposit()
    st.sim.sync()
    return st


# ---------------------------------------------------------------------------- one pass
def _buffer(s, name):
    """A library buffer copied into a tensor on the GPU."""
    kind = s._dtype(name)
    t = torch.empty(s._shape(name) if name not in ("KEYS", "PERM") else (s.num_particles(),),
                    dtype=torch.from_numpy(np.empty(0, kind)).dtype, device="cuda")
    bd._check(s.lib.pic_copy_buffer(s.h, bd.BUF[name], ctypes.c_void_p(t.data_ptr()), t.numel() * t.element_size(), 0),
              "pic_copy_buffer")
    return t


def _by_id(s):
    """The particles on the GPU as [7 (x y z ux uy uz w), id], in the form's own width."""
    n = s.num_particles()
    a = torch.empty((7, n), dtype=torch.float64, device="cuda")
    ids = torch.empty(n, dtype=torch.int32, device="cuda")
    ptrs = (ctypes.c_void_p * 7)(*[a[k].data_ptr() for k in range(7)])
    bd._check(s.lib.pic_read_particles(s.h, ptrs, ctypes.c_void_p(ids.data_ptr()), n, 0), "pic_read_particles")
    if s.cfg.precision != bd.PIC_FP64:
        a = a.float()
    out = torch.empty_like(a)
    out[:, ids] = a
    return {k: out[i] for i, k in enumerate(bd.SOA)}


DIAG = ("W", "z_mean", "sigma_z", "gamma_mean", "emit_nx", "emit_ny", "sigma_gamma_mean")


def run(st):
    c = st.case
    if c["kind"] == "setup":
        s = bd.Sim(st.cfg)
        out = {k: _buffer(s, k) for k in ("KPERP", "HANKEL_INV", "HANKEL_FWD", "KZ_MOD")}
        s.close()
        return out
    if c["kind"] == "scan":
        st.batch.launch(1)
        st.batch.origin.synchronize()
        return [{k: _buffer(s, k) for k in ("E", "B", "RHO_PREV_H")} for s in st.sims]
    s = st.sim
    if c["kind"] == "particles":
        s.write_particles(st.P)
        s.sort()
        out = {"KEYS": _buffer(s, "KEYS"), "PERM": _buffer(s, "PERM")}
        s.gather_push(True)
        s.deposit(bd.PIC_DEP_RHO)
        out["DEP"] = _buffer(s, "DEP")
    elif c["kind"] == "field":
        for _ in range(c["cycles"]):
            s.field_step()
        return {k: _buffer(s, k) for k in ("E", "B", "EH", "BH", "RHO_PREV_H")}
    else:
        s.step(c["cycles"])
        out = {k: _buffer(s, k) for k in ("E", "B", "RHO_PREV_H")}
    out.update(_by_id(s))
    if c["diag"]:
        d = s.diagnostics(*st.beam)
        wide = np.float64 if c["form"] == "fp64" else np.float32
        out.update({"beam_" + k: wide(d[k]) for k in DIAG})
    return out


# ---------------------------------------------------------------------------- least work
def _work(c):
    """Bytes and operations of one cycle (or pass) that the method cannot do without."""
    r = 8 if c["form"] == "fp64" else 4
    Nz, Nr, Nm = c["Nz"], c["Nr"], c["Nm"]
    n = Nz * c["ppz"] * Nr * c["ppr"] * c["ppt"] + c["beam"]
    G = Nm * Nr * Nz
    state = (6 * 8 + 8 + 4) if r == 8 else 52
    push = n * (state + (6 * 8 if r == 8 else 44))
    deposit, gather_push = n * 40 * (2 * Nm - 1), n * (200 + 6 * (8 + 21 * (Nm - 1)))
    dht, fft = 4.0 * Nz * Nr * Nr * Nm, 5.0 * Nz * math.log2(Nz) * Nm * Nr
    solve = 10 * dht + 10 * fft + 150.0 * G
    if c["kind"] == "particles":
        return {"bytes": 60 * n + push + 8 * n + 10 * G * 2 * r, "flops": deposit + gather_push}
    if c["kind"] == "field":
        # sources in, the spectral state in and out, E and B out, the tables of the update
        return {"bytes": (4 + 6 + 6 + 2 + 6) * G * 2 * r + 6 * G * r, "flops": solve}
    # a cycle: E, B in and out, the spectral state in and out, the particles in and out
    return {"bytes": (12 + 12 + 2) * G * 2 * r + 6 * G * r + push, "flops": solve + deposit + gather_push}


def work(case):
    c = dict(case)
    if c["kind"] == "setup":   # the matrices, their inverses and the tables; one SVD-sized factorisation each
        n2 = 3 * c["Nm"] * c["Nr"] ** 2
        return {"bytes": 2.0 * 8 * n2 + 6 * 8 * c["Nm"] * c["Nr"] * c["Nz"], "flops": 20.0 * n2 * c["Nr"]}
    if c["kind"] == "scan":
        each = [_work(m) for m in _members(c)]
        return {k: c["cycles"] * sum(w[k] for w in each) for k in ("bytes", "flops")}
    w = _work(c)
    return {k: v * (1 if c["kind"] == "particles" else c["cycles"]) for k, v in w.items()}


# ---------------------------------------------------------------------------- in 64 bits
C0, EPS0 = 299792458.0, 8.8541878128e-12
MU0, QE, ME = 1.0 / (EPS0 * C0 * C0), 1.602176634e-19, 9.1093837015e-31


def _bessel(n, x):
    """J_n(x) by the trapezoidal rule on its integral over a full period (Bessel's integral),
    which converges faster than any power once the points outnumber x."""
    pts = int(float(x.max())) + 80
    out = torch.zeros_like(x)
    for k in range(pts):
        t = math.pi * (k + 0.5) / pts
        out += torch.cos(n * t - x * math.sin(t))
    return out / pts


class _Exact:
    """The PIC cycle of the method in plain 64-bit torch."""

    def __init__(self, c, dr=CELL, matrices_only=False):
        f8 = {"dtype": torch.float64, "device": "cuda"}
        self.c, self.dz, self.dr = c, CELL, dr
        self.Nz, self.Nr, self.Nm = c["Nz"], c["Nr"], c["Nm"]
        self.L, self.R, self.dt = self.Nz * CELL, self.Nr * dr, c["cdt"] * CELL / W.C_LIGHT
        r = (torch.arange(self.Nr, **f8) + 0.5) * dr
        self.vol = 2 * math.pi * r * dr * self.dz
        self.kperp, self.inv, self.fwd = [], [], []
        for m in range(self.Nm):
            b = (torch.arange(1, self.Nr + 1, **f8) + 0.5 * m - 0.25) * math.pi
            x = b - (4 * m * m - 1) / (8 * b)
            for _ in range(8):
                f = _bessel(m, x)
                x = x - f / (0.5 * (_bessel(m - 1, x) - _bessel(m + 1, x)))
            kp = x / self.R
            self.kperp.append(kp)
            B = [_bessel(p, r[:, None] * kp[None, :]) for p in (m - 1, m, m + 1)]
            self.inv.append(B)
            self.fwd.append([torch.from_numpy(np.linalg.pinv(b.cpu().numpy(), rtol=1e-3)).cuda() for b in B])
        kz = 2 * math.pi * torch.fft.fftfreq(self.Nz, d=self.dz, **f8)
        self.Kz = kz.clone()
        if c["order"]:
            n, a = c["order"] // 2, 1.0
            self.Kz.zero_()
            for j in range(1, n + 1):
                a *= (n - j + 1) / (n + j)
                self.Kz += (2 if j % 2 else -2) * a * torch.sin(kz * (j * self.dz)) / (j * self.dz)
        if matrices_only:
            return
        Kp = torch.stack(self.kperp)[:, :, None]
        self.Kp, Kz = Kp, self.Kz[None, None, :]
        K2 = Kp * Kp + Kz * Kz
        K = torch.sqrt(K2)
        x = C0 * self.dt * K
        s, co = torch.sin(x), torch.cos(x)
        an, ap, pw, fact = torch.zeros_like(x), torch.zeros_like(x), torch.ones_like(x), 1.0
        for k in range(1, 10):   # power series of the two charge coefficients for small x
            fact *= (2 * k) * (2 * k + 1)
            an += (-1) ** k * pw / fact
            ap += (-1) ** k * 2 * k * pw / fact
            pw = pw * x * x
        small, t = x < 0.25, (C0 * self.dt) ** 2
        self.an = torch.where(small, t * an, (s / x - 1) / K2)
        self.ap = torch.where(small, t * ap, (co - s / x) / K2)
        self.C, self.SK, self.omc, self.K2 = co, s / K, 2 * torch.sin(0.5 * x) ** 2 / K2, K2
        self.T = (torch.cos(0.5 * Kp * dr) * torch.cos(0.5 * kz * self.dz)[None, None, :]) ** 2

    # transforms: (+, -, z) carry the orders m + 1, m - 1, m
    def _mat(self, mats, slot, F):
        return torch.stack([torch.view_as_complex((mats[m][slot] @ torch.view_as_real(F[m]).reshape(self.Nr, -1))
                                                  .reshape(self.Nr, self.Nz, 2)) for m in range(self.Nm)])

    def forward(self, F, slot):
        return self._mat(self.fwd, slot, torch.fft.fft(F, dim=-1))

    def forward_vector(self, V):
        return [self.forward(0.5 * (V[0] - 1j * V[1]), 2), self.forward(0.5 * (V[0] + 1j * V[1]), 0), self.forward(V[2], 1)]

    def inverse_vector(self, V):
        p, m, z = [torch.fft.ifft(self._mat(self.inv, k, v), dim=-1) for k, v in zip((2, 0, 1), V)]
        return [p + m, 1j * (p - m), z]

    def curl(self, V):
        Kp, Kz = self.Kp, self.Kz
        return [Kz * V[0] - 0.5j * Kp * V[2], -Kz * V[1] - 0.5j * Kp * V[2], 1j * Kp * (V[0] + V[1])]

    def grad(self, X):
        return [-0.5 * self.Kp * X, 0.5 * self.Kp * X, 1j * self.Kz * X]

    def field_step(self, dep):
        rho = self.T * self.forward(dep[0], 1)
        J = [self.T * v for v in self.forward_vector(dep[1:])]
        div = self.Kp * (J[0] - J[1]) + 1j * self.Kz * J[2]
        J = [a + b for a, b in zip(J, self.grad(((rho - self.rho) / self.dt + div) / self.K2))]
        X = self.grad((self.an * rho + self.ap * self.rho) / EPS0)
        cE, cB, cJ = self.curl(self.Eh), self.curl(self.Bh), self.curl(J)
        E = [self.C * e + C0 * self.SK * b - self.SK / (EPS0 * C0) * j + x for e, b, j, x in zip(self.Eh, cB, J, X)]
        B = [self.C * b - self.SK / C0 * e + MU0 * self.omc * j for b, e, j in zip(self.Bh, cE, cJ)]
        self.Eh, self.Bh, self.rho = E, B, rho
        self.E, self.B = self.inverse_vector(E), self.inverse_vector(B)

    # particles
    @staticmethod
    def polar(x, y):
        r = torch.sqrt(x * x + y * y)
        one = torch.where(r > 0, r, torch.ones_like(r))
        return r, torch.where(r > 0, x / one, torch.ones_like(r)), torch.where(r > 0, y / one, torch.zeros_like(r))

    def nodes(self, z, r):
        """(flat node, weight, is the ghost node) of the four nodes of each particle."""
        u, v = z / self.dz, r / self.dr - 0.5
        fi, fj = torch.floor(u), torch.floor(v)
        i0, j0 = fi.long() % self.Nz, fj.long()
        for i, wz in ((i0, 1 - (u - fi)), ((i0 + 1) % self.Nz, u - fi)):
            for j, wr in ((j0, 1 - (v - fj)), (j0 + 1, v - fj)):
                w = torch.where(j < self.Nr, wz * wr, torch.zeros_like(wz))
                yield torch.where(j < 0, -1 - j, j).clamp(max=self.Nr - 1) * self.Nz + i, w, j < 0

    def deposit(self, x, y, z, values):
        """Per value (weight, radial-or-azimuthal?) the mode grids [Nm, Nr, Nz]."""
        r, c, s = self.polar(x, y)
        e1, out = torch.complex(c, s), []
        nodes = list(self.nodes(z, r))
        for val, rt in values:
            grid, ph = torch.zeros((self.Nm, self.Nr * self.Nz), dtype=torch.complex128, device="cuda"), torch.ones_like(e1)
            for m in range(self.Nm):
                fold = -1.0 if (m + rt) % 2 else 1.0
                for at, w, ghost in nodes:
                    a = val * torch.where(ghost, fold * w, w) * ph
                    torch.view_as_real(grid[m]).index_add_(0, at, torch.view_as_real(a))
                ph = ph * e1
            out.append(grid.reshape(self.Nm, self.Nr, self.Nz) / self.vol[None, :, None])
        return out

    def gather(self, x, y, z):
        r, c, s = self.polar(x, y)
        e1, F = torch.complex(c, -s), []
        nodes = list(self.nodes(z, r))
        for k, G in enumerate(self.E + self.B):
            tot, ph = torch.zeros_like(x), torch.ones_like(e1)
            for m in range(self.Nm):
                fold, flat = (-1.0 if (m + (k % 3 < 2)) % 2 else 1.0), G[m].reshape(-1)
                v = sum(torch.where(g, fold * w, w) * flat[at] for at, w, g in nodes)
                tot = tot + (2.0 if m else 1.0) * (v * ph).real
                ph = ph * e1
            F.append(tot)
        return [F[0] * c - F[1] * s, F[0] * s + F[1] * c, F[2], F[3] * c - F[4] * s, F[3] * s + F[4] * c, F[5]]

    def wrap(self, z):
        z = torch.where(z >= self.L, z - self.L, z)
        return torch.where(z < 0, z + self.L, z)

    def push(self, P, back=None, shift=False):
        """Boris push, two half moves, wall; returns J at the half step and its positions."""
        act, z0 = P["w"] != 0, P["z"]
        k = -QE * self.dt / (2 * ME)
        F = self.gather(P["x"], P["y"], P["z"])
        E, t = [k * f for f in F[:3]], [k * f for f in F[3:]]
        cross = lambda a, b: [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]  # noqa: E731
        gam = lambda u: torch.sqrt(1 + sum(a * a for a in u) / (C0 * C0))  # noqa: E731
        u = [P[n] + e for n, e in zip(("ux", "uy", "uz"), E)]
        g0 = gam(u)
        t = [a / g0 for a in t]
        f = 2 / (1 + sum(a * a for a in t))
        up = [a + b for a, b in zip(u, cross(u, t))]
        u = [a + f * b + e for a, b, e in zip(u, cross(up, t), E)]
        g1 = gam(u)
        h = [0.5 * self.dt * a / g1 for a in u]
        x, y, z = P["x"] + h[0], P["y"] + h[1], self.wrap(P["z"] + h[2])
        _, c, s = self.polar(x, y)
        v, q = [a / g1 for a in u], -QE * P["w"]
        J = self.deposit(x, y, z, [(q * (c * v[0] + s * v[1]), 1), (q * (c * v[1] - s * v[0]), 1), (q * v[2], 0)])
        x, y, z = x + h[0], y + h[1], self.wrap(z + h[2])
        r = torch.sqrt(x * x + y * y)
        out, rs = r >= self.R, torch.where(r >= self.R, r, torch.ones_like(r))
        f, ur = torch.where(out, (2 * self.R - r) / rs, torch.ones_like(r)), (u[0] * x + u[1] * y) / rs
        u[0], u[1] = torch.where(out, u[0] - 2 * ur * x / rs, u[0]), torch.where(out, u[1] - 2 * ur * y / rs, u[1])
        for n, a in zip(("x", "y", "z", "ux", "uy", "uz"), (x * f, y * f, z, *u)):
            P[n] = torch.where(act, a, P[n])
        if back is not None:   # the moving window removes what it leaves behind
            zo = z0 - back
            zo = torch.where(zo < 0, zo + self.L, zo)
            gone = act & (zo + 2 * h[2] - (self.dz if shift else 0.0) < 0)
            for n in ("w", "ux", "uy", "uz"):
                P[n] = torch.where(gone, torch.zeros_like(P[n]), P[n])
        return J

    def rho_of(self, P, sel=slice(None)):
        return self.deposit(P["x"][sel], P["y"][sel], P["z"][sel], [(-QE * P["w"][sel], 0)])[0]

    def start(self, P, n_plasma, gamma):
        """The initial state: ions, the beam's own fields, rho^0."""
        self.ion = -self.rho_of(P, slice(0, n_plasma))
        rho = self.T * self.forward(self.rho_of(P, slice(n_plasma, None)), 1)
        phi = rho / (EPS0 * (self.Kp ** 2 + self.Kz ** 2 / gamma ** 2))
        self.Eh = [0.5 * self.Kp * phi, -0.5 * self.Kp * phi, -1j * self.Kz * phi / gamma ** 2]
        zero = torch.zeros_like(phi)
        self.Bh = self.curl([zero, zero, math.sqrt(1 - 1 / gamma ** 2) * phi / C0])
        self.rho = self.T * self.forward(self.rho_of(P) + self.ion, 1)
        self.E, self.B = self.inverse_vector(self.Eh), self.inverse_vector(self.Bh)

    def window(self, P, n_plasma):
        n = n_plasma // 4
        k = torch.arange(n, dtype=torch.float64, device="cuda")
        park = {"x": (torch.floor(k / self.Nz) % self.Nr + 0.5) * self.dr, "z": (k % self.Nz + 0.5) * self.dz}
        self.tpl = {a: P[a][:n_plasma].clone() for a in ("x", "y", "z", "w")}
        self.col = torch.floor(self.tpl["z"] / self.dz).long().clamp(0, self.Nz - 1)
        for a in bd.SOA:
            P[a] = torch.cat([P[a], park.get(a, torch.zeros_like(k))])

    def cycles(self, P, count):
        shifts = 0
        for i in range(count):
            back, shift = None, False
            if self.c["window"]:
                back, shift = shifts % self.Nz * self.dz, self.c["cdt"] == 1.0 or i % 2 == 1
            J = self.push(P, back, shift)
            col = shifts % self.Nz
            if shift:
                fresh, free = (self.col == col).nonzero()[:, 0], (P["w"] == 0).nonzero()[:, 0]
                k = min(len(fresh), len(free))
                for a in bd.SOA:
                    P[a] = P[a].index_put((free[:k],), self.tpl[a][fresh[:k]] if a in self.tpl else P[a].new_zeros(k))
            self.field_step([self.rho_of(P) + self.ion] + J)
            if shift:
                for real, spec in ((self.E, self.Eh), (self.B, self.Bh)):
                    only = [torch.zeros_like(f) for f in real]
                    for o, f in zip(only, real):
                        o[:, :, col] = f[:, :, col]
                        f[:, :, col] = 0
                    for k, d in enumerate(self.forward_vector(only)):
                        spec[k] = spec[k] - d
                shifts += 1

    def fields(self):
        return {"E": torch.stack(self.E), "B": torch.stack(self.B), "RHO_PREV_H": self.rho}

    def beam(self, P, lo, hi):
        x, y, z, ux, uy, uz, w = [P[k][lo:hi] for k in bd.SOA]
        mean = lambda a: float((w * a).sum() / w.sum())  # noqa: E731
        emit = lambda a, u: math.sqrt(mean((a - mean(a)) ** 2) * mean((u - mean(u)) ** 2)  # noqa: E731
                                      - mean((a - mean(a)) * (u - mean(u))) ** 2) / C0
        gam, sz = torch.sqrt(1 + (ux * ux + uy * uy + uz * uz) / (C0 * C0)), math.sqrt(mean((z - mean(z)) ** 2))
        d, ns = z - (mean(z) - 3 * sz), math.ceil(6 * sz / 0.5e-6)
        ok = (d >= 0) & (d < 6 * sz)
        at = torch.floor(d[ok] / 0.5e-6).long().clamp(max=ns - 1)
        add = lambda v: torch.zeros(ns, dtype=v.dtype, device="cuda").index_add_(0, at, v)  # noqa: E731
        sw, sg = add(w[ok]), add(w[ok] * gam[ok])
        full = sw > 0
        var = add(w[ok] * (gam[ok] - (sg / torch.where(full, sw, torch.ones_like(sw)))[at]) ** 2)
        vals = (float(w.sum()), mean(z), sz, mean(gam), emit(x, ux), emit(y, uy), float(torch.sqrt(var[full] / sw[full]).mean()))
        return {"beam_" + k: np.float64(v) for k, v in zip(DIAG, vals)}


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "setup":
        e = _Exact(c, CELL * (1 + 1e-3 * (seed % 97)), matrices_only=True)
        return {"KPERP": torch.stack(e.kperp), "HANKEL_INV": torch.stack([torch.stack(b) for b in e.inv]),
                "HANKEL_FWD": torch.stack([torch.stack(b) for b in e.fwd]), "KZ_MOD": e.Kz}
    if c["kind"] == "scan" or c["Nz"] * c["Nr"] * c["Nm"] > 5e6:
        return None   # minutes of 64-bit products
    e = _Exact(c)
    P, npl, gamma = _particles(c, seed)
    n = len(P["x"])
    del P["id"]
    e.start(P, npl, gamma)
    if c["window"]:
        e.window(P, npl)
    if c["kind"] == "field":
        q = -QE * P["w"]
        _, co, si = e.polar(P["x"], P["y"])
        g = torch.sqrt(1 + (P["ux"] ** 2 + P["uy"] ** 2 + P["uz"] ** 2) / (C0 * C0))
        v = [P[k] / g for k in ("ux", "uy", "uz")]
        dep = e.deposit(P["x"], P["y"], P["z"], [(q, 0), (q * (co * v[0] + si * v[1]), 1), (q * (co * v[1] - si * v[0]), 1),
                                                 (q * v[2], 0)])
        dep[0] = dep[0] + e.ion
        for _ in range(c["cycles"]):
            e.field_step(dep)
        return dict(e.fields(), EH=torch.stack(e.Eh), BH=torch.stack(e.Bh))
    if c["kind"] == "particles":
        J = e.push(P)
        return dict(P, KEYS=None, PERM=None, DEP=torch.stack([e.rho_of(P) + e.ion] + J))
    e.cycles(P, c["cycles"])
    out = dict(e.fields(), **P)
    if c["diag"]:
        out.update(e.beam(P, npl, n))
    return out
