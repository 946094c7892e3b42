"""The FP64 form's linear weights at the edges of their cells: particles on, and a few ulps to both
sides of, the nodes in z and r, on the axis, at both ends of the box, at the wall and outside it,
with spacings that are and are not powers of two, deposited and pushed against the oracle."""
import numpy as np
import pytest

from oracle import psatd_rz as O
from paper_1611_05712_gb300 import binding as bd
from gpu_helpers import per_slice_err, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_05712_gb300.build import build
    build()


@pytest.mark.parametrize("Nz,Nr,dz,dr", [(8, 4, 2.0 ** -24, 2.0 ** -25), (64, 16, 0.05e-6, 0.05e-6),
                                         (1800, 100, 0.05e-6, 0.03e-6), (4096, 64, 1 / 3, 0.7)])
def test_weights_at_cell_edges(Nz, Nr, dz, dr):
    Nm, n = 3, 4000
    g = O.Grid(Nz, Nr, Nm, dz, dr, 0.01 * min(dz, dr) / O.C_LIGHT)
    rng = np.random.default_rng(Nz)
    z, r = rng.integers(0, Nz, n) * dz, (rng.integers(0, Nr, n) + 0.5 * rng.integers(0, 2, n)) * dr
    for _ in range(3):   # steps of one ulp up or down, or none
        z = np.nextafter(z, z + rng.integers(-1, 2, n) * dz)
        r = np.nextafter(r, r + rng.integers(-1, 2, n) * dr)
    far = rng.random(n) < 0.4
    z[far], r[far] = g.L * rng.random(far.sum()), g.R * rng.random(far.sum())
    r[:50] = 0.0
    r[50:60] = 1e-200
    z[60:70], z[70:80] = 0.0, 1e-300
    z = np.clip(z, 0.0, np.nextafter(g.L, 0.0))
    r = np.abs(r)
    th = np.where(rng.random(n) < 0.5, 0.5 * np.pi * rng.integers(0, 4, n), rng.uniform(0, 2 * np.pi, n))
    P = {"x": r * np.cos(th), "y": r * np.sin(th), "z": z, "ux": np.zeros(n), "uy": np.zeros(n), "uz": np.zeros(n),
         "w": rng.uniform(0.5, 2.0, n), "id": np.arange(n, dtype=np.int32)}
    s = bd.Sim(bd.make_config(Nz, Nr, Nm, dz, dr, g.dt, 0, True, bd.PIC_FP64, n))
    s.write_particles(P)
    s.deposit(bd.PIC_DEP_RHO)
    # z / dz and r / dr below 2^12 and 2^7: their float64 roundings move a weight by up to Nz 2^-53
    tol = (16 + 2 * Nz) * 2.0 ** -53
    rho = O.deposit_rho(g, P["x"], P["y"], P["z"], P["w"], -O.Q_E)
    assert per_slice_err(s.get("DEP")[0:1], rho[None]) < tol
    # the gather at rest: the momentum is the field at the particle to first order; the fields' double
    # words and their sums add a few 2^-48
    keep = np.hypot(P["x"], P["y"]) < 0.98 * g.R   # no reflection
    P = {k: v[keep] for k, v in P.items()}
    P["id"] = np.arange(keep.sum(), dtype=np.int32)
    s.write_particles(P)
    crand = lambda sh, a: a * (rng.normal(size=sh) + 1j * rng.normal(size=sh))  # noqa: E731
    a = 1e-4 * O.M_E * O.C_LIGHT / (O.Q_E * g.dt)
    E, B = crand((3, Nm, Nr, Nz), a), crand((3, Nm, Nr, Nz), a / O.C_LIGHT)
    s.set("E", E)
    s.set("B", B)
    s.gather_push(fuse_current=False)
    zero = np.zeros((Nm, Nr, Nz), complex)
    st = O.State(g, 0, False, -O.Q_E, O.M_E, None, None, None, tuple(E), tuple(B), None, None, zero, zero,
                 {k: v.copy() for k, v in P.items()})
    O.gather_push(st)
    got = s.read_particles()
    s.close()
    for k in ("ux", "uy", "uz"):
        assert rel_err(got[k], st.p[k]) < tol + 2.0 ** -44, k


def test_radius_that_overflows():
    """x^2 + y^2 beyond the largest float64: the weights are NaN, at the axis row, and so is the push."""
    Nz, Nr, dz = 64, 16, 0.05e-6
    P = {k: np.zeros(3) for k in ("ux", "uy", "uz")}
    P.update(x=np.array([dz, 1e200, 3 * dz]), y=np.zeros(3), z=np.array([2.3, 20.4, 40.5]) * dz, w=np.ones(3),
             id=np.arange(3, dtype=np.int32))
    s = bd.Sim(bd.make_config(Nz, Nr, 2, dz, dz, dz / O.C_LIGHT, 0, True, bd.PIC_FP64, 3))
    s.write_particles(P)
    s.deposit(bd.PIC_DEP_RHO)
    want = np.zeros((Nr, Nz), bool)
    want[0, 20:22] = True
    assert np.array_equal(np.isnan(s.get("DEP")[0]).any(axis=0), want)
    s.gather_push(fuse_current=False)
    got = s.read_particles()
    s.close()
    assert np.array_equal(np.isnan(got["ux"]), P["x"] == 1e200)
