"""The FP64 deposits' products (q w, shape weights, 1/V, velocity, mode phase) factor by factor:
particles far enough apart that every node holds one contribution, with weights over 500 binary
orders of magnitude, azimuths on and a hair off the axes, velocities from rest to c, next to the
axis, the wall and both ends of the box, 1 to 4 modes, against the oracle's plain float64 products;
and a weight that is not finite."""
import numpy as np
import pytest

from oracle import psatd_rz as O
from paper_1611_05712_gb300 import binding as bd

pytestmark = pytest.mark.gpu

DZ = 0.05e-6
Nz, Nr = 64, 32


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_05712_gb300.build import build
    build()


def _particles(rng):
    iz, ir = (a.ravel() for a in np.meshgrid(np.arange(0, Nz, 4), np.arange(0, Nr, 4), indexing="ij"))
    n = iz.size
    z, r = (iz + rng.uniform(0.1, 0.9, n)) * DZ, (ir + rng.uniform(0.1, 0.4, n)) * DZ
    th = rng.uniform(0, 2 * np.pi, n)
    axis = rng.random(n) < 0.4
    th[axis] = 0.5 * np.pi * rng.integers(0, 4, axis.sum()) + rng.choice([0.0, 1e-12, -1e-7], axis.sum())
    u = rng.normal(size=(3, n)) * 10.0 ** rng.uniform(-3, 12, n)
    u[:, rng.random(n) < 0.2] = 0.0
    return {"x": r * np.cos(th), "y": r * np.sin(th), "z": z, "ux": u[0], "uy": u[1], "uz": u[2],
            "w": 10.0 ** rng.uniform(-80, 80, n), "id": np.arange(n, dtype=np.int32)}


@pytest.mark.parametrize("Nm", [1, 2, 3, 4])
def test_products_of_single_contributions(Nm):
    rng = np.random.default_rng(Nm)
    P = _particles(rng)
    g = O.Grid(Nz, Nr, Nm, DZ, DZ, DZ / O.C_LIGHT)
    s = bd.Sim(bd.make_config(Nz, Nr, Nm, DZ, DZ, g.dt, 0, True, bd.PIC_FP64, len(P["x"])))
    s.write_particles(P)
    s.deposit()
    got = s.get("DEP")
    s.close()
    ig = O.inv_gamma(P["ux"], P["uy"], P["uz"])
    v = [P[k] * ig for k in ("ux", "uy", "uz")]
    J = O.deposit_current(g, P["x"], P["y"], P["z"], *v, P["w"], -O.Q_E)
    ref = np.stack([O.deposit_rho(g, P["x"], P["y"], P["z"], P["w"], -O.Q_E), *J])
    # a contribution's factors differ by a few ulps between the two (r, the azimuth and r/dr come
    # from other roundings; r/dr - floor loses up to 5 bits at r = 32 dr and the weights another
    # 3.3 bits at 0.1); each node's scale is its own charge times the speed that reaches it
    speed = np.concatenate([[1.0], [1.0, 1.0, 1.0]])
    rho0 = np.abs(ref[0, 0])
    vmax = np.zeros((Nr, Nz))
    i0, j0 = np.floor(P["z"] / DZ).astype(int), np.floor(np.hypot(P["x"], P["y"]) / DZ - 0.5).astype(int)
    sp = np.sqrt(v[0] ** 2 + v[1] ** 2 + v[2] ** 2)
    for a in (0, 1):
        for b in (0, 1):
            jj = np.where(j0 + b < 0, 0, j0 + b)
            ok = jj < Nr
            np.maximum.at(vmax, (jj[ok], (i0[ok] + a) % Nz), sp[ok])
    axis_row = np.zeros((Nr, 1), bool)
    axis_row[0] = True   # node 0 of the axis cell sums a node and its ghost: no single scale there
    for c in range(4):
        scale = rho0 * (speed[c] if c == 0 else vmax)
        for m in range(Nm):
            bad = (np.abs(got[c, m] - ref[c, m]) > 1e-12 * scale) & ~axis_row
            assert not bad.any(), (c, m)
            assert (got[c, m][rho0 == 0] == 0).all()
            top = np.abs(ref[c, m][0]).max()
            assert np.abs(got[c, m][0] - ref[c, m][0]).max() <= 1e-11 * top


def test_weight_that_is_not_finite():
    rng = np.random.default_rng(7)
    P = _particles(rng)
    P["w"][:] = 1.0
    P["w"][40] = np.nan
    s = bd.Sim(bd.make_config(Nz, Nr, 2, DZ, DZ, DZ / O.C_LIGHT, 0, True, bd.PIC_FP64, len(P["x"])))
    s.write_particles(P)
    s.deposit()
    got = s.get("DEP")
    s.close()
    # its nodes: the ghost node of the axis cell is node 0 itself
    i0, j0 = int(P["z"][40] / DZ), int(np.floor(np.hypot(P["x"][40], P["y"][40]) / DZ - 0.5))
    want = np.zeros((Nr, Nz), bool)
    want[max(j0, 0):j0 + 2, i0:i0 + 2] = True
    assert np.array_equal(np.isnan(got).any(axis=(0, 1)), want)
