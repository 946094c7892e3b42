"""FP64 deposits of particles with an infinity, a NaN or a subnormal number among their factors
(weight, charge, velocity, mode phase), which the integer products do not hold: the values of plain
float64 products, for particles far enough apart that every node holds one particle's contributions,
at rest and moving, on the axis cell, on a row of z nodes and on the last radial nodes."""
import math

import numpy as np
import pytest

from oracle import psatd_rz as O
from paper_1611_05712_gb300 import binding as bd

pytestmark = pytest.mark.gpu

D = 2.0 ** -24   # metres: z on a node is exact
Nz, Nr = 48, 16


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_05712_gb300.build import build
    build()


def _particles(weights, momenta):
    """One particle per weight and momentum, four rows apart in z, at changing radii and azimuths."""
    rows = [(w, u) for w in weights for u in momenta]
    n = len(rows)
    assert 4 * n <= Nz
    i = np.arange(n)
    r = (np.array([0.25, 5.75, 14.75, 15.75])[i % 4]) * D
    th = np.array([0.0, 0.5 * np.pi, 1.1, -2.3])[(i + i // 4) % 4]
    x, y = r * np.cos(th), r * np.sin(th)
    x[th == 0.5 * np.pi] = 0.0
    z = (4 * i + np.where(i % 3 == 2, 0.0, 0.375)) * D
    u = np.array([q for _, q in rows], dtype=float).T
    return {"x": x, "y": y, "z": z, "ux": u[0], "uy": u[1], "uz": u[2], "w": np.array([w for w, _ in rows]),
            "id": np.arange(n, dtype=np.int32)}


def _products(P, Nm, q):
    """Plain float64 products and sums: [rho, J_r, J_theta, J_z][mode][r][z], and the same of magnitudes."""
    out = np.zeros((4, Nm, Nr, Nz, 2))
    mag = np.zeros((4, Nm, Nr, Nz))
    g = O.Grid(Nz, Nr, Nm, D, D, D / O.C_LIGHT)
    inv_v = 1.0 / g.cell_volume()
    ig = O.inv_gamma(P["ux"], P["uy"], P["uz"])
    for k in range(len(P["x"])):
        x, y, r = P["x"][k], P["y"][k], np.hypot(P["x"][k], P["y"][k])
        c, s = x / r, y / r
        vx, vy, vz = (P[a][k] * ig[k] for a in ("ux", "uy", "uz"))
        u, v = P["z"][k] / D, r / D - 0.5
        i0, j0 = int(np.floor(u)), int(np.floor(v))
        vel = (1.0, c * vx + s * vy, c * vy - s * vx, vz)
        for iz, wz in ((i0, 1 - (u - i0)), (i0 + 1, u - i0)):
            for j, wr in ((j0, 1 - (v - j0)), (j0 + 1, v - j0)):
                if j >= Nr:
                    continue
                gq = wz * (wr * (inv_v[max(j, 0)] * (q * P["w"][k])))
                if gq == 0.0:
                    continue
                for a in range(4):
                    ph = (1.0, 0.0)
                    for m in range(Nm):
                        fold = (-1.0) ** m if a in (0, 3) else (-1.0) ** (m + 1)
                        f = gq * vel[a] * (fold if j < 0 else 1.0)
                        at = (a, m, max(j, 0), iz % Nz)
                        out[at][0] += f * ph[0]
                        if m:
                            out[at][1] += f * ph[1]
                        mag[at] += abs(gq) * (math.hypot(vx, vy, vz) if a else 1.0)
                        ph = (c, s) if m == 0 else (ph[0] * c - ph[1] * s, ph[0] * s + ph[1] * c)
    return out, mag


REST, SLOW, FAST = (0.0, 0.0, 0.0), (0.0, 0.0, 3e-312), (1e8, -2e8, 5e8)


@pytest.mark.parametrize("weights,momenta,q", [
    ((np.nan, 1.0), (REST, FAST), 1.0),
    ((np.inf, -np.inf, 2.5e-310, 1e30), (REST, SLOW, FAST), -1.0),
    ((5e-324, 1e60, 3.0), (SLOW, FAST, (0.0, 2e-308, 0.0), (1e-309, 0.0, 1e5)), 1.0),
    ((1e40, np.nan), (REST, FAST), 1e-310),
    ((1e-3, 1.0), (REST, FAST), np.inf),
])
@pytest.mark.parametrize("Nm", [1, 2, 4])
def test_factors_out_of_range(weights, momenta, q, Nm):
    P = _particles(weights, momenta)
    with np.errstate(all="ignore"):
        ref, mag = _products(P, Nm, q)
    for what in (bd.PIC_DEP_RHO, bd.PIC_DEP_J, bd.PIC_DEP_RHO | bd.PIC_DEP_J):
        s = bd.Sim(bd.make_config(Nz, Nr, Nm, D, D, D / O.C_LIGHT, 0, True, bd.PIC_FP64, len(P["x"]), q=q))
        s.write_particles(P)
        s.deposit(what)
        dep = s.get("DEP")
        s.close()
        got = np.stack([dep.real, dep.imag], axis=-1)
        a = slice(0 if what & bd.PIC_DEP_RHO else 1, 4 if what & bd.PIC_DEP_J else 1)
        g, e, m = got[a], ref[a], mag[a]
        assert np.array_equal(np.isnan(g), np.isnan(e))
        inf = np.isinf(e)
        assert np.array_equal(g[inf], e[inf])
        ok = np.isfinite(e)
        # a few ulps of r, the azimuth, r/dr (times 32 and 4 where the weight is 1/4) and the factors;
        # a result below the normal range is off by one or two of its units
        tol = np.broadcast_to((1e-12 * np.where(np.isfinite(m), m, 0.0))[..., None], e.shape) + 1e-323
        assert (np.abs(g[ok] - e[ok]) <= tol[ok]).all()


@pytest.mark.parametrize("top", [2.0 ** 1022, 1.7e308, 2.0 ** 1021])
def test_largest_results(top):
    """Charges a node holds up to the largest float64: finite where the product is."""
    # z on a row of nodes and r halfway between two radial nodes: two contributions of half the charge
    r = 6.0 * D
    inv_v = 1.0 / O.Grid(Nz, Nr, 1, D, D, D / O.C_LIGHT).cell_volume()
    w = top / max(0.5 * inv_v[5:7])
    P = {"x": np.array([r]), "y": np.zeros(1), "z": np.array([8 * D]), "ux": np.zeros(1), "uy": np.zeros(1),
         "uz": np.zeros(1), "w": np.array([w]), "id": np.zeros(1, np.int32)}
    s = bd.Sim(bd.make_config(Nz, Nr, 1, D, D, D / O.C_LIGHT, 0, True, bd.PIC_FP64, 1, q=1.0))
    s.write_particles(P)
    s.deposit(bd.PIC_DEP_RHO)
    rho = s.get("DEP")[0, 0].real
    s.close()
    # r, r/dr and the products: a few ulps, as above
    assert np.isfinite(rho).all() and (np.abs(rho[5:7, 8] / (0.5 * w * inv_v[5:7]) - 1) < 1e-13).all()
