"""Cell keys of the FP64 form at the cell boundaries (particles per cell; stable counting sort):
coordinates a few ulps to both sides of z = i dz and r = j dr, at the ends of the box, on the
axis and with tiny and signed-zero coordinates, bit-exact against the rounded quotients."""
import numpy as np
import pytest

from oracle import psatd_rz as O
from paper_1611_05712_gb300 import binding as bd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_05712_gb300.build import build
    build()


@pytest.mark.parametrize("Nz,Nr,dz,dr", [(8, 4, 0.05e-6, 0.05e-6), (1800, 400, 0.05e-6, 0.03e-6), (4096, 1024, 1 / 3, 0.7)])
def test_keys_at_cell_boundaries(Nz, Nr, dz, dr):
    g = O.Grid(Nz, Nr, 1, dz, dr, 0.5 * dz / O.C_LIGHT)
    rng = np.random.default_rng(Nz)
    n = 20000
    i, j = rng.integers(0, Nz, n), rng.integers(0, Nr, n)
    z, r = i * dz, j * dr
    for _ in range(3):   # steps of one ulp up or down, or none
        z = np.nextafter(z, z + rng.integers(-1, 2, n) * dz)
        r = np.nextafter(r, r + rng.integers(-1, 2, n) * dr)
    far = rng.random(n) < 0.3
    z[far], r[far] = (i[far] + rng.random(far.sum())) * dz, (j[far] + rng.random(far.sum())) * dr
    z = np.clip(z, 0.0, np.nextafter(g.L, 0.0))
    th = np.where(rng.random(n) < 0.5, 0.5 * np.pi * rng.integers(0, 4, n), rng.uniform(0, 2 * np.pi, n))
    x, y = r * np.cos(th), r * np.sin(th)
    x[:4], y[:4], z[:4] = (0.0, -0.0, 1e-300, 1e-170), (0.0, 0.0, -1e-310, 1e-170), (0.0, -0.0, 1e-300, 5e-324)
    P = {"x": x, "y": y, "z": z, "ux": np.zeros(n), "uy": np.zeros(n), "uz": np.zeros(n), "w": np.ones(n),
         "id": np.arange(n, dtype=np.int32)}
    s = bd.Sim(bd.make_config(Nz, Nr, 1, dz, dr, g.dt, 0, True, bd.PIC_FP64, n))
    s.write_particles(P)
    s.sort()
    keys = O.cell_keys(g, x, y, z)
    assert np.array_equal(s.get("KEYS"), keys)
    assert np.array_equal(s.get("PERM"), O.sort_permutation(keys))
    s.close()
