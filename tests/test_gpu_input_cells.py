"""Particle input of the mixed forms: float64 positions into cells and float fractions, on the cell
boundaries and a few ulps to both sides, negative, tiny, zero and outside the box in z, with spacings
that are and are not powers of two, read back against the positions written."""
import numpy as np
import pytest

from paper_1611_05712_gb300 import binding as bd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_05712_gb300.build import build
    build()


@pytest.mark.parametrize("Nz,Nr,dz,dr", [(16, 8, 2.0 ** -24, 2.0 ** -25), (3125, 176, 0.05e-6, 0.03e-6), (4096, 1000, 1 / 3, 0.7)])
def test_positions_survive(Nz, Nr, dz, dr):
    n = 20000
    rng = np.random.default_rng(Nz)
    P = {k: rng.normal(0, 3e8, n) for k in ("ux", "uy", "uz")}
    P.update(w=rng.uniform(0.5, 2.0, n), id=np.arange(n, dtype=np.int32))
    for k, N, d in (("x", Nr, dr), ("y", Nr, dr), ("z", Nz, dz)):
        v = rng.integers(-N if k != "z" else 0, N, n) * d
        for _ in range(3):   # steps of one ulp up or down, or none
            v = np.nextafter(v, v + rng.integers(-1, 2, n) * d)
        far = rng.random(n) < 0.4
        v[far] = rng.uniform(-N if k != "z" else 0, N, far.sum()) * d
        v[:4] = 0.0, -0.0, 1e-300, 5e-324
        v[4:6] = 1e-12 * d, 0.5 * d
        P[k] = v
    P["x"][6:8], P["y"][6:8] = -1e-300, -1e-12 * dr
    P["z"][10:20] = rng.uniform(-2, 3, 10) * Nz * dz
    s = bd.Sim(bd.make_config(Nz, Nr, 1, dz, dr, 0.5 * min(dz, dr) / 299792458.0, 0, True, bd.PIC_MIXED_TF32X3, n))
    s.write_particles(P)
    got = s.read_particles()
    s.close()
    # a fraction's float rounding (2^-25 of a cell) and the float64 roundings of the way back
    for k, N, d in (("x", Nr, dr), ("y", Nr, dr)):
        assert np.abs(got[k] - P[k]).max() <= (2.0 ** -25 + 2 * N * 2.0 ** -52) * d, k
    L = Nz * dz
    dist = np.abs(got["z"] - P["z"])
    dist = np.minimum(dist % L, L - dist % L)   # the box is periodic
    assert dist.max() <= (2.0 ** -25 + 16 * Nz * 2.0 ** -52) * dz
    assert (got["z"] >= 0).all() and (got["z"] < L * (1 + 2.0 ** -52)).all()
