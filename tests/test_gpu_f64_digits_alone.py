"""The eight-digit FP64 DHT by itself: panels that are zero but for their first column in z have a z-DFT that both
row kernels form exactly (every coefficient is that column), so the product of the Hankel matrix is all that is
compared with extended precision."""
import numpy as np
import pytest

from paper_1611_05712_gb300 import binding as bd

pytestmark = pytest.mark.gpu

DZ = 0.05e-6
SLOT = (1, 2, 0, 1)   # Hankel order slot of rho, J_+, J_-, J_z


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_05712_gb300.build import build
    build()


@pytest.mark.parametrize("Nr,Nm", [(257, 2), (288, 1), (320, 2), (511, 1), (513, 1), (700, 1), (1024, 1)])
@pytest.mark.parametrize("kind", ["random", "beam", "spread"])
def test_product_alone(Nr, Nm, kind):
    Nz = 16
    rng = np.random.default_rng(Nr)
    dep = np.zeros((4, Nm, Nr, Nz), complex)
    # both parts of a value and both currents within a factor of two: their sums are exact in the rows
    a = rng.uniform(1, 2, size=(4, Nm, Nr)) * rng.choice([-1, 1], size=(4, Nm, Nr)) + 1j * rng.uniform(1, 2, size=(4, Nm, Nr))
    j = np.arange(Nr)
    if kind == "beam":
        a = a * 2.0 ** -np.round((20.0 * j / Nr) ** 2)
    if kind == "spread":
        a = a * 2.0 ** np.round(rng.uniform(-20, 0, size=Nr))
    a = np.round(a * 2.0 ** 40) * 2.0 ** -40   # 41 significant bits: halves and sums stay exact
    dep[..., 0] = a
    s = bd.Sim(bd.make_config(Nz, Nr, Nm, DZ, DZ, DZ / 299792458.0, 32, True, bd.PIC_FP64, 0))
    s.set("DEP", dep)
    s.forward_transform()
    got = s.get("SRC_H")
    s.set_dht_path(bd.PIC_DHT_F64_GEMM)
    s.forward_transform()
    gemm = s.get("SRC_H")
    mats = s.get("HANKEL_FWD")
    s.close()
    d = a.astype(np.clongdouble)
    X = np.stack([d[0], (d[1] - 1j * d[2]) / 2, (d[1] + 1j * d[2]) / 2, d[3]])
    for c in range(4):
        for m in range(Nm):
            M = mats[m, SLOT[c]].astype(np.longdouble)
            ref = (M @ X[c, m])[:, None] * np.ones(Nz)
            e8, eg = (np.abs(v[c, m] - ref).astype(float) for v in (got, gemm))
            # one rounding of each part, and the digits' worst case: products left out and operands' rounding
            # below 2^-59 of row maximum x column maximum a term
            top = np.abs(M).astype(float).max(1)[:, None] * np.maximum(np.abs(X[c, m].real), np.abs(X[c, m].imag)).astype(float).max()
            assert (e8 <= 2.0 ** -53 * np.abs(ref).astype(float) + 2 ** 0.5 * Nr * 2.0 ** -59 * top).all(), (c, m)
            assert np.linalg.norm(e8) <= np.linalg.norm(eg), (c, m)
