"""The FP64 push's reciprocal square root and its quotient 2 / (1 + t^2), read off single particles: both are formed
from the float32 unit's approximations and one step, and stay within about an ulp over the whole range of their
arguments (mantissas and even and odd exponents)."""
import numpy as np
import pytest

from oracle import psatd_rz as O
from paper_1611_05712_gb300 import binding as bd

pytestmark = pytest.mark.gpu

LD = np.longdouble


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_05712_gb300.build import build
    build()


def _set(n, **k):
    P = {a: np.zeros(n) for a in bd.SOA}
    P.update(w=np.ones(n), id=np.arange(n, dtype=np.int32), **k)
    return P


def test_inverse_gamma():
    """A particle on the axis with u_x = 1 m/s and no fields moves by dt / gamma, exactly rounded up to
    1/gamma's own error when dt is a power of two: u_z sets gamma."""
    n, D, dt = 60000, 1.0, 2.0 ** -40
    rng = np.random.default_rng(1)
    uz = np.concatenate([10.0 ** rng.uniform(-3, 150, n // 2), 10.0 ** rng.uniform(7, 10, n // 2)])
    s = bd.Sim(bd.make_config(24, 8, 1, D, D, dt, 0, True, bd.PIC_FP64, n))
    s.write_particles(_set(n, ux=np.ones(n), uz=uz, z=np.full(n, 12.3 * D)))
    s.gather_push(False)
    got = s.read_particles()["x"]
    s.close()
    ref = 1 / np.sqrt(1 + (1 + uz.astype(LD) ** 2) / LD(O.C_LIGHT) ** 2)
    # the argument within 2.5 roundings (2^-53 each) of its value, half of that in the root, and an ulp (2^-52)
    assert (np.abs(got.astype(LD) / dt / ref - 1) < 2.0 ** -51).all()


@pytest.mark.parametrize("D", [1e-12, 1e-6, 1.0, 1e3, 1e9])
def test_azimuth(D):
    """J_r / J_z of a particle moving along x and z is cos(theta) v_x / v_z = (x / r) v_x / v_z."""
    Nz, Nr = 3 * 512, 64
    rng = np.random.default_rng(2)
    i = np.arange(Nz // 3)
    r, th = rng.uniform(0.6, Nr - 1.6, i.size) * D, rng.uniform(0, 2 * np.pi, i.size)
    x, y = r * np.cos(th), r * np.sin(th)
    P = _set(i.size, x=x, y=y, z=(3 * i + 0.5) * D, ux=np.full(i.size, 2.0 ** 20), uz=np.full(i.size, 2.0 ** 20))
    s = bd.Sim(bd.make_config(Nz, Nr, 1, D, D, 1e-12, 0, True, bd.PIC_FP64, i.size, q=1.0))
    s.write_particles(P)
    s.deposit(bd.PIC_DEP_J)
    J = s.get("DEP")[1:, 0].real
    s.close()
    j = np.floor(np.hypot(x, y) / D - 0.5).astype(int)
    ratio = J[0, j, 3 * i] / J[2, j, 3 * i]
    ref = x.astype(LD) / np.sqrt(x.astype(LD) ** 2 + y.astype(LD) ** 2)
    # x^2 + y^2 within a rounding, half of it in the root, an ulp, and a rounding each of x / r, the two
    # currents and their quotient here
    assert (np.abs(ratio / ref - 1) < 8 * 2.0 ** -53).all()


def test_rotation_quotient():
    """A particle with u_x = 1 m/s in B_z alone leaves with u_y = -2 t / (1 + t^2), t = q dt B_z / (2 m)."""
    Nz, D, dt = 3 * 700, 1.0, 2.0 ** -20   # not a power of two: float64 gather
    i = np.arange(Nz // 3)
    rng = np.random.default_rng(3)
    t = 2.0 ** rng.uniform(-30, 60, i.size) * rng.choice([-1, 1], i.size)
    t[::5] = 2.0 ** rng.uniform(60, 505, t[::5].size)
    s = bd.Sim(bd.make_config(Nz, 8, 1, D, D, dt, 0, True, bd.PIC_FP64, i.size, q=1.0, mass=1.0))
    B = s.zeros("B")
    b = t * 2.0 ** 21   # k = q dt / (2 m) = 2^-21
    for a in range(2):  # the particle's two z nodes, all radii
        B[2, 0, :, 3 * i + a] = b[:, None]
    s.set("B", B)
    s.write_particles(_set(i.size, x=np.full(i.size, 2.5 * D), z=(3 * i + 0.5) * D, ux=np.ones(i.size)))
    s.gather_push(False)
    uy = s.read_particles()["uy"]
    s.close()
    ref = -2 * t.astype(LD) / (1 + t.astype(LD) ** 2)
    # the gathered field within 3 roundings (2^-53), 1 + t^2 one more, the quotient an ulp (2^-52), its product
    # with t another rounding
    assert (np.abs(uy / ref - 1) < 2.0 ** -50).all()
