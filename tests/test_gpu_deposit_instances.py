"""FP64 deposits and pushes of sets on both sides of the sizes where the kernels' register budgets change (sets that
one, or two, waves of CTAs hold): every particle counted once, in each combination of rho and J."""
import numpy as np
import pytest

from oracle import psatd_rz as O
from paper_1611_05712_gb300 import binding as bd
from gpu_helpers import per_slice_err

pytestmark = pytest.mark.gpu

D = 0.05e-6
Nz, Nr = 32, 16
WAVE = 152 * 256   # particles of one CTA on every SM


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_05712_gb300.build import build
    build()


def _particles(n):
    rng = np.random.default_rng(n)
    r, th = (Nr - 1.5) * D * np.sqrt(rng.uniform(0.01, 1, n)), rng.uniform(0, 2 * np.pi, n)
    u = rng.normal(size=(3, n)) * 0.5 * O.C_LIGHT
    return {"x": r * np.cos(th), "y": r * np.sin(th), "z": rng.uniform(0, Nz * D, n), "ux": u[0], "uy": u[1], "uz": u[2],
            "w": rng.uniform(1, 2, n), "id": np.arange(n, dtype=np.int32)}


@pytest.mark.parametrize("n", [2 * WAVE, 2 * WAVE + 1, 3 * WAVE, 3 * WAVE + 1, 122572, 122573, 140083, 140084, 4 * WAVE,
                               4 * WAVE + 1, 6 * WAVE, 6 * WAVE + 1])
@pytest.mark.parametrize("Nm", [2, 3, 4])
def test_sets_around_the_waves(n, Nm):
    P = _particles(n)
    g = O.Grid(Nz, Nr, Nm, D, D, 0.5 * D / O.C_LIGHT)
    ig = O.inv_gamma(P["ux"], P["uy"], P["uz"])
    J = O.deposit_current(g, P["x"], P["y"], P["z"], *(P[k] * ig for k in ("ux", "uy", "uz")), P["w"], -O.Q_E)
    ref = np.stack([O.deposit_rho(g, P["x"], P["y"], P["z"], P["w"], -O.Q_E), *J])
    s = bd.Sim(bd.make_config(Nz, Nr, Nm, D, D, g.dt, 0, True, bd.PIC_FP64, n))
    s.write_particles(P)
    # sums of n / 512 contributions of either sign, each a few ulps off, in any order
    for what, part in ((bd.PIC_DEP_RHO, slice(0, 1)), (bd.PIC_DEP_J, slice(1, 4)), (3, slice(0, 4))):
        s.deposit(what)
        assert per_slice_err(s.get("DEP")[part], ref[part]) < 1e-12
    # a push without fields: J at the half step
    s.gather_push(True)
    h = 0.5 * g.dt
    x, y, z = (P[a] + h * P["u" + a] * ig for a in "xyz")
    keep = np.hypot(P["x"] + 2 * h * P["ux"] * ig, P["y"] + 2 * h * P["uy"] * ig) < Nr * D   # momenta not reflected
    got = s.read_particles()
    assert np.array_equal(got["ux"][keep], P["ux"][keep])
    J = O.deposit_current(g, x, y, np.mod(z, Nz * D), *(P[k] * ig for k in ("ux", "uy", "uz")), P["w"], -O.Q_E)
    assert per_slice_err(s.get("DEP")[1:], np.stack(J)) < 1e-12
    s.close()
