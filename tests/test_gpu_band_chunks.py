"""Mixed-form deposits (particles' linear weights, one shared band per chunk of particles) at the
particle numbers where the split into chunks changes: one chunk, the shortest chunks, full waves of
them and one more particle, and past the last balanced wave."""
import numpy as np
import pytest

from oracle import psatd_rz as O
from paper_1611_05712_gb300 import binding as bd
from gpu_helpers import per_slice_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_05712_gb300.build import build
    build()


@pytest.mark.parametrize("n", [1, 127, 129, 304 * 128, 304 * 128 + 1, 304 * 160 + 1, 304 * 1024, 304 * 1024 + 1,
                               3 * 304 * 1024 + 1])
def test_chunks(n):
    Nz, Nr, Nm, dz = 96, 24, 2, 0.05e-6
    g = O.Grid(Nz, Nr, Nm, dz, dz, dz / O.C_LIGHT)
    rng = np.random.default_rng(n)
    r = g.R * 0.98 * np.sqrt(rng.uniform(0, 1, n))
    th = rng.uniform(0, 2 * np.pi, n)
    P = dict(x=r * np.cos(th), y=r * np.sin(th), z=rng.uniform(0, g.L, n), ux=rng.normal(0, 3e7, n),
             uy=rng.normal(0, 3e7, n), uz=rng.normal(1e8, 3e8, n), w=rng.uniform(0.5, 2.0, n) * 1e4,
             id=np.arange(n, dtype=np.int32))
    s = bd.Sim(bd.make_config(Nz, Nr, Nm, dz, dz, g.dt, 0, True, bd.PIC_MIXED_TF32X3, n))
    s.write_particles(P)
    s.sort()
    P = s.read_particles()
    s.deposit(bd.PIC_DEP_RHO | bd.PIC_DEP_J)
    dep = s.get("DEP")
    # float weights and phases, a few 2^-24 each, in the sums of every slice
    ig = O.inv_gamma(P["ux"], P["uy"], P["uz"])
    J = O.deposit_current(g, P["x"], P["y"], P["z"], P["ux"] * ig, P["uy"] * ig, P["uz"] * ig, P["w"], -O.Q_E)
    assert per_slice_err(dep[0:1], O.deposit_rho(g, P["x"], P["y"], P["z"], P["w"], -O.Q_E)[None]) < 1e-5
    assert per_slice_err(dep[1:], np.stack(J)) < 1e-5
    # the push deposits its current from the same chunks: with no fields, J half a step on
    s.gather_push(fuse_current=True)
    push = s.get("DEP")
    h = 0.5 * g.dt
    x, y, z = P["x"] + h * P["ux"] * ig, P["y"] + h * P["uy"] * ig, (P["z"] + h * P["uz"] * ig) % g.L
    J = O.deposit_current(g, x, y, z, P["ux"] * ig, P["uy"] * ig, P["uz"] * ig, P["w"], -O.Q_E)
    assert per_slice_err(push[1:], np.stack(J)) < 1e-5
    s.close()
