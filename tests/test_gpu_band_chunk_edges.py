"""Mixed-form deposits at the particle numbers where the chunks of a shared band end, for each chunk length that
can be chosen (pic_set_tuning), in both mixed forms' particle kernels: rho and J, and the push's J and rho."""
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


@pytest.mark.parametrize("chunk", [512, 1024, 2048])
@pytest.mark.parametrize("off", [-1, 0, 1])
@pytest.mark.parametrize("chunks", [1, 2, 304])
def test_ends_of_chunks(chunk, off, chunks):
    n = chunk * chunks + off
    Nz, Nr, Nm, dz = 64, 20, 2, 0.05e-6
    g = O.Grid(Nz, Nr, Nm, dz, dz, dz / O.C_LIGHT)
    rng = np.random.default_rng(n)
    r = g.R * 0.98 * np.sqrt(rng.uniform(0, 1, n))
    th = rng.uniform(0, 2 * np.pi, n)
    P = dict(x=r * np.cos(th), y=r * np.sin(th), z=rng.uniform(0, g.L, n), ux=rng.normal(0, 3e7, n),
             uy=rng.normal(0, 3e7, n), uz=rng.normal(1e8, 3e8, n), w=rng.uniform(0.5, 2.0, n) * 1e4,
             id=np.arange(n, dtype=np.int32))
    s = bd.Sim(bd.make_config(Nz, Nr, Nm, dz, dz, g.dt, 0, True, bd.PIC_MIXED_TF32X3, n))
    s.set_tuning(band_chunk=chunk)
    s.write_particles(P)
    s.sort()
    P = s.read_particles()
    s.deposit(bd.PIC_DEP_RHO | bd.PIC_DEP_J)
    dep = s.get("DEP")
    s.gather_push(fuse_current=True)
    push = s.get("DEP")
    s.close()
    # float weights and phases, a few 2^-24 each, in the sums of every slice
    ig = O.inv_gamma(P["ux"], P["uy"], P["uz"])
    v = [P[k] * ig for k in ("ux", "uy", "uz")]
    J = O.deposit_current(g, P["x"], P["y"], P["z"], *v, P["w"], -O.Q_E)
    assert per_slice_err(dep[0:1], O.deposit_rho(g, P["x"], P["y"], P["z"], P["w"], -O.Q_E)[None]) < 1e-5
    assert per_slice_err(dep[1:], np.stack(J)) < 1e-5
    h = 0.5 * g.dt   # no fields: J half a step on
    J = O.deposit_current(g, P["x"] + h * v[0], P["y"] + h * v[1], (P["z"] + h * v[2]) % g.L, *v, P["w"], -O.Q_E)
    assert per_slice_err(push[1:], np.stack(J)) < 1e-5
