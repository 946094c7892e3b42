"""FP64 DHT whose panels' digit planes share memory with the spare particle buffer: held by it, held in
part and not at all, with either particle buffer current.  Field steps leave the particles as they are,
and give bit for bit what a handle without particles gives."""
import numpy as np
import pytest

from oracle import psatd_rz as O
from paper_1611_05712_gb300 import binding as bd

pytestmark = pytest.mark.gpu
D = 0.05e-6


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_05712_gb300.build import build
    build()


def _sim(Nz, Nr, Nm, n):
    return bd.Sim(bd.make_config(Nz, Nr, Nm, D, D, 0.5 * D / O.C_LIGHT, 16, True, bd.PIC_FP64, n))


@pytest.mark.parametrize("Nz,Nr,Nm,counts", [(48, 300, 1, (1, 20000, 47000, 100000)), (64, 32, 2, (1, 3000, 9830, 20000)),
                                             (27, 40, 3, (50000,))])
def test_planes_in_the_spare_buffer(Nz, Nr, Nm, counts):
    rng = np.random.default_rng(Nr)
    dep = rng.normal(size=(4, Nm, Nr, Nz)) + 1j * rng.normal(size=(4, Nm, Nr, Nz))
    dep[:, 0].imag = 0.0

    def fields(s, steps=2):
        s.set("DEP", dep)
        for _ in range(steps):
            s.field_step()
        return [s.get(k) for k in ("E", "B", "EH", "BH", "RHO_PREV_H")]

    s = _sim(Nz, Nr, Nm, 0)
    want = fields(s)
    s.close()
    for n in counts:
        r, th = rng.uniform(0, (Nr - 1) * D, n), rng.uniform(0, 2 * np.pi, n)
        P = {"x": r * np.cos(th), "y": r * np.sin(th), "z": rng.uniform(0, Nz * D, n), "ux": rng.normal(size=n),
             "uy": rng.normal(size=n), "uz": rng.normal(size=n), "w": np.ones(n), "id": np.arange(n, dtype=np.int32)}
        for sorts in (0, 1, 2):   # the current buffer: first, second, first
            s = _sim(Nz, Nr, Nm, n)
            s.write_particles(P)
            for _ in range(sorts):
                s.sort()
            before = s.read_particles()
            got = fields(s)
            after = s.read_particles()
            s.close()
            for a, b in zip(got, want):
                assert np.array_equal(a, b)
            for k in before:
                assert np.array_equal(before[k], after[k]), k
