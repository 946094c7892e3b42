"""The stable counting sort by cell at the cell counts where its routines change (one particle, a
warp, the largest cell ordered particle by particle, the first crowded ones, several merge passes),
in the first and last cells and across the blocks of the scan, bit for bit in both forms."""
import numpy as np
import pytest

from oracle import psatd_rz as O
from paper_1611_05712_gb300 import binding as bd

pytestmark = pytest.mark.gpu

COUNTS = [1, 2, 3, 31, 32, 33, 64, 127, 128, 129, 130, 2048, 2049, 4097, 5000]


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_05712_gb300.build import build
    build()


@pytest.mark.parametrize("precision", [bd.PIC_FP64, bd.PIC_MIXED_TF32X3])
@pytest.mark.parametrize("Nz,Nr", [(8, 4), (64, 63), (64, 64), (2048, 1024)])
def test_cell_counts(precision, Nz, Nr):
    ncell, dz = Nz * Nr, 0.05e-6
    g = O.Grid(Nz, Nr, 1, dz, dz, 0.5 * dz / O.C_LIGHT)
    rng = np.random.default_rng(ncell)
    cells = np.unique(np.concatenate([[0, ncell - 1, min(4095, ncell - 1), min(4096, ncell - 1)],
                                      rng.choice(ncell, min(11, ncell // 3), replace=False)]))
    key = np.concatenate([np.repeat(cells, rng.permutation(COUNTS)[: len(cells)]), rng.integers(0, ncell, 3000)])
    rng.shuffle(key)
    n = len(key)
    th = 0.5 * np.pi * rng.integers(0, 4, n)   # on the axes of x and y, at the cells' centres
    r = (key % Nr + 0.5) * dz
    P = {"x": r * np.round(np.cos(th)), "y": r * np.round(np.sin(th)), "z": (key // Nr + 0.5) * dz,
         "ux": rng.normal(size=n), "uy": np.zeros(n), "uz": np.zeros(n), "w": np.ones(n),
         "id": np.arange(n, dtype=np.int32)}
    s = bd.Sim(bd.make_config(Nz, Nr, 1, dz, dz, g.dt, 0, True, precision, n))
    s.write_particles(P)
    before = s.read_particles()
    for _ in range(2):   # from random order, then from the sorted one
        s.sort()
        perm = np.argsort(key, kind="stable")
        assert np.array_equal(s.get("KEYS"), key)
        assert np.array_equal(s.get("PERM"), perm)
        got = s.read_particles()
        for k in before:
            assert np.array_equal(got[k], before[k][perm]), k
        key, before = key[perm], got
    s.close()
