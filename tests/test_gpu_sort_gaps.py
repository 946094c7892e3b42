"""The mixed form's sort, whose permutation finds the cells of 32 places at a time from the cells' ends in sets of 1.5 M
particles and more: particles a fixed number of cells apart (one to beyond the 128 cells that are searched), cells
that end with the 32 places and around them, and inactive particles behind them (moving window), bit for bit; the
same in small sets, which go by the keys."""
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


def _check(Nz, Nr, key, window=False):
    n = len(key)
    rng = np.random.default_rng(n)
    key = rng.permutation(key)
    r = (key % Nr + 0.5) * D
    P = {"x": r, "y": np.zeros(n), "z": (key // Nr + 0.5) * D, "ux": rng.normal(size=n), "uy": np.zeros(n), "uz": np.zeros(n),
         "w": np.ones(n), "id": np.arange(n, dtype=np.int32)}
    s = bd.Sim(bd.make_config(Nz, Nr, 1, D, D, 0.5 * D / O.C_LIGHT, 0, True, bd.PIC_MIXED_TF32X3, n + 200))
    s.write_particles(P)
    if window:   # 77 inactive particles appended
        s.init_background(n)
        s.init_fields()
        s.window_setup(n, 1, 77)
    before = s.read_particles()
    s.sort()
    perm, got = s.get("PERM"), s.read_particles()
    s.close()
    want = np.argsort(key, kind="stable")
    assert np.array_equal(perm[:n], want)
    for k in before:
        assert np.array_equal(got[k][:n], before[k][:n][want]), k
    if window:
        assert (got["w"][n:] == 0).all() and sorted(perm[n:]) == list(range(n, n + 77))


@pytest.mark.parametrize("gap", [1, 2, 3, 31, 32, 33, 63, 127, 128, 129, 500])
@pytest.mark.parametrize("n", [1, 31, 33, 700])
def test_gaps(gap, n):
    Nr = 64
    Nz = max(8, 2 * ((gap * n) // (2 * Nr) + 2))
    _check(Nz if Nz <= 4096 else 8192, Nr, np.arange(n) * gap + 5)


@pytest.mark.parametrize("counts", [(32, 32, 32), (31, 1, 32, 33), (64, 0, 0, 63, 1), (128, 129, 127), (1, 2000, 31, 96), (16,) * 40,
                                    (5, 130, 0, 27, 3, 95)])
@pytest.mark.parametrize("window", [False, True])
def test_cells_around_the_places(counts, window):
    key = np.repeat(np.arange(len(counts)) * 3, counts)
    _check(16, 16, key, window)


@pytest.mark.parametrize("n", [(3 << 19) - 1, 3 << 19, (3 << 19) + 1, (3 << 19) + 77777])
@pytest.mark.parametrize("window", [False, True])
def test_sets_that_are_searched(n, window):
    Nz, Nr = 2048, 512   # 1 M cells
    parts, at = [], 7
    for counts in ((32, 32, 32), (31, 1, 32, 33), (64, 0, 0, 63, 1), (128, 129, 127), (1, 2000, 31, 96), (5, 130, 0, 27, 3, 95)):
        parts.append(np.repeat(at + np.arange(len(counts)), counts))
        at += len(counts) + 300
    for gap in (2, 3, 16, 31, 32, 33, 63, 127, 128, 129, 500):
        parts.append(at + gap * np.arange(400))
        at += gap * 400
    left = n - sum(len(p) for p in parts)
    cells = Nz * Nr - at - 100000   # the rest at 3 a cell, the last 100000 cells empty but for two
    parts.append(at + np.arange(left - 2) % cells)
    parts.append(np.array([Nz * Nr - 50000, Nz * Nr - 1]))
    _check(Nz, Nr, np.concatenate(parts), window)
