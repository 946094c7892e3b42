"""The block fixed-point z-DFT of the FP64 form (section "Finite order pseudo-spectral solvers":
Fourier transform along z) over every kind of length and row: each power of two and several
short rows per CTA, every radix first, last and alone, up to the longest rows; random, spiky,
sinusoidal and widely scaled rows.

Reference: the z-DFT in extended precision, through the library's own Hankel matrices (only a
few radial rows are filled, and 260 radial nodes take the eight-digit product, so that the rows'
arithmetic is what is measured), beside the IEEE float64 rows of PIC_DHT_F64_GEMM.
"""
import numpy as np
import pytest

from paper_1611_05712_gb300 import binding as bd

pytestmark = pytest.mark.gpu

DZ = 0.05e-6
NR = 260
ROWS = (0, 77, 259)


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_05712_gb300.build import build
    build()


def _sim(Nz):
    return bd.Sim(bd.make_config(Nz, NR, 1, DZ, DZ, DZ / 299792458.0, 32, True, bd.PIC_FP64, 0))


def _rows(kind, rng, shape):
    a = rng.normal(size=shape) + 1j * rng.normal(size=shape)
    n = shape[-1]
    if kind == "spikes":
        keep = np.zeros(n, bool)
        keep[rng.choice(n, 3, replace=False)] = True
        a = a * keep
    elif kind == "bump":     # a bunch: a few per cent of the row, decaying over 12 decades
        a = a * np.exp(-0.5 * ((np.arange(n) - 0.6 * n) / (0.02 * n + 1)) ** 2)
    return a


def _dft(X, sign):
    """sum_i X_i exp(sign 2 pi i k i / n) in extended precision, non-zero columns only."""
    n = X.shape[-1]
    used = np.flatnonzero((X != 0).any(axis=tuple(range(X.ndim - 1))))
    t = (np.arange(n)[None, :] * used[:, None]) % n
    ph = 2 * np.arccos(np.longdouble(-1)) * t.astype(np.longdouble) / n
    return X[..., used] @ (np.cos(ph) + sign * 1j * np.sin(ph))


def _close(got, ieee, ref):
    """No further off than the IEEE rows, or within one rounding of the result."""
    err = [np.linalg.norm(np.abs(a - ref).astype(float)) for a in (got, ieee)]
    norm = np.linalg.norm(np.abs(ref).astype(float))
    assert err[0] <= max(1.25 * err[1], 2.0 ** -53 * norm), (err[0] / norm, err[1] / norm)


RANDOM = [8, 9, 10, 12, 14, 15, 16, 21, 24, 32, 35, 45, 49, 64, 100, 125, 128, 147, 243, 256, 343]
LONG = [512, 525, 1000, 1024, 1323, 2048, 2187, 2401, 3125, 4000, 4096, 8192]


@pytest.mark.parametrize("Nz,kind,scale", [(n, "random", 1.0) for n in RANDOM] + [(n, "spikes", 1.0) for n in LONG]
                         + [(243, "bump", 1.0), (256, "bump", 1.0), (64, "random", 1e-290), (60, "random", 1e280),
                            (256, "random", 1e120)])
def test_forward_rows(Nz, kind, scale):
    s = _sim(Nz)
    rng = np.random.default_rng(Nz)
    dep = np.zeros((4, 1, NR, Nz), complex)
    dep[:, :, ROWS] = scale * _rows(kind, rng, (4, 1, len(ROWS), Nz))
    s.set("DEP", dep)
    s.forward_transform()
    got = s.get("SRC_H")
    s.set_dht_path(bd.PIC_DHT_F64_GEMM)
    s.forward_transform()
    ieee = s.get("SRC_H")
    mats = s.get("HANKEL_FWD")[0]
    s.close()
    d = dep[:, 0, ROWS].astype(np.clongdouble) / scale
    X = _dft(np.stack([d[0], (d[1] - 1j * d[2]) / 2, (d[1] + 1j * d[2]) / 2, d[3]]), -1)
    for c, slot in enumerate((1, 2, 0, 1)):
        ref = mats[slot][:, ROWS].astype(np.longdouble) @ X[c]
        _close(got[c, 0] / scale, ieee[c, 0] / scale, ref)


@pytest.mark.parametrize("Nz", [8, 12, 20, 27, 35, 64, 98])
def test_inverse_rows(Nz):
    s = _sim(Nz)
    rng = np.random.default_rng(Nz)
    eh = np.zeros((3, 1, NR, Nz), complex)
    eh[:, :, ROWS] = _rows("random", rng, (3, 1, len(ROWS), Nz))
    s.set("EH", eh)
    s.inverse_transform()
    got = s.get("E")
    s.set_dht_path(bd.PIC_DHT_F64_GEMM)
    s.inverse_transform()
    ieee = s.get("E")
    mats = s.get("HANKEL_INV")[0]
    s.close()
    p, m, z = (mats[k][:, ROWS].astype(np.longdouble) @ eh[c, 0, ROWS].astype(np.clongdouble)
               for c, k in enumerate((2, 0, 1)))
    ref = _dft(np.stack([p + m, 1j * (p - m), z]), +1) / Nz
    for c in range(3):
        _close(got[c, 0], ieee[c, 0], ref[c])


def test_longest_inverse_rows_undo_the_forward_ones():
    """8192 and 4000 points there and back (the scaling by 1/N and the last pass's exponent)."""
    for Nz in (4000, 8192):
        s = _sim(Nz)
        rng = np.random.default_rng(Nz)
        E = np.zeros((3, 1, NR, Nz), complex)
        # a field of the transforms' range: the inverse transform of a random spectrum
        eh = np.zeros_like(E)
        eh[:, :, 3:200:7] = rng.normal(size=(3, 1, 29, Nz)) + 1j * rng.normal(size=(3, 1, 29, Nz))
        s.set("EH", eh)
        s.inverse_transform()
        E = s.get("E")
        s.fields_to_spectral()
        s.inverse_transform()
        back = s.get("E")
        s.close()
        assert np.abs(back - E).max() < 1e-12 * np.abs(E).max()
