"""The digit-sliced FP64 DHT at the edges of its two forms (section "Finite order
pseudo-spectral solvers": Hankel transform along r): radial sizes around the 256 rows where the
six-digit form ends and the accumulators of the eight-digit form are first drained, around
multiples of its 64-row tiles and 32-wide K chunks, and the smallest and largest grids.

Reference: the library's own matrices times the z-DFT of the panel in extended precision, so
that only the transforms' arithmetic is compared.  The z lengths are not powers of two, so the
rows are IEEE float64 FFTs on both paths.
"""
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


def _sim(Nz, Nr, Nm):
    return bd.Sim(bd.make_config(Nz, Nr, Nm, DZ, DZ, DZ / 299792458.0, 32, True, bd.PIC_FP64, 0))


def _panel(kind, rng, shape):
    j = np.arange(shape[2])[None, None, :, None]
    a = rng.normal(size=shape) + 1j * rng.normal(size=shape)
    if kind == "beam":      # on the axis, where the forward matrices' entries are small
        a = np.exp(-(20.0 * j / shape[2]) ** 2) * (1 + 1e-3 * a)
    if kind == "spread":    # columns and rows over many orders of magnitude
        a = a * 10.0 ** rng.uniform(-9, 9, size=(1, 1, 1, shape[3])) * 10.0 ** rng.uniform(-6, 0, size=(1, 1, shape[2], 1))
    return a


def _reference(mats, dep):
    """rho^, J_+^, J_-^, J_z^ in extended precision, and the z-transformed panels."""
    ld = np.longdouble
    n = dep.shape[-1]
    ph = 2 * np.arccos(ld(-1)) * ((np.arange(n)[:, None] * np.arange(n)[None, :]) % n).astype(ld) / n
    W = np.cos(ph) - 1j * np.sin(ph)
    d = dep.astype(np.clongdouble)
    parts = np.stack([d[0], (d[1] - 1j * d[2]) / 2, (d[1] + 1j * d[2]) / 2, d[3]])
    X = parts @ W
    out = np.empty_like(X)
    for c in range(4):
        for m in range(dep.shape[1]):
            out[c, m] = mats[m, SLOT[c]].astype(ld) @ X[c, m]
    return out, X


@pytest.mark.parametrize("Nz,Nr,Nm", [(12, 4, 1), (10, 33, 3), (14, 63, 2), (12, 255, 1), (20, 256, 2), (12, 257, 1),
                                      (10, 320, 2), (14, 511, 1), (12, 513, 1), (10, 1024, 1)])
@pytest.mark.parametrize("kind", ["random", "beam", "spread"])
def test_forward_transform_against_extended_precision(Nz, Nr, Nm, kind):
    s = _sim(Nz, Nr, Nm)
    rng = np.random.default_rng(Nz + 13 * Nr)
    dep = _panel(kind, rng, (4, Nm, Nr, Nz))
    s.set("DEP", dep)
    s.forward_transform()
    got = s.get("SRC_H")
    s.set_dht_path(bd.PIC_DHT_F64_GEMM)
    s.forward_transform()
    gemm = s.get("SRC_H")
    mats = s.get("HANKEL_FWD")
    s.close()
    ref, X = _reference(mats, dep)
    err = lambda a: np.abs(a - ref).astype(float)  # noqa: E731
    # worst case of the digits: K 2^-46 of (row maximum x column maximum); the rows' own FFT
    # error (about 1e-15 of the row's norm) passes through the matrix
    for c in range(4):
        for m in range(Nm):
            A = np.abs(mats[m, SLOT[c]])
            bound = 2.0 ** -46 * Nr * A.max(1)[:, None] * np.abs(X[c, m]).astype(float).max(0)[None, :]
            fft = 1e-15 * np.log2(Nz) * (A @ np.linalg.norm(dep[:, m].astype(complex), axis=(0, 2)))[:, None]
            assert (err(got)[c, m] <= bound + fft).all(), (c, m)
    if Nr > 256:   # the eight-digit form took the float64 product's place: no less accurate
        for c in range(4):
            for m in range(Nm):
                assert np.linalg.norm(err(got)[c, m]) <= 1.1 * np.linalg.norm(err(gemm)[c, m]) + 2.0 ** -53 * \
                    np.linalg.norm(np.abs(ref[c, m]).astype(float)), (c, m)


@pytest.mark.parametrize("Nr", [64, 300])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_input_reaches_the_outputs(Nr, bad):
    """A NaN or an infinity in E_z makes the whole of E_z^ non-finite (the z-DFT spreads it over
    the row, the product over the radial wavenumbers) and leaves the other components alone."""
    s = _sim(12, Nr, 1)
    rng = np.random.default_rng(Nr)
    E = rng.normal(size=(3, 1, Nr, 12)) + 1j * rng.normal(size=(3, 1, Nr, 12))
    s.set("E", E)
    s.fields_to_spectral()
    ref = s.get("EH")
    E[2, 0, Nr // 2, 5] = bad
    s.set("E", E)
    s.fields_to_spectral()
    got = s.get("EH")
    s.close()
    assert not np.isfinite(got[2]).any()
    assert np.isfinite(ref).all() and np.array_equal(got[:2], ref[:2])
