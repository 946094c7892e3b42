"""Inverse block fixed-point rows of the FP64 form at the lengths where their kernels change (CTAs of 256, 512
and 1024 threads, the longest rows of two shared buffers, 1/N that is no power of two), on sparse spectra, against
extended precision: no further off than 1.25 times the IEEE float64 rows or one rounding of the norm, whichever is more."""
import numpy as np
import pytest

from paper_1611_05712_gb300 import binding as bd
from test_gpu_fft_fixed import NR, ROWS, _close, _dft, _rows, _sim

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_05712_gb300.build import build
    build()


@pytest.mark.parametrize("Nz,scale", [(n, 1.0) for n in (128, 256, 512, 525, 1024, 1323, 2048, 2187, 3125, 4000, 4096, 8192)]
                         + [(1323, 1e-290), (2048, 1e280), (4096, 1e120)])
def test_long_inverse_rows(Nz, scale):
    s = _sim(Nz)
    rng = np.random.default_rng(Nz)
    eh = np.zeros((3, 1, NR, Nz), complex)
    eh[:, :, ROWS] = scale * _rows("spikes", rng, (3, 1, len(ROWS), Nz))
    s.set("EH", eh)
    s.inverse_transform()
    got = s.get("E")
    s.set_dht_path(bd.PIC_DHT_F64_GEMM)
    s.inverse_transform()
    ieee = s.get("E")
    mats = s.get("HANKEL_INV")[0]
    s.close()
    p, m, z = (mats[k][:, ROWS].astype(np.longdouble) @ (eh[c, 0, ROWS].astype(np.clongdouble) / scale)
               for c, k in enumerate((2, 0, 1)))
    ref = _dft(np.stack([p + m, 1j * (p - m), z]), +1) / Nz
    for c in range(3):
        _close(got[c, 0] / scale, ieee[c, 0] / scale, ref[c])
