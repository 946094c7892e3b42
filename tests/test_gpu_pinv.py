"""The forward Hankel matrices against numpy's pseudo-inverse (R-dht reading: singular values
<= 1e-3 sigma_max dropped) over radial sizes from the smallest to the largest: with no, one and
several modes' near-null directions, values just above and just below the cut (Nr = 9: 1.02e-3;
Nr = 64, m = 3: 9.1e-4), sizes around the tiles of the elimination, odd ones among them."""
import numpy as np
import pytest

from oracle import psatd_rz as O
from paper_1611_05712_gb300 import binding as bd

pytestmark = pytest.mark.gpu

DZ = 0.05e-6


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_05712_gb300.build import build
    build()


@pytest.mark.parametrize("Nr", [4, 5, 8, 9, 16, 31, 33, 48, 63, 64, 65, 100, 129, 240, 257, 400, 1000])
def test_pseudo_inverses(Nr):
    Nm = 4 if Nr < 300 else 2
    s = bd.Sim(bd.make_config(8, Nr, Nm, DZ, DZ, DZ / O.C_LIGHT, 0, True, bd.PIC_FP64, 0))
    B, M = s.get("HANKEL_INV"), s.get("HANKEL_FWD")
    s.close()
    h = O.hankel_setup(O.Grid(8, Nr, Nm, DZ, DZ, DZ / O.C_LIGHT))
    for m in range(Nm):
        for slot in range(3):
            # numpy's own error grows with the kept condition (up to 1e3) times its rounding
            ref = h.M[m][slot]
            assert np.abs(M[m, slot] - ref).max() < 1e-12 * np.abs(ref).max(), (m, slot)
            assert np.abs(M[m, slot] @ B[m, slot] @ M[m, slot] - M[m, slot]).max() < 1e-12 * np.abs(ref).max(), (m, slot)
