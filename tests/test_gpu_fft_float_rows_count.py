"""The float z-DFT's plans change with the number of rows (radices up to 8, or composite ones): up to 900 points
on both sides of that line, and the lengths beyond whose composite plans differ in kind (three different
radices, odd ones alone, the longest turns of a CTA), with rows enough to take them, there and back
against numpy's float64 transform."""
import numpy as np
import pytest

from oracle import psatd_rz as O
from paper_1611_05712_gb300 import binding as bd
from gpu_helpers import per_slice_err

pytestmark = pytest.mark.gpu

DZ = 0.05e-6


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_05712_gb300.build import build
    build()


def _check(Nz, Nr, Nm):
    g = O.Grid(Nz, Nr, Nm, DZ, DZ, DZ / O.C_LIGHT)
    s = bd.Sim(bd.make_config(Nz, Nr, Nm, DZ, DZ, g.dt, 0, True, bd.PIC_MIXED_TF32X3, 0))
    h = O.hankel_setup(g)
    rng = np.random.default_rng(Nz)
    crand = lambda *sh: rng.normal(size=sh) + 1j * rng.normal(size=sh)  # noqa: E731
    dep, eh = crand(4, Nm, Nr, Nz), crand(3, Nm, Nr, Nz)
    s.set("DEP", dep)
    s.forward_transform()
    fwd = s.get("SRC_H")
    s.set("EH", eh)
    s.inverse_transform()
    inv = s.get("E")
    s.close()
    # float rows: about 2^-24 a pass and twiddle of the row's norm, the largest of Nr Nz values some 5
    # times that; the matrices' float products, sums of up to Nr terms, add about as much
    assert per_slice_err(fwd, np.stack(O.forward_sources(g, h, *dep))) < 1e-5
    assert per_slice_err(inv, np.stack(O.inverse_vector(g, h, *eh))) < 1e-5


@pytest.mark.parametrize("Nr", [149, 150])   # 596 and 600 rows
@pytest.mark.parametrize("Nz", [9, 10, 12, 14, 15, 18, 24, 28, 35, 54, 90, 98, 135, 144, 150, 196, 225, 240, 250, 343, 504,
                                525, 729, 750, 900])
def test_short_rows_on_both_sides_of_the_line(Nz, Nr):
    _check(Nz, Nr, 1)


@pytest.mark.parametrize("Nz,Nr,Nm", [(1000, 532, 2), (1536, 342, 2), (1680, 304, 2), (2401, 228, 2), (3125, 152, 2),
                                      (7203, 76, 2), (8100, 38, 2)])
def test_long_rows_in_composite_passes(Nz, Nr, Nm):
    _check(Nz, Nr, Nm)
