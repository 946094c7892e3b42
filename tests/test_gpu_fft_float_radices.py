"""The float z-DFT of 7-smooth lengths (section "Finite order pseudo-spectral solvers": Fourier
transform along z) over every radix of its passes, single and composite, as first, middle and
last pass and alone, there and back, against numpy's float64 transform."""
import numpy as np
import pytest

from oracle import psatd_rz as O
from paper_1611_05712_gb300 import binding as bd
from gpu_helpers import per_slice_err

pytestmark = pytest.mark.gpu

DZ = 0.05e-6
# two to five passes; 10, 12, 14, 15, 9 alone; 24 = 6 4, 18 = 3 6, 28 = 7 4, 100, 144, 196 squares of
# composites, 225 = 15 15, 240 = 15 16, 210, 504, 1680 three different ones, 1536 = 12 8 16,
# 3600 and 6300 the longest turns of a CTA, 7203 = 7^4 3 and 7776 = 2^5 3^5 the most passes
SIZES = [9, 10, 12, 14, 15, 18, 20, 24, 28, 35, 36, 42, 54, 60, 90, 98, 100, 135, 144, 150, 196, 210, 225, 240, 250, 343,
         504, 525, 729, 1000, 1536, 1680, 2187, 2401, 3125, 3600, 6300, 7203, 7776, 8100]


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_05712_gb300.build import build
    build()


@pytest.mark.parametrize("Nz", SIZES)
def test_float_rows(Nz):
    g = O.Grid(Nz, 5, 1, DZ, DZ, DZ / O.C_LIGHT)
    s = bd.Sim(bd.make_config(Nz, 5, 1, DZ, DZ, g.dt, 0, True, bd.PIC_MIXED_TF32X3, 0))
    h = O.hankel_setup(g)
    rng = np.random.default_rng(Nz)
    crand = lambda *sh: rng.normal(size=sh) + 1j * rng.normal(size=sh)  # noqa: E731
    dep, eh = crand(4, 1, 5, Nz), crand(3, 1, 5, Nz)
    s.set("DEP", dep)
    s.forward_transform()
    fwd = s.get("SRC_H")
    s.set("EH", eh)
    s.inverse_transform()
    inv = s.get("E")
    s.close()
    # float rows: about 2^-24 a pass and twiddle of the row's norm, the largest of 5 Nz values some
    # 4 times that; the matrices' products add about as much
    assert per_slice_err(fwd, np.stack(O.forward_sources(g, h, *dep))) < 3e-6
    assert per_slice_err(inv, np.stack(O.inverse_vector(g, h, *eh))) < 3e-6


@pytest.mark.parametrize("Nz,Nr", [(1500, 700), (2187, 480), (3600, 320), (6300, 180), (7776, 160)])
def test_float_rows_of_many(Nz, Nr):
    """Beyond 900 points the composite radices need more rows than the SMs hold."""
    g = O.Grid(Nz, Nr, 1, DZ, DZ, DZ / O.C_LIGHT)
    s = bd.Sim(bd.make_config(Nz, Nr, 1, DZ, DZ, g.dt, 0, True, bd.PIC_MIXED_TF32X3, 0))
    h = O.hankel_setup(g)
    rng = np.random.default_rng(Nz)
    dep = rng.normal(size=(4, 1, Nr, Nz)) + 1j * rng.normal(size=(4, 1, Nr, Nz))
    eh = rng.normal(size=(3, 1, Nr, Nz)) + 1j * rng.normal(size=(3, 1, Nr, Nz))
    s.set("DEP", dep)
    s.forward_transform()
    fwd = s.get("SRC_H")
    s.set("EH", eh)
    s.inverse_transform()
    inv = s.get("E")
    s.close()
    # as above; the matrices' float products are sums of up to Nr terms here
    assert per_slice_err(fwd, np.stack(O.forward_sources(g, h, *dep))) < 1e-5
    assert per_slice_err(inv, np.stack(O.inverse_vector(g, h, *eh))) < 1e-5
