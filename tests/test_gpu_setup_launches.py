"""Set-up of handles with few radial nodes goes straight to the one-sided Jacobi SVD: its sweeps over so small
matrices take fewer launches than the elimination, and are not run after it."""
import pytest

from paper_1611_05712_gb300 import binding as bd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_05712_gb300.build import build
    build()


@pytest.mark.parametrize("Nm", [1, 4])
@pytest.mark.parametrize("Nr,most", [(4, 40), (6, 60), (9, 90), (12, 100), (13, 115)])
def test_launches(Nr, most, Nm):
    # a sweep over Nr columns is Nr - 1 rounds (Nr if odd), and 5 or 6 sweeps converge; the rest of
    # set-up takes 16; elimination takes 95 and one per row (9 rows in 4 modes took both)
    s = bd.Sim(bd.make_config(8, Nr, Nm, 5e-8, 5e-8, 1e-16, 16, True, bd.PIC_FP64, 1))
    n = s.launch_count()
    s.close()
    assert n <= most
