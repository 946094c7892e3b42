"""FP64 gather (power-of-two z lengths: weights from 62-bit fractions) of a particle a hair off a node in
z and in r: the weight of the far node is the product of two small fractions, down to 2^-100, and counts as
much as in float64 when the field is at that node alone."""
import numpy as np
import pytest

from oracle import psatd_rz as O
from paper_1611_05712_gb300 import binding as bd

pytestmark = pytest.mark.gpu

D = 2.0 ** -24   # metres: the particle's coordinates are exact


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_05712_gb300.build import build
    build()


@pytest.mark.parametrize("ez,er", [(5, 5), (30, 30), (33, 30), (40, 30), (50, 30), (60, 30), (61, 30), (20, 2)])
def test_product_of_small_fractions(ez, er):
    Nz, Nr, Nm = 64, 8, 2
    dt = D / O.C_LIGHT
    s = bd.Sim(bd.make_config(Nz, Nr, Nm, D, D, dt, 0, True, bd.PIC_FP64, 1, q=1.0, mass=1e-26))
    P = {"x": np.array([(0.5 + 2.0 ** -er) * D]), "y": np.zeros(1), "z": np.array([2.0 ** -ez * D]), "ux": np.zeros(1),
         "uy": np.zeros(1), "uz": np.zeros(1), "w": np.ones(1), "id": np.zeros(1, np.int32)}
    s.write_particles(P)
    E = s.zeros("E")
    top = 2.0 ** (ez + er) * 1e3 * 1e-26 / dt   # the push gives 1000 m/s; fields lie below 2^128
    E[2, 0, 1, 1] = top
    s.set("E", E)
    s.gather_push(False)
    uz = s.read_particles()["uz"][0]
    s.close()
    # the radius within two ulps (2^-52 of a cell, of a fraction of 2^-er), the weight within 2^-48
    # and a few ulps of the push
    assert abs(uz / 1e3 - 1) < 2.0 ** (er - 52) + 1e-13
