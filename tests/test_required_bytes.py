"""Workspace of FP64 handles beyond 256 radial nodes: the eight digit planes of the DHT take no memory of
their own where the spare particle buffer holds them (host-only)."""
import os
import shutil

import pytest

from paper_1611_05712_gb300 import binding as bd


@pytest.fixture(scope="module")
def lib():
    if shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("nvcc not available")
    from paper_1611_05712_gb300.build import build
    build()
    return bd.load()


def _bytes(Nz, Nr, Nm, n):
    return bd.required_bytes(bd.make_config(Nz, Nr, Nm, 5e-8, 5e-8, 1e-16, 0, True, bd.PIC_FP64, n))


# bytes these handles took with the float64 SIMT product alone, and what the matrices' planes (96 B a
# matrix entry and mode, less 48 of set-up scratch) may add
@pytest.mark.parametrize("Nz,Nr,Nm,n,plain", [(1800, 400, 2, 5000000, 1418413568), (4096, 512, 3, 12 * 4096 * 512, 7157555200),
                                              (8192, 1024, 3, 12 * 8192 * 1024, 28624261120)])
def test_planes_in_the_spare_buffer(lib, Nz, Nr, Nm, n, plain):
    assert _bytes(Nz, Nr, Nm, n) <= plain + 48 * Nm * Nr * (Nr + 8) + (1 << 20)


@pytest.mark.parametrize("Nz,Nr,Nm", [(1800, 400, 2), (600, 640, 2), (4096, 1024, 1)])
def test_a_larger_particle_buffer_takes_the_planes(lib, Nz, Nr, Nm):
    # below the size that holds the planes, a particle more costs its one buffer (60 B) and 12 B of
    # sort keys and places, not both buffers
    a, b = _bytes(Nz, Nr, Nm, 32), _bytes(Nz, Nr, Nm, 100032)
    assert abs((b - a) - 72 * 100000) < 1 << 14
