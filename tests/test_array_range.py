"""The address checks that decide whether a kernel may work on a caller's device arrays themselves
(csrc/array_range.cuh), compiled for the host: an array that ends past its allocation, or shares a byte
with the workspace, is never taken for one that does not."""
import ctypes
import os
import random
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include "array_range.cuh"
extern "C" int inside(uint64_t base, uint64_t bytes, uint64_t p, int64_t n, uint64_t size) {
  return pic::array_inside(base, bytes, p, n, size);
}
extern "C" int apart(uint64_t p, int64_t n, uint64_t size, uint64_t q, uint64_t bytes) {
  return pic::array_apart(p, n, size, q, bytes);
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("range")
    (d / "range.cpp").write_text(SRC)
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-I", os.path.join(ROOT, "paper_1611_05712_gb300", "csrc"),
                    str(d / "range.cpp"), "-o", str(d / "range.so")], check=True)
    so = ctypes.CDLL(str(d / "range.so"))
    so.inside.argtypes = [ctypes.c_uint64, ctypes.c_uint64, ctypes.c_uint64, ctypes.c_int64, ctypes.c_uint64]
    so.apart.argtypes = [ctypes.c_uint64, ctypes.c_int64, ctypes.c_uint64, ctypes.c_uint64, ctypes.c_uint64]
    return so


@pytest.mark.parametrize("base", [1 << 40, (1 << 64) - (1 << 20)])
def test_inside(lib, base):
    b = 1 << 19
    for size in (4, 8):
        full = b // size
        assert lib.inside(base, b, base, full, size) and not lib.inside(base, b, base, full + 1, size)
        assert lib.inside(base, b, base + b - size, 1, size) and not lib.inside(base, b, base + b - size, 2, size)
        assert not lib.inside(base, b, base + b - 1, 1, size) and not lib.inside(base, b, base - size, 1, size)
        assert not lib.inside(base, b, base + b + 8, 1, size) and not lib.inside(base, b, base, (1 << 63) - 1, size)
        assert lib.inside(base, b, base + b, 0, size) and not lib.inside(base, b, base, -1, size)
    rng = random.Random(3)
    for _ in range(2000):
        p, n, size = base + rng.randrange(-64, b + 64), rng.randrange(0, b // 4 + 16), rng.choice((4, 8))
        assert bool(lib.inside(base, b, p, n, size)) == (p >= base and p + n * size <= base + b)


def test_apart(lib):
    rng = random.Random(5)
    for _ in range(4000):
        p, q = 4096 + rng.randrange(400), 4096 + rng.randrange(400)
        n, size, nb = rng.randrange(0, 30), rng.choice((4, 8)), rng.randrange(0, 200)
        assert bool(lib.apart(p, n, size, q, nb)) == (not set(range(p, p + n * size)) & set(range(q, q + nb)))
