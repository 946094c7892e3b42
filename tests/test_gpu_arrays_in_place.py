"""Particle sets in device arrays that end with their allocation: written and read in place by the
library's kernels, bit for bit, in both forms."""
import ctypes

import numpy as np
import pytest

from oracle import psatd_rz as O
from paper_1611_05712_gb300 import binding as bd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_05712_gb300.build import build
    build()


@pytest.mark.parametrize("precision", [bd.PIC_FP64, bd.PIC_MIXED_TF32X3])
@pytest.mark.parametrize("n", [1, 257, 30001])
def test_arrays_at_the_end_of_their_allocation(precision, n):
    import torch
    D = 0.05e-6
    torch.cuda.empty_cache()
    # an allocation of its own for every array: 32 MiB each, its last n elements
    pool = [torch.empty((32 << 20) // 8, dtype=torch.float64, device="cuda") for _ in range(7)]
    ids = torch.empty((32 << 20) // 4, dtype=torch.int32, device="cuda")
    rng = np.random.default_rng(n)
    r, th = rng.uniform(0, 31 * D, n), rng.uniform(0, 2 * np.pi, n)
    P = {"x": r * np.cos(th), "y": r * np.sin(th), "z": rng.uniform(0, 63.9 * D, n), "ux": rng.normal(size=n),
         "uy": rng.normal(size=n), "uz": rng.normal(size=n), "w": rng.uniform(1, 2, n), "id": np.arange(n, dtype=np.int32)}
    dev = {k: pool[i][-n:].copy_(torch.from_numpy(P[k])) for i, k in enumerate(bd.SOA)}
    dev["id"] = ids[-n:].copy_(torch.from_numpy(P["id"]))
    sims = [bd.Sim(bd.make_config(64, 32, 1, D, D, D / O.C_LIGHT, 0, True, precision, n)) for _ in range(2)]
    k0 = sims[0].launch_count()
    sims[0].write_particles(dev)
    assert sims[0].launch_count() == k0 + 1   # one kernel on the arrays themselves
    sims[1].write_particles(P)
    a, b = (s.read_particles() for s in sims)
    for t in dev.values():
        t.fill_(-1)
    ptrs = (ctypes.c_void_p * 7)(*[dev[k].data_ptr() for k in bd.SOA])
    bd._check(sims[0].lib.pic_read_particles(sims[0].h, ptrs, ctypes.c_void_p(dev["id"].data_ptr()), n, 0), "read")
    for k in a:
        assert np.array_equal(a[k], b[k]) and np.array_equal(a[k], dev[k].cpu().numpy()), k
    for s in sims:
        s.close()
