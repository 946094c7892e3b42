"""Batched graphs of simulations with a sort interval: the sorts in a graph may be odd in number, and every
launch still advances the particles that the launch before it left."""
import pytest

from oracle import psatd_rz as O
from paper_1611_05712_gb300 import binding as bd
from paper_1611_05712_gb300 import workloads as W
from gpu_helpers import by_id, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1611_05712_gb300.build import build
    build()


@pytest.mark.parametrize("precision,tol", [(bd.PIC_FP64, 1e-12), (bd.PIC_MIXED_TF32X3, 1e-5)])
@pytest.mark.parametrize("interval,cycles", [(1, 2), (2, 2), (2, 4), (3, 2), (3, 4), (4, 4), (16, 2)])
def test_launches_follow_one_another(precision, tol, interval, cycles):
    import torch
    w = W.tiny(order_p=16, seed=21, Nz=96, Nr=24, Nm=2, n_beam=400)
    w.dt = 0.5 * w.dz / O.C_LIGHT
    P, npl, beams = W.particles(w)
    a = bd.Sim.from_workload(w, P, npl, beams, precision=precision, stream=torch.cuda.Stream())
    b = bd.Sim.from_workload(w, P, npl, beams, precision=precision)
    for s in (a, b):
        s.set_sort_interval(interval)
    batch = bd.Batch([a], cycles=cycles)
    batch.launch(3)
    batch.origin.synchronize()
    b.step(3 * cycles)
    a.sync()
    # tolerances of the batch tests: the orders of atomic additions differ
    for name in ("E", "B", "RHO_PREV_H"):
        assert rel_err(a.get(name), b.get(name)) < tol, name
    pa, pb = by_id(a.read_particles()), by_id(b.read_particles())
    for k in bd.SOA:
        assert rel_err(pa[k], pb[k]) < tol, k
    batch.close()
    a.close()
    b.close()
