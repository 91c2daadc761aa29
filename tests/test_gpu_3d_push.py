"""The two forms of the 3D push (few particles: tiles split over blocks, particles over four lanes; many: a block per
tile, a lane per particle) and the sort by cell, on boxes whose sides are no multiple of the tile (4 x 4 x 16 cells),
against the 3D FP64 CPU oracle: relative L2 <= 1e-10 on the fields, the particle state and the charge density, as every
FP64 comparison of the 3D path (sums of some hundred terms in another order: 1e-14)."""
import numpy as np
import pytest

from paper_1009_2727_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL64 = 1e-10
PER_SM = 256


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("many", [False, True])
@pytest.mark.parametrize("order,gather", [(3, "energy"), (3, "momentum"), (1, "energy")])
def test_3d_push_forms(orc, many, order, gather):
    import torch
    from paper_1009_2727_gb300.pic import Simulation
    w = W.shrink3(W.parity_3d(), 29, 27, 70, order=order, gather=gather)
    w["plasma"].update(dict(ppc_x=4, ppc_y=3, ppc_z=5) if many else dict(ppc_x=2, ppc_y=1, ppc_z=3))
    g = Simulation(w, precision="fp64")
    o = orc.Sim3(w)
    g.step(16)
    o.step(16)
    g.sync()
    n = g.stats()["n_electrons"]
    few_max = PER_SM * torch.cuda.get_device_properties(0).multi_processor_count
    assert n > 1000 and (n > few_max) == many, n
    for grp in ((0, 1, 2), (3, 4, 5), (9,)):
        a = np.stack([g.field(c) for c in grp])
        b = np.stack([o.rho() if c == 9 else o.field(c) for c in grp])
        assert rel(a, b) <= TOL64, grp
    pg, po = g.particles(0), o.particles(0)
    po = {k: v[po["alive"]] for k, v in po.items()}
    ig, io = np.argsort(pg["id"], kind="stable"), np.argsort(po["id"], kind="stable")
    assert np.array_equal(pg["id"][ig], po["id"][io])
    for k in ("x", "y", "z", "w"):
        assert rel(pg[k][ig], po[k][io]) <= TOL64, k
    assert rel(np.stack([pg[k][ig] for k in ("ux", "uy", "uz")]), np.stack([po[k][io] for k in ("ux", "uy", "uz")])) <= TOL64


def test_3d_grid_that_fills_the_chip(orc):
    """a grid past the lines below which a filter pass takes all components in one launch and Faraday tiles of two x nodes:
    antenna in vacuum with PML, compensated filter and damping against the oracle, 1e-10"""
    from paper_1009_2727_gb300.pic import Simulation
    w = W.shrink3(W.parity_3d(), 49, 50, 1000, theta=0.2, filter_passes=2, filter_compensate=1)
    del w["plasma"]
    w["laser"]["t_peak"] = 4e-15
    g = Simulation(w, precision="fp64")
    o = orc.Sim3(w)
    g.step(8)
    o.step(8)
    g.sync()
    assert np.abs(o.field(1)).max() > 0
    for grp in ((0, 1, 2), (3, 4, 5)):
        a = np.stack([g.field(c) for c in grp])
        b = np.stack([o.field(c) for c in grp])
        assert rel(a, b) <= TOL64, grp
