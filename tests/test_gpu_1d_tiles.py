"""1D field tiles and push blocks at their edges against the 1D FP64 oracle: node counts at and next to a multiple of the
64-node tile, filters of small and full reach across the tiles, the window's shift through the fused field kernel, one
step per call against many, electron counts around a block."""
import numpy as np
import pytest

from paper_1009_2727_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL64 = 1e-10   # FP64 sums in another order over 120 steps: the bound of the other FP64 parity tests


def fields_close(g, o):
    for grp in ((0, 1, 2), (3, 4, 5)):
        a, b = (np.stack([s.field(c) for c in grp]) for s in (g, o))
        assert np.linalg.norm(a - b) <= TOL64 * np.linalg.norm(b)


@pytest.mark.parametrize("nz,strides,gather,order,ppc", [
    (383, (), "energy", 3, 4), (384, (1, 2), "momentum", 3, 2), (385, (1, 2, 4), "energy", 1, 3),
    (447, (1, 2, 4), "momentum", 3, 1)])
def test_boosted_tiles(nz, strides, gather, order, ppc):
    import oracle
    from paper_1009_2727_gb300.pic import Simulation
    w = W.parity_1d()
    w.update(nz=nz, filter_strides=list(strides), gather=gather, order=order)
    if strides:
        w["filter_passes"] = 4
    dz = (1.0 + np.sqrt(1 - 1 / w["gamma_boost"] ** 2)) * w["gamma_boost"] * w["dz_lab"]
    w["plasma"].update(ppc_z=ppc, z_start_lab=w["gamma_boost"] * 90 * dz)
    w["laser"]["z_antenna"] = 70 * dz
    g, o = Simulation(w), oracle.Sim1(w)
    for n in (1, 2, 117):
        g.step(n)
        o.step(n)
        g.sync()
        fields_close(g, o)
    pg, po = g.particles(0), o.particles(0)
    a, b = np.argsort(pg["id"], kind="stable"), np.argsort(po["id"], kind="stable")
    assert np.array_equal(pg["id"][a], po["id"][b])
    assert np.abs(pg["z"][a] - po["z"][b]).max() <= TOL64 * np.abs(po["z"]).max()
    g.close()


@pytest.mark.parametrize("nz,courant", [(255, 1.0), (256, 0.7), (320, 1.0)])
def test_window_tiles(nz, courant):
    import oracle
    from paper_1009_2727_gb300.pic import Simulation
    w = W.app1_lwfa(True)
    dz = w["dz_lab"]
    w.update(nz=nz, precision="fp64", courant=courant, filter_gather=1)
    w["plasma"].update(ppc_z=3, z_start_lab=(nz - 50) * dz)
    w["laser"].update(z_antenna=(nz - 60) * dz, t_peak=0.2 * w["laser"]["tau_fwhm"])
    g, o = Simulation(w), oracle.Sim1(w)
    for n in (1, 40, 160):
        g.step(n)
        o.step(n)
        g.sync()
        fields_close(g, o)
    assert len(g.particles(0)["z"]) == len(o.particles(0)["z"])
    g.close()
