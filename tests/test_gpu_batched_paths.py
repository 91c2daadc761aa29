"""The batched ensemble step where its kernels differ from a single run's: chunks at rest through inflow, several sorts and
plasma leaving at -z, and filters with strides (the tile kernels there, two-pass kernels in a run alone). Against each run
alone: FP64 to 1e-11 over 25 steps (the filters' sums of up to 41 terms per axis in another order, 9e-15 each, twice a step;
atomic sums in another order), mixed to 1e-4 on the
fields and 1e-3 cells on the positions, as the comparison of resting with pushed chunks."""
import numpy as np
import pytest

from paper_1009_2727_gb300 import capi
from paper_1009_2727_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def boosted(nx, nz, ppc, laser=True):
    w = W.shrink(W.stage_2d(5.0), nx, nz, precision="mixed")
    w["pml_cells"] = 6
    dz = (1.0 + np.sqrt(1 - 1 / 25.0)) * 5.0 * w["dz_lab"]
    w["laser"].update(z_antenna=24 * dz, t_peak=6e-15)
    # the plasma's front has streamed out through -z by the end
    w["plasma"].update(ppc_x=ppc, ppc_z=ppc, z_start_lab=5.0 * 120 * dz, ramp_lab=2e-6)
    w["sort_every"] = 32
    if not laser:
        del w["laser"]
    return w


@pytest.mark.parametrize("laser", [True, False], ids=["laser", "dark"])
@pytest.mark.parametrize("graphs", [True, False], ids=["graphs", "launches"])
def test_chunks_at_rest(laser, graphs):
    from paper_1009_2727_gb300.pic import Ensemble, Simulation
    ws = [boosted(96, 256, 2, laser), boosted(80, 288, 4, laser), boosted(112, 240, 1, laser)]
    ens = Ensemble(ws)
    assert ens.batched
    ens.use_graphs(graphs)
    ens.step(260)
    ens.sync()
    for m, w in zip(ens.members, ws):
        alone = Simulation(w)
        f = np.full(alone.shape, 1e-25)     # no chunk of the run alone is at rest
        for c in range(6):
            alone.set_field(c, f)
        alone.step(260)
        alone.sync()
        assert m.push_counts()[1] > 0 and alone.push_counts()[1] == 0
        pa, pb = m.particles(capi.ELECTRONS), alone.particles(capi.ELECTRONS)
        a, b = np.argsort(pa["id"], kind="stable"), np.argsort(pb["id"], kind="stable")
        assert len(a) > 0 and np.array_equal(pa["id"][a], pb["id"][b])
        for k in ("x", "z"):
            assert np.abs(pa[k][a] - pb[k][b]).max() <= 1e-3 * alone.stats()["dz"]
        if laser:
            for grp in ((0, 1, 2), (3, 4, 5)):
                x, y = (np.stack([s.field(c) for c in grp]) for s in (m, alone))
                assert np.linalg.norm(x - y) <= 1e-4 * np.linalg.norm(y)
        alone.close()
    ens.close()


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-11), ("mixed", 1e-4)])
@pytest.mark.parametrize("over", [dict(filter_strides=[1, 2]), dict(filter_passes=2, filter_compensate=0, filter_stride=5),
                                  dict(filter_strides=[1, 2, 3], filter_passes=2, filter_gather=0)],
                         ids=["S12", "stride5", "S123-J"])
def test_strided_filters(precision, tol, over):
    from paper_1009_2727_gb300.pic import Ensemble, Simulation
    ws = []
    for nx, nz in ((120, 256), (144, 320)):
        w = W.shrink(W.stage_2d(5.0), nx, nz)
        w.update(precision=precision, pml_cells=6, **over)
        strides = w.get("filter_strides") or [w["filter_stride"]]
        halo = (w["filter_passes"] + w["filter_compensate"]) * sum(strides)
        dz = (1.0 + np.sqrt(1 - 1 / 25.0)) * 5.0 * w["dz_lab"]
        ant = 6 + 3 + halo + 5
        w["laser"].update(z_antenna=ant * dz, t_peak=4e-15)
        w["plasma"].update(ppc_x=2, ppc_z=2, z_start_lab=5.0 * (ant + 4) * dz)
        ws.append(w)
    ens = Ensemble(ws)
    assert ens.batched
    ens.step(25)
    ens.sync()
    for m, w in zip(ens.members, ws):
        alone = Simulation(w)
        alone.step(25)
        alone.sync()
        for grp in ((0, 1, 2), (3, 4, 5)):
            x, y = (np.stack([s.field(c) for c in grp]) for s in (m, alone))
            assert np.abs(y).max() > 0 and np.linalg.norm(x - y) <= tol * np.linalg.norm(y)
        alone.close()
    ens.close()
