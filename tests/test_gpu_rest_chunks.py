"""Chunks of electrons at rest in a field-free window (only their box moves with the frame) against the same run pushed
particle by particle: a field of 1e-25 V/m on every node keeps every window from being field-free and moves nothing
(a kick of 1e-30 m/s against FP32 momenta of 1e5 and more where the laser acts).

Runs in which plasma streams across the whole domain (inflow, sorts at several cadences, exit with ghosts), with and
without a laser, and the lab-frame moving window; powers of two and other particles per cell (no pairs: always pushed).
The two agree to FP32 rounding of the laser-driven part (the deposits' atomics sum in varying order): 1e-4 on the fields,
1e-3 cells on the positions; which electrons are there agrees exactly."""
import numpy as np
import pytest

from paper_1009_2727_gb300 import workloads as W
from paper_1009_2727_gb300 import capi

pytestmark = pytest.mark.gpu


def boosted(ppc, tile_steps, laser):
    w = W.shrink(W.stage_2d(5.0), 96, 256, precision="mixed")
    w["pml_cells"] = 6
    dz = (1.0 + np.sqrt(1 - 1 / 25.0)) * 5.0 * w["dz_lab"]
    w["laser"].update(z_antenna=24 * dz, t_peak=6e-15)
    # the plasma's front enters the domain and has streamed out through -z by the end
    w["plasma"].update(ppc_x=ppc, ppc_z=ppc, z_start_lab=5.0 * 120 * dz, ramp_lab=2e-6)
    if not laser:
        del w["laser"]
    return w, dict(tile=tile_steps[0], sort_every=tile_steps[1]), 260


def window():
    w = W.shrink(W.stage_2d(1.0), 96, 256, precision="mixed")
    dz = w["dz_lab"]
    w.update(pml_cells=6, moving_window=1, window_beta=1.0, gamma_boost=1.0)
    w["laser"].update(z_antenna=200 * dz, t_peak=6e-15)
    w["plasma"].update(ppc_x=2, ppc_z=2, z_start_lab=215 * dz, ramp_lab=2e-6)
    return w, dict(tile=(8, 16), sort_every=16), 260


@pytest.mark.parametrize("case", [
    boosted(1, ((8, 32), 32), True), boosted(2, ((8, 16), 16), True), boosted(4, ((16, 16), 64), True),
    boosted(4, ((8, 8), 8), False), boosted(3, ((8, 32), 32), True), window()],
    ids=["ppc1", "ppc2", "ppc4", "ppc4-dark", "ppc3", "window"])
def test_rest_chunks(case):
    from paper_1009_2727_gb300.pic import Simulation
    w, layout, steps = case
    sims = [Simulation(w, **layout) for _ in range(2)]
    f = np.full(sims[1].shape, 1e-25)
    for c in range(6):
        sims[1].set_field(c, f)
    for s in sims:
        s.step(steps // 2)
        s.sync()
    na, nb = (s.particles(capi.ELECTRONS) for s in sims)
    assert np.array_equal(np.sort(na["id"]), np.sort(nb["id"])) and len(na["id"]) > 0
    for s in sims:
        s.step(steps - steps // 2)
        s.sync()
    pa, pb = (s.particles(capi.ELECTRONS) for s in sims)
    a, b = np.argsort(pa["id"], kind="stable"), np.argsort(pb["id"], kind="stable")
    assert np.array_equal(pa["id"][a], pb["id"][b])
    dz = sims[0].stats()["dz"]
    for k in ("x", "z"):
        assert np.abs(pa[k][a] - pb[k][b]).max(initial=0.0) <= 1e-3 * dz
    if "laser" in w:
        for grp in ((0, 1, 2), (3, 4, 5)):
            x, y = (np.stack([s.field(c) for c in grp]) for s in sims)
            assert np.linalg.norm(x - y) <= 1e-4 * np.linalg.norm(y)
    else:
        assert sims[0].stats()["field_energy"] <= 1e-3   # nothing but FP32 residue of leaving electrons
    for s in sims:
        s.close()
