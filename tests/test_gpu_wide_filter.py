"""The two-pass wide filters (strides, stride sets, more than six passes) in whole steps against the FP64 oracle: grids
at the edges of the passes' blocks (64 rows, 256 columns), the widest halo, a filter of the current alone (with the
rigid ions' column current and without), of the gathered fields alone, both precisions.

FP64 bound 1e-10 as in the other parity tests (sums of at most 81 terms in FP64 over 30 steps); mixed path 1e-3 on E and
B, the path's stated target."""
import numpy as np
import pytest

from paper_1009_2727_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def run(nx, nz, steps, precision="fp64", ppc=2, **over):
    import oracle
    from paper_1009_2727_gb300.pic import Simulation
    w = W.shrink(W.stage_2d(5.0), nx, nz)
    w.update(precision=precision, **over)
    strides = w.get("filter_strides") or [w["filter_stride"]]
    halo = (w["filter_passes"] + w["filter_compensate"]) * sum(strides)
    dz = (1.0 + np.sqrt(1 - 1 / 25.0)) * 5.0 * w["dz_lab"]
    w["pml_cells"] = 6
    ant = 6 + 3 + halo + 5
    w["laser"].update(z_antenna=ant * dz, t_peak=4e-15)
    w["plasma"].update(ppc_x=ppc, ppc_z=ppc, z_start_lab=5.0 * (ant + 4) * dz)
    g, o = Simulation(w), oracle.Sim(w)
    g.step(steps)
    o.step(steps)
    g.sync()
    err = max(np.linalg.norm(a - b) / np.linalg.norm(b)
              for a, b in ((np.stack([s.field(c) for c in grp]) for s in (g, o)) for grp in ((0, 1, 2), (3, 4, 5))))
    g.close()
    return err


@pytest.mark.parametrize("nx,nz,over", [
    (127, 255, dict(filter_strides=[1, 2, 4])), (128, 256, dict(filter_strides=[1, 2, 3], filter_passes=3)),
    (129, 257, dict(filter_strides=[1, 2], filter_gather=0)), (112, 511, dict(filter_passes=7, filter_J=0)),
    (130, 300, dict(filter_passes=1, filter_compensate=0, filter_stride=3)),
    (191, 320, dict(filter_passes=7, filter_compensate=0, filter_stride=5)),
    (100, 260, dict(filter_passes=2, filter_stride=2, filter_J=1, filter_gather=0))])
def test_wide_filter_fp64(nx, nz, over):
    assert run(nx, nz, 30, **over) <= 1e-10


@pytest.mark.parametrize("ppc", [2, 3])
def test_wide_filter_mixed(ppc):
    # three particles per cell: the ions are a column current, added as the x pass reads J_z
    assert run(140, 300, 30, precision="mixed", ppc=ppc, filter_strides=[1, 2, 3]) <= 1e-3
