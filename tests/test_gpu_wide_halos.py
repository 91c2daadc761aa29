"""The two-pass wide filters' forms by the halo's remainder modulo four (each has its own first and last blocks), in both
precisions, from the smallest halo they take (8 cells; narrower strided ones go to the tile kernels) to the widest, against
the FP64 oracle: 1e-10 in FP64, 1e-3 in mixed precision, as the other parity tests."""
import numpy as np
import pytest

from paper_1009_2727_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FILTERS = {8: dict(filter_passes=8), 9: dict(filter_passes=9), 10: dict(filter_passes=5, filter_stride=2),
           11: dict(filter_passes=11), 25: dict(filter_passes=5, filter_stride=5), 28: dict(filter_passes=4, filter_strides=[1, 2, 4]),
           35: dict(filter_passes=4, filter_compensate=1, filter_strides=[1, 2, 4]), 40: dict(filter_passes=8, filter_stride=5)}


def error(halo, precision, nx, nz):
    import oracle
    from paper_1009_2727_gb300.pic import Simulation
    w = W.shrink(W.stage_2d(5.0), nx, nz)
    w.update(dict(filter_compensate=0), precision=precision, pml_cells=6, **FILTERS[halo])
    strides = w.get("filter_strides") or [w["filter_stride"]]
    assert halo == (w["filter_passes"] + w["filter_compensate"]) * sum(strides)
    dz = (1.0 + np.sqrt(1 - 1 / 25.0)) * 5.0 * w["dz_lab"]
    ant = 6 + 3 + halo + 5
    w["laser"].update(z_antenna=ant * dz, t_peak=4e-15)
    w["plasma"].update(ppc_x=2, ppc_z=2, z_start_lab=5.0 * (ant + 4) * dz)
    g, o = Simulation(w), oracle.Sim(w)
    g.step(30)
    o.step(30)
    g.sync()
    err = max(np.linalg.norm(a - b) / np.linalg.norm(b)
              for a, b in ((np.stack([s.field(c) for c in grp]) for s in (g, o)) for grp in ((0, 1, 2), (3, 4, 5))))
    g.close()
    return err


@pytest.mark.parametrize("halo", [8, 9, 10, 11, 25, 28])
def test_fp64(halo):
    assert error(halo, "fp64", 130, 259) <= 1e-10


@pytest.mark.parametrize("halo", [8, 9, 10, 11, 25, 28, 35, 40])
def test_mixed(halo):
    assert error(halo, "mixed", 133, 301) <= 1e-3
