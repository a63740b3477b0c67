"""The solver switches can be taken back, and one that does not concern a pass
leaves its route alone."""
import numpy as np
import pytest

import workloads as W
from oracle import pw

pytestmark = pytest.mark.gpu

gw = pytest.importorskip("paper_1408_3036_gb300")


@pytest.fixture(scope="module")
def cell():
    from paper_1408_3036_gb300 import _build
    _build.build()
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = W.tiny().cells[0]
    gs = pw.ground_state_dense(pw.Sphere(c.L, c.N, c.ecut), c.vloc, c.n_occ)
    k = gw.Cell(c.L, c.N, c.ecut, c.vloc)
    k.set_occupied(gs.C, gs.eps)
    yield k
    k.close()


def apply(cell, om, prec=gw.GW_MIXED, nb=1):
    return cell.apply_chi0(W.random_fields(9, nb, cell.N ** 3), [om], prec)


def replays(cell, **kw):
    apply(cell, 0.3 + 0.1j, **kw)
    return cell.stats()["graph_replays"]


def test_graphs_can_be_taken_back(cell):
    before = apply(cell, 0.3 + 0.1j)
    assert cell.stats()["graph_replays"] == 0
    cell.set_graphs(1)
    assert replays(cell) > 0
    cell.set_graphs(-1)
    assert np.array_equal(apply(cell, 0.3 + 0.1j), before) and cell.stats()["graph_replays"] == 0


@pytest.mark.parametrize("on", [0, 1])
def test_tensor_cores_concern_wide_mixed_passes_only(cell, on):
    """256 columns or more, mixed: one launch per step; all others keep the column solver."""
    nb = 128 // cell.n_occ + 1                 # two shifts per state and field
    assert replays(cell, nb=nb) == 0
    cell.set_tensor_cores(on)
    assert replays(cell) == 0 and replays(cell, nb=nb, prec=gw.GW_FP64) == 0
    assert replays(cell, nb=nb) > 0
    cell.set_tensor_cores(-1)
    assert replays(cell, nb=nb) == 0


def test_wait_limit_without_leaving_the_default(cell):
    apply(cell, 0.0)
    before = cell.stats()["cluster"]
    assert before > 0
    cell.set_cg_kernel(gw.GW_CG_PERSISTENT, 1 << 22)
    apply(cell, 0.0)
    assert cell.stats()["cluster"] == 0
    cell.set_cg_kernel(gw.GW_CG_CLUSTER, 1 << 24)
    apply(cell, 0.0)
    assert cell.stats()["cluster"] == before
