"""The column solver on spheres that nearly fill their grids (or are as large as
its clusters hold), with a rough potential, so that every input and output of
every radix counts; vectors in shared and in global memory for each kind of
solve, one thread per entry and per component, projector rows in groups of 1, 2,
4, 5 and 6.  Against the solvers of one launch per step.

Spheres: wells 6 to 8 Ha deep, |H - E| < 40 Ha and 0.2 Ha or more to the nearest
transition: condition below 200, states converged to 1e-11.  Two solutions of
backward error 1e-13 (1e-10 mixed), ten times that where the refinement
stagnates, differ by less than 2 10 1e-13 200 + 1e-11 / 0.2: 1e-9 and, mixed,
1e-6.  Rows: as the other tests of this solver (gaps above 0.01 Ha)."""
import numpy as np
import pytest

import workloads as W
from oracle import pw
from tests.conftest import rel

pytestmark = pytest.mark.gpu

gw = pytest.importorskip("paper_1408_3036_gb300")

TOL = {gw.GW_FP64: 1e-9, gw.GW_MIXED: 1e-6}
# radii (grid indices) that a cluster of 16 still holds; elsewhere 0.93 of the largest
LARGEST = {gw.GW_FP64: {45: 18.5, 48: 18.5, 50: 18, 54: 17.5, 60: 16.5, 64: 15.5, 72: 13.5, 80: 13},
           gw.GW_MIXED: {48: 21, 50: 22, 54: 22, 60: 22, 64: 22, 72: 21.5, 80: 21}}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1408_3036_gb300 import _build
    _build.build()
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def both(k, gap, prec):
    f = W.random_fields(k.N, 1, k.ng)
    oms = (0.0, 0.4 * gap, 0.3 + 0.1j)
    one = []
    for om in oms:
        one.append(k.apply_chi0(f, [om], prec))
        st = k.stats()
        assert st["cluster"] > 0 and st["graph_replays"] == 0       # the column solver ran
    k.set_cg_kernel(gw.GW_CG_MULTI_LAUNCH)
    k.set_graphs(1)
    for om, a in zip(oms, one):
        assert rel(a, k.apply_chi0(f, [om], prec)) < TOL[prec]
        assert om == 0.0 or k.stats()["graph_replays"] > 0
    k.close()


@pytest.mark.parametrize("prec", [gw.GW_FP64, gw.GW_MIXED])
@pytest.mark.parametrize("N", [12, 15, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 80])
def test_spheres_that_fill_the_grid(N, prec):
    from paper_1408_3036_gb300.groundstate import lowest_states
    most = (N - 1) // 2
    radius = LARGEST[prec].get(N, most if N < 20 else 0.93 * most)
    L = 0.5 * N
    ecut = 0.5 * (2.0 * np.pi * (radius + 1e-6) / L) ** 2
    rng = np.random.default_rng(N)
    v = np.clip(0.3 * rng.standard_normal(N ** 3), -1.0, 1.0)
    for depth in (-8.0, -7.0, -6.0):
        v += W.gaussian_wells(L, N, rng.uniform(0.0, L, size=(1, 3)), depth, 0.8).reshape(-1)
    k = gw.Cell(L, N, ecut, v)
    eps, psi, res = lowest_states(k, 3, tol=1e-11)
    n = 1 + int(np.argmax(np.diff(eps)))
    gap = float(eps[n] - eps[n - 1])
    assert res < 1e-11 and gap > 0.35
    k.set_occupied(psi[:n], eps[:n])
    both(k, gap, prec)


@pytest.mark.parametrize("prec", [gw.GW_FP64, gw.GW_MIXED])
@pytest.mark.parametrize("nocc", [1, 5, 70, 85, 97])
def test_rows_in_groups(nocc, prec):
    N, L = 20, 10.0
    rng = np.random.default_rng(nocc)
    v = W.gaussian_wells(L, N, rng.uniform(0.0, L, size=(3, 3)), -2.0, 1.0)
    gs = pw.ground_state_dense(pw.Sphere(L, N, 5.0), v, nocc + 3)
    gaps = gs.eps_all[nocc:nocc + 4] - gs.eps_all[nocc - 1:nocc + 3]
    n = nocc + int(np.argmax(gaps))
    assert gaps.max() > 0.01
    k = gw.Cell(L, N, 5.0, v)
    k.set_occupied(gs.C_all[:n], gs.eps_all[:n])
    both(k, float(gaps.max()), prec)
