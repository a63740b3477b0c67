"""The column solver (one thread-block cluster per pair of real columns or per
complex column, the default route of the Sternheimer passes) against the
multi-launch solvers, over every pair of radices it has, odd numbers of columns
and states, one column up to more than the clusters that run at once, and
projectors of one to many rows per warp.

Both routes meet the same FP64 backward error (1e-13, mixed 1e-10), so their
results differ by at most about twice that times the condition number: the gap
of these cells is above 0.01 Ha, the real frequency 0.4 of it (so every shift is
0.006 Ha or more from a transition), and |H - E| < 12 Ha, hence below 2e3:
1e-9 in FP64 and 1e-6 for the mixed path."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

gw = pytest.importorskip("paper_1408_3036_gb300")

TOL = {0: 1e-9, 1: 1e-6}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1408_3036_gb300 import _build
    _build.build()
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


def cell_of(N, L, ecut, nocc):
    from oracle import pw
    rng = np.random.default_rng(100 * N + nocc)
    v = W.gaussian_wells(L, N, rng.uniform(0.0, L, size=(3, 3)), -2.0, 1.0)
    gs = pw.ground_state_dense(pw.Sphere(L, N, ecut), v, nocc + 3)
    gaps = gs.eps_all[nocc:nocc + 4] - gs.eps_all[nocc - 1:nocc + 3]
    n = nocc + int(np.argmax(gaps))
    assert gaps.max() > 0.01
    c = gw.Cell(L, N, ecut, v)
    c.set_occupied(gs.C_all[:n], gs.eps_all[:n])
    return c, float(gaps.max())


def both_routes(c, gap, f, om, prec):
    om = 0.4 * gap if om == "real" else om
    one = c.apply_chi0(f, [om], prec)
    assert c.stats()["launch_ctas"] > 0 and c.stats()["graph_replays"] == 0
    c.set_cg_kernel(gw.GW_CG_MULTI_LAUNCH)
    c.set_graphs(0)
    return one, c.apply_chi0(f, [om], prec)


# (12 = 3 4) .. (80 = 8 10): every first radix 3 4 5 6 8 and second 4 5 6 8 9 10
@pytest.mark.parametrize("N", [12, 15, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 80])
@pytest.mark.parametrize("om", [0.0, "real", 0.3 + 0.1j])
def test_grid_sizes(N, om):
    f = W.random_fields(5, 1, N ** 3)
    for prec in (gw.GW_FP64, gw.GW_MIXED):
        c, gap = cell_of(N, 6.0, 3.0, 3)
        a, b = both_routes(c, gap, f, om, prec)
        c.close()
        assert rel(a, b) < TOL[prec]


@pytest.mark.parametrize("nocc,nb", [(1, 1), (1, 3), (5, 7), (17, 2), (33, 3), (66, 5)])
@pytest.mark.parametrize("om", [0.0, "real", 0.3 + 0.1j])
def test_columns_and_rows(nocc, nb, om):
    for prec in (gw.GW_FP64, gw.GW_MIXED):
        c, gap = cell_of(20, 8.0, 4.0, nocc)
        f = W.random_fields(6, nb, 20 ** 3)
        a, b = both_routes(c, gap, f, om, prec)
        c.close()
        assert rel(a, b) < TOL[prec]


def test_full_sphere_and_complex_fields():
    """A sphere that fills the grid (2 max|n| = N - 1, every plane present) and
    complex fields at a real and a complex frequency."""
    L, N = 10.0, 15
    ecut = 0.5 * (2.0 * np.pi * 7.4 / L) ** 2
    for om in ("real", 0.3 + 0.1j):
        c, gap = cell_of(N, L, ecut, 4)
        f = W.random_fields(7, 2, N ** 3, complex_=True)
        a, b = both_routes(c, gap, f, om, gw.GW_FP64)
        c.close()
        assert rel(a, b) < TOL[0]


@pytest.mark.parametrize("om", [0.957 + 0.1j, -0.957 - 0.1j, 0.05 - 0.02j, 3.0 + 0.5j, 0.5j])
def test_preconditioner_of_the_shift(om):
    """Denominators around zero (real parts inside the kinetic spectrum, either
    sign of the imaginary part) against the solver without a preconditioner:
    |Im| >= 0.02 and |H - E| < 15 Ha keep the condition number below 2e3.  A
    single-precision pass ends with its columns, not with the 1000 iterations
    of the stagnation window."""
    for prec in (gw.GW_FP64, gw.GW_MIXED):
        c, _ = cell_of(20, 8.0, 4.0, 5)
        f = W.random_fields(8, 4, 20 ** 3, complex_=True)
        a = c.apply_chi0(f, [om], prec)
        assert c.stats()["max_iter"] < 900
        c.set_precond(0)
        b = c.apply_chi0(f, [om], prec)
        c.close()
        assert rel(a, b) < TOL[prec]
