"""What a Sternheimer solve must not depend on, whatever route it takes."""
import numpy as np
import pytest

import workloads as W
from oracle import pw, response
from tests.conftest import rel

pytestmark = pytest.mark.gpu

gw = pytest.importorskip("paper_1408_3036_gb300")


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1408_3036_gb300 import _build
    _build.build()
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.fixture(scope="module")
def system():
    """16^3, 179 plane waves, 6 states: gap 0.052 Ha, |H - E| < 12 Ha."""
    L, N, ecut = 8.0, 16, 4.0
    rng = np.random.default_rng(1604)
    v = W.gaussian_wells(L, N, rng.uniform(0.0, L, size=(3, 3)), -2.0, 1.0)
    gs = pw.ground_state_dense(pw.Sphere(L, N, ecut), v, 6)
    gap = float(gs.eps_all[6] - gs.eps_all[5])
    assert gap > 0.05
    return L, N, ecut, v, gs, gap


def cell_of(system, shift=0.0):
    L, N, ecut, v, gs, _ = system
    c = gw.Cell(L, N, ecut, v + shift)
    c.set_occupied(gs.C_all[:6], gs.eps_all[:6] + shift)
    return c


def omega_of(om, gap):
    return 0.4 * gap if om == "real" else om


# |H - E| < 12 Ha and shifts 0.03 Ha or more from a transition: condition below
# 400.  Two solutions of backward error tol (10 tol where the refinement
# stagnates) differ by less than 2 10 tol 400, so 1e-6 and 1e-8 for 1e-10, 1e-12.
@pytest.mark.parametrize("tol,err", [(1e-10, 1e-6), (1e-12, 1e-8)])
@pytest.mark.parametrize("om", [0.0, "real", 0.3 + 0.1j])
def test_amplitude_of_the_field(system, om, tol, err):
    """chi0 is linear: a small field takes the passes of a large one, and the
    mixed path reaches the same accuracy."""
    c = cell_of(system)
    c.set_solver(tol=tol)
    f = W.random_fields(3, 2, system[1] ** 3)
    om = omega_of(om, system[5])
    one = c.apply_chi0(f, [om], gw.GW_MIXED)
    passes = c.stats()["outer"]
    for s in (1e-12, 1e-16, 1e-20, 1e-30, 1e20):
        assert rel(c.apply_chi0(s * f, [om], gw.GW_MIXED) / s, one) < err
        assert c.stats()["outer"] <= passes + 1
    c.close()


# FP64: backward error 1e-13 (1e-12), condition below 400: 2 1e-12 400
@pytest.mark.parametrize("prec,tol,err", [(gw.GW_FP64, 1e-13, 1e-9), (gw.GW_MIXED, 1e-10, 1e-6),
                                          (gw.GW_MIXED, 1e-12, 1e-8)])
@pytest.mark.parametrize("om", [0.0, "real", 0.3 + 0.1j])
def test_fields_of_different_size_in_one_call(system, om, prec, tol, err):
    """Columns that are real in real space run in pairs, two to a complex
    transform: the large one's rounding errors stay out of the small one."""
    c = cell_of(system)
    c.set_solver(tol=tol)
    om = omega_of(om, system[5])
    f = W.random_fields(4, 3, system[1] ** 3)
    one = c.apply_chi0(f, [om], prec)[0]
    size = np.array([1.0, 1e-6, 1e-18])
    two = c.apply_chi0(f * size[:, None], [om], prec)[0]
    c.close()
    for b in range(3):
        assert rel(two[b] / size[b], one[b]) < err


@pytest.mark.parametrize("d", [1e-4, 1e-6])
def test_fp64_next_to_a_transition(system, d):
    """A real frequency d Ha above the second-lowest transition: one column's
    solution is 1e4 .. 1e6 times its partners'.  Backward error 1e-13 and
    |H - E| < 12 Ha: 2 1e-13 12 / d of that column (and the transition energy
    itself is known to 1e-14 / d)."""
    gs = system[4]
    t = np.sort((gs.eps_all[6:, None] - gs.eps_all[None, :6]).ravel())
    assert np.abs(t[:8] - t[1] - d).min() > 0.9 * d
    c = cell_of(system)
    f = W.random_fields(5, 2, system[1] ** 3)
    a = c.apply_chi0(f, [float(t[1] + d)], gw.GW_FP64)[0]
    c.close()
    for b in range(2):
        assert rel(a[b], np.real(response.chi0_sos(gs, f[b], float(t[1] + d)))) < 4e-12 / d


@pytest.mark.parametrize("im", [0.0, 1e-4])
def test_mixed_next_to_transitions(system, im):
    """Real frequencies all over the spectrum and 1e-3 .. 1e-6 Ha next to its
    transitions: an indefinite column holds a large residual over a flat
    quasi-residual for a while, which must not end its pass.  Five passes suffice (as many as
    the solver of one launch per step takes for these); backward error 1e-10,
    10 times that where the refinement stagnates, |H - E| < 12 Ha."""
    gs = system[4]
    t = np.sort((gs.eps_all[6:, None] - gs.eps_all[None, :6]).ravel())
    rng = np.random.default_rng(5)
    oms = np.concatenate([rng.uniform(0.05, 2.5, 60), t[rng.integers(0, 500, 60)]
                          + rng.choice([-1, 1], 60) * 10 ** rng.uniform(-6, -3, 60)])
    c = cell_of(system)
    f = W.random_fields(3, 2, system[1] ** 3)
    passes = []
    for om in oms:
        w = complex(om, im) if im else float(om)
        a = c.apply_chi0(f, [w], gw.GW_MIXED)[0]
        passes.append(c.stats()["outer"])
        d = max(np.abs(t - om).min(), im)
        for b in range(2):
            ref = response.chi0_sos(gs, f[b], w)
            assert rel(a[b], ref if im else np.real(ref)) < 2 * 10 * 1e-10 * 12 / d
    c.close()
    assert max(passes) <= 5


# Shifting V rounds V - E by up to 10 Ha 2^-53 (FP32 passes: 2^-24, corrected by
# the refinement) and the target by |A| in it: the errors of the solves as above.
@pytest.mark.parametrize("prec,err", [(gw.GW_FP64, 1e-9), (gw.GW_MIXED, 1e-6)])
@pytest.mark.parametrize("om", [0.0, "real", 0.3 + 0.1j, 0.957 + 0.1j, 0.4j])
def test_zero_of_the_potential(system, om, prec, err):
    """V + c with the energies + c is the same system: the same answer in the
    same number of iterations (within a few, for the roundings)."""
    om = omega_of(om, system[5])
    f = W.random_fields(3, 2, system[1] ** 3)
    c = cell_of(system)
    one, its = c.apply_chi0(f, [om], prec), c.stats()["mean_iter"]
    c.close()
    for shift in (-5.0, 1.0, 3.0, 10.0):
        c = cell_of(system, shift)
        two, its2 = c.apply_chi0(f, [om], prec), c.stats()["mean_iter"]
        c.close()
        assert rel(two, one) < err
        assert its2 <= 1.25 * its + 2
