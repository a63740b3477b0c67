"""The FP64 projector and residual on half the sphere (kernels_half.cu) against
the oracle's sums over the whole one, through the model operator (two
projections, no solve) and one static application (the residual): tiles of 4
rows and 4 or 2 columns with every remainder, one to many chunks of entries,
real and complex columns, and imaginary frequencies, where a real field takes
one solve for both signs.

The model operator is FP64 arithmetic only: 1e-12 of the largest value, as the
other tests of it; the static and imaginary ones solve to 1e-13 (condition
below 2e3: 1e-9)."""
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


def cell_of(N, L, ecut, nocc):
    rng = np.random.default_rng(7 * N + nocc)
    v = W.gaussian_wells(L, N, rng.uniform(0.0, L, size=(3, 3)), -2.0, 1.0)
    sph = pw.Sphere(L, N, ecut)
    gs = pw.ground_state_dense(sph, v, nocc)
    gaps = gs.eps_all[nocc:nocc + 4] - gs.eps_all[nocc - 1:nocc + 3]
    n = nocc + int(np.argmax(gaps))
    gs = pw.ground_state_dense(sph, v, n)
    c = gw.Cell(L, N, ecut, v)
    c.set_occupied(gs.C, gs.eps)
    return c, gs


@pytest.mark.parametrize("N,L,ecut,nocc,nb", [(12, 6.0, 3.0, 1, 1), (15, 7.0, 3.0, 4, 3), (18, 6.0, 3.0, 5, 2),
                                              (20, 9.0, 4.5, 17, 5), (96, 5.0, 3.0, 6, 1), (20, 9.0, 4.5, 34, 1)])
def test_against_the_oracle(N, L, ecut, nocc, nb):
    c, gs = cell_of(N, L, ecut, nocc)
    f = W.random_fields(11, nb, gs.sph.ng)
    c.set_operator(gw.GW_OP_MODEL)
    for om in (0.0, 0.15, 0.2 + 0.1j, 0.3j):
        dn = c.apply_chi0(f, [om], gw.GW_FP64)[0]
        for b in range(nb):
            ref = response.chi0_model(gs, f[b], om)
            assert rel(dn[b], ref if np.iscomplexobj(dn) else ref.real) < 1e-12
    c.set_operator(gw.GW_OP_STERNHEIMER)
    for om in (0.0, 0.3j):
        dn = c.apply_chi0(f, [om], gw.GW_FP64)[0]
        for b in range(nb):
            ref = response.chi0_sos(gs, f[b], om)
            assert rel(dn[b], ref if np.iscomplexobj(dn) else np.real(ref)) < 1e-9
    c.close()
