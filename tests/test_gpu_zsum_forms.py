"""The z-sum forms and lists of the quadrature kernels where they can go wrong:
odd and short z-grids (a lone last step, remainders shared by several lanes),
G_mci from 1 to 32 (cells per group, lists that end part full), |phi| on both
sides of the direct / telescoped boundary, plans far from f_ref.

Against the FP64 oracle.  FP64 1e-9.  FP32 SCI/XCI 5e-6 as for the row nodes;
with MCI cells 2e-5: a cell's point carries ~6e-8 |phi| L rad of phase error
(|phi| L < 1e5 here, 6e-3), random over > 100 points of a share below 5%."""
import numpy as np
import pytest

from paper_2401_18022_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eng():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2401_18022_gb300 import api
    return api.Engine(0)


@pytest.mark.parametrize("n_edges", [2, 3, 4, 6, 18, 66, 130])
def test_step_counts(eng, orc, n_edges):
    wl = W.tiny(G=24, n_edges=n_edges)
    np.testing.assert_allclose(eng.eta(wl)["sigma"], orc.sigma(wl), rtol=5e-6)
    np.testing.assert_allclose(eng.eta(wl, precision=1)["sigma"], orc.sigma(wl), rtol=1e-9)


@pytest.mark.parametrize("raman", [False, True])
@pytest.mark.parametrize("g_mci,n_edges", [(1, 34), (2, 9), (3, 34), (5, 33), (8, 2), (12, 18), (16, 33), (31, 9),
                                           (32, 10)])
def test_mci_lists(eng, orc, g_mci, n_edges, raman):
    wl = W.subset_plan(W.uwb(G=16, n_edges=n_edges, cell_set=W.CELLS_ALL),
                       np.array([100, 101, 102, 103, 110, 111, 140]), "seven").with_(G_mci=g_mci)
    if raman:
        wl = W.raman(wl)
    ref = orc.sigma(wl)
    np.testing.assert_allclose(eng.eta(wl)["sigma"], ref, rtol=2e-5)
    np.testing.assert_allclose(eng.eta(wl, precision=1)["sigma"], ref, rtol=1e-9)


@pytest.mark.parametrize("shift", [-40.0, 0.0, 40.0])
def test_plan_far_from_reference(eng, orc, shift):
    """F_c - f_ref of tens of THz: the step rows are taken about the CUT."""
    wl = W.tiny(G=48, n_edges=33)
    wl = wl.with_(f_ref_THz=wl.f_ref_THz + shift)
    np.testing.assert_allclose(eng.eta(wl)["sigma"], orc.sigma(wl), rtol=5e-6)


def test_gradient_sums_split_over_blocks(eng):
    """The Raman-ODE row gather and the eight-lane tile sums: CUT shards and
    one call give the same eta, bit for bit."""
    wl = W.tiny(G=33, n_edges=33)
    a, b = eng.eta(wl)["sigma"], eng.eta(wl, cuts=[3, 1])["sigma"]
    assert a[3] == b[0] and a[1] == b[1]
