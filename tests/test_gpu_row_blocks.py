"""Blocks of low rows (quad_nodes.cuh) where the bracket of Eq. phi vanishes
inside a piece: the own cell of one channel at the zero-dispersion wavelength,
many spans or a wide channel, so that the blocks reach far up.

Blocks that hold every row of a piece: small phases, a coarse lower limit of
upsilon1, where the rows' weights make the sum.

FP32 kernels against the FP64 path, 5e-6 as for the row nodes (blocks whose
node count followed |phi| of the last row were off by 1.9e-5 to 7.5e-5, with
the rows' count for the blocks by up to 3.6e-5)."""
import numpy as np
import pytest

from paper_2401_18022_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _check(wl, raman):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2401_18022_gb300 import api
    eng = api.Engine(0)
    if raman:
        wl = W.raman(wl)
    ref = eng.eta(wl, precision=1)["eta"]
    np.testing.assert_allclose(eng.eta(wl)["eta"], ref, rtol=5e-6)
    np.testing.assert_allclose(eng.grad(wl)["eta"], ref, rtol=5e-6)


@pytest.mark.parametrize("B,G,spans", [(0.096, 256, 20), (0.15, 256, 34), (0.096, 512, 26), (0.2, 512, 1)])
@pytest.mark.parametrize("raman", [False, True])
def test_bracket_vanishes_in_the_block(B, G, spans, raman):
    wl = W.subset_plan(W.oband(G=G, cell_set=W.CELLS_SCI_XCI), np.array([20]), "one")
    _check(wl.with_(f_THz=np.array([W.thz_from_nm(1310.0)]), B_THz=np.array([B]), n_spans=spans), raman)


@pytest.mark.parametrize("lam_nm,n,G,n_edges", [(1310.13, 3, 33, 41), (1311.19, 1, 16, 113), (1302.46, 1, 16, 17)])
@pytest.mark.parametrize("raman", [False, True])
def test_block_of_every_row(lam_nm, n, G, n_edges, raman):
    wl = W.subset_plan(W.oband(G=G, n_edges=n_edges, cell_set=W.CELLS_SCI_XCI), np.arange(n), "narrow")
    f = W.thz_from_nm(lam_nm) + 0.032 * 1.04 * np.arange(n)
    _check(wl.with_(f_THz=f, B_THz=np.full(n, 0.032), eps_v1=1e-3), raman)
