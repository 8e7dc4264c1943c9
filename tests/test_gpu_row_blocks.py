"""Blocks of low rows (quad_nodes.cuh) where the bracket of Eq. phi vanishes
inside a piece: the own cell of one channel at the zero-dispersion wavelength,
many spans or a wide channel, so that the blocks reach far up.

FP32 kernels against the FP64 path, 5e-6 as for the row nodes (blocks whose
node count followed |phi| of the last row were off by 1.9e-5 to 7.5e-5)."""
import numpy as np
import pytest

from paper_2401_18022_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,G,spans", [(0.096, 256, 20), (0.15, 256, 34), (0.096, 512, 26), (0.2, 512, 1)])
@pytest.mark.parametrize("raman", [False, True])
def test_bracket_vanishes_in_the_block(B, G, spans, raman):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2401_18022_gb300 import api
    eng = api.Engine(0)
    wl = W.subset_plan(W.oband(G=G, cell_set=W.CELLS_SCI_XCI), np.array([20]), "one")
    wl = wl.with_(f_THz=np.array([W.thz_from_nm(1310.0)]), B_THz=np.array([B]), n_spans=spans)
    if raman:
        wl = W.raman(wl)
    ref = eng.eta(wl, precision=1)["eta"]
    np.testing.assert_allclose(eng.eta(wl)["eta"], ref, rtol=5e-6)
    np.testing.assert_allclose(eng.grad(wl)["eta"], ref, rtol=5e-6)
