"""MCI cells at phases past 2^22 revolutions: the sum at an empty slot (P = 0)
whose only terms are two cells 20 to 60 THz away, at 8.2e6 and 1.5e7 revolutions.

The sign of the dispersion turns phi into -phi and S into its conjugate, so the
sums agree but for FP32 rounding (1e-6); a phase reduction that takes
half-integers for integers on one side of zero does not (9 % at one span).  The
phases themselves are beyond FP32 (0.5 revolutions of rounding), so against FP64
the sum is a sample over ~1,500 points, each as scattered as an exponential
variable at most: 3 %, 20 % allowed."""
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


def plan(D, spans, P0=0.0):
    wl = W.subset_plan(W.tiny(G=4, n_edges=113, cell_set=W.CELLS_ALL), np.arange(4), "far")
    return wl.with_(f_THz=np.array([180.0, 200.0, 220.0, 240.0]), f_ref_THz=210.0, B_THz=np.full(4, 0.096),
                    alpha_per_km=np.full(4, 0.005), alpha_R_per_km=0.005, P_W=np.array([P0, 1e-2, 1e-2, 1e-2]),
                    Cr=0.0, D_ref=D, S_ref=0.0, n_spans=spans, G_mci=32)


@pytest.mark.parametrize("spans", [1, 3, 10])
@pytest.mark.parametrize("raman", [False, True])
def test_empty_slot(eng, spans, raman):
    wl = [plan(D, spans) for D in (34.0, -34.0)]
    if raman:
        wl = [W.raman(w, ode_h_km=2.0) for w in wl]
    got = [eng.eta(w)["sigma"][0] for w in wl]
    assert got[0] > 0.0 and abs(got[0] / got[1] - 1.0) < 1e-6
    if spans == 1:
        assert abs(got[0] / eng.eta(wl[0], precision=1)["sigma"][0] - 1.0) < 0.2


@pytest.mark.parametrize("spans", [1, 3, 10])
def test_adjoint(eng, spans):
    """The adjoint's own forward sum; a power of 1e-22 W leaves only the far cells."""
    got = [eng.grad(plan(D, spans, 1e-22))["eta"][0] for D in (34.0, -34.0)]
    assert got[0] > 0.0 and abs(got[0] / got[1] - 1.0) < 1e-6
