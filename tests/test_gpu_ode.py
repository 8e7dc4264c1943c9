"""The Raman ODE and its adjoint at the sizes where their layout changes: one
warp, a warp's edge, several blocks to a cluster, more warps than blocks.

Against the FP64 oracle (the ODE, through the SNR of the plain FP64 path: rtol
1e-9, the same RK4 steps with sums in another order) and against central
differences of the FP64 path (the adjoint; 1e-3 as for every gradient here)."""
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


def _plan(n, df_max=15.0, photon=1, **kw):
    idx = np.sort(np.random.default_rng(n).choice(589, size=n, replace=False))
    wl = W.subset_plan(W.uwb(G=4, n_edges=6, p_dbm=3.0), idx, f"uwb-{n}")
    return W.raman(wl, raman_max_THz=df_max, photon=photon, **kw)


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 65, 97, 160, 257])
@pytest.mark.parametrize("df_max,photon", [(15.0, 1), (-1.0, 0)])
def test_ode_sizes(eng, orc, n, df_max, photon):
    wl = _plan(n, df_max, photon, ode_h_km=2.0)
    cuts = sorted({0, n // 2, n - 1})
    ref = orc.sigma(wl, cuts=cuts)
    np.testing.assert_allclose(eng.eta(wl, cuts=cuts, precision=1)["sigma"], ref, rtol=1e-9)


def test_ode_widest_plan(eng, orc):
    """2,048 channels: 64 warps, four to a block."""
    f = 190.0 + 0.01 * np.arange(2048)
    lam = W.nm_from_thz(f)
    wl = W._plan("wide", f, np.full(2048, 0.009), W.dbm_to_w(np.full(2048, -6.0)),
                 np.full(2048, 0.05), lam, W.aeff_model_um2(lam), W.band_nf_db(lam), n2_m2_per_W=2.6e-20,
                 gamma_fixed=1.3, L_km=80.0, f_ref_THz=200.0, D_ref=17.0, S_ref=0.057, Sdot_ref=0.0, Cr=0.028,
                 alpha_R_per_km=0.05, G=2, n_edges=4, cell_set=0)
    wl = W.raman(wl, ode_h_km=10.0, aeff_scaling=False)
    ref = orc.sigma(wl, cuts=[0, 1000, 2047])
    np.testing.assert_allclose(eng.eta(wl, cuts=[0, 1000, 2047], precision=1)["sigma"], ref, rtol=1e-9)


@pytest.mark.parametrize("n,photon", [(2, 1), (33, 0), (65, 1), (130, 1)])
def test_adjoint_sizes(eng, n, photon):
    wl = _plan(n, photon=photon)
    g = eng.grad(wl)["dT_dP"]
    for j in sorted({0, n // 2, n - 1}):
        h = 1e-4 * np.log(10.0) / 10.0
        P = [wl.P_W.copy(), wl.P_W.copy()]
        P[0][j] *= np.exp(h)
        P[1][j] *= np.exp(-h)
        T = [eng.snr(wl, P=p, precision=1)["T"] for p in P]
        fd = (T[0] - T[1]) / (P[0][j] - P[1][j])
        assert abs(g[j] - fd) <= 1e-3 * max(abs(fd), 1e-3 * np.abs(g).max())
