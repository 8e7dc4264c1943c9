"""The FP64 sums behind the gradient over many tiles: the Raman-ODE row gather
(16 warps to a channel, more than 32 rows to each), the PSD and step buckets
(eight warps to a CUT's tiles, more than 32 channels), the eight-lane tile sums.

Bit for bit reproducible; CUT shards, whose warps take other shares of the rows,
add up to the same gradient but for the order of FP64 sums (1e-11 of the largest
entry: ~1e4 terms of 1e-16 with cancellation of up to 10)."""
import numpy as np
import pytest

from paper_2401_18022_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [33, 70])
@pytest.mark.parametrize("raman", [False, True])
def test_gradient_sums(n, raman):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2401_18022_gb300 import api
    eng = api.Engine(0)
    wl = W.subset_plan(W.uwb(G=12, n_edges=35), np.arange(300, 300 + n), "block").with_(snr_trx_dB=20.0)
    if raman:
        wl = W.raman(wl, ode_h_km=2.0)
    g = eng.grad(wl)
    np.testing.assert_array_equal(eng.grad(wl)["dT_dP"], g["dT_dP"])
    shards = [list(range(0, n, 3)), list(range(1, n, 3)) + list(range(2, n, 3))]
    eta = np.full(n, np.nan)
    engs = [api.Engine(0) for _ in shards]
    for e, cuts in zip(engs, shards):
        eta[cuts] = e.grad_shard_fwd(wl, cuts)
    np.testing.assert_array_equal(eta, g["eta"])
    parts = [e.grad_shard_bwd(eta, with_direct=k == 0)["dT_dP"] for k, e in enumerate(engs)]
    assert np.abs(sum(parts) - g["dT_dP"]).max() < 1e-11 * np.abs(g["dT_dP"]).max()
