"""Error of the FP32 sums against the FP64 path where small phases make them: all
terms add up, so what the special-function unit cuts off would show (2.5e-7 of
|S|^2).  The nodes are raised by its mean; the rounding of the rest is below
1.5e-7 (2-norm over the channels, mean of four launch profiles)."""
import numpy as np
import pytest

from paper_2401_18022_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _band65():
    wl = W.subset_plan(W.uwb(G=64, n_edges=97), np.arange(300, 365), "band")
    return wl.with_(n_spans=3)


@pytest.mark.parametrize("plan", [lambda: W.tiny(G=64), lambda: W.tiny(G=16), _band65], ids=["G64", "G16", "band65"])
@pytest.mark.parametrize("kind", ["closed", "raman", "closed_grad", "raman_grad"])
def test_error_against_fp64(plan, kind):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2401_18022_gb300 import api
    eng, wl = api.Engine(0), plan()
    if kind.startswith("raman"):
        wl = W.raman(wl)
    call = eng.grad if kind.endswith("grad") else eng.eta
    err = []
    for seed in range(4):
        P = W.dbm_to_w(np.random.default_rng(seed).normal(1.0, 1.5, wl.n_ch))
        ref = eng.eta(wl, P, precision=1)["eta"]
        err.append(np.linalg.norm(call(wl, P)["eta"] - ref) / np.linalg.norm(ref))
    assert np.mean(err) < 1.5e-7
