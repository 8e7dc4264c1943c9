"""Which problems the allocation-free call takes: 80 bytes a piece, 24 a tile of
2^20 grid points, 392 a z-step, 76 a channel against 4 MiB, whatever the tables
of the kernels need.  n channels have n (2 n + 1) SCI and XCI pieces."""
import ctypes

import numpy as np
import pytest

from paper_2401_18022_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,G,n_edges,taken", [
    (141, 1024, 3, True),      # 39,903 pieces, each a tile of its own: 4.17 MB (of 4.19)
    (142, 1024, 3, False),     # 40,470 pieces: 4.22 MB
    (141, 640, 3, True),       # two pieces to a tile: 3.70 MB
    (149, 16, 2049, False),    # 44,551 pieces and 2,048 steps: 4.39 MB
    (149, 16, 1025, True),     # 3.99 MB
    (100, 64, 113, True)])
def test_limit(n, G, n_edges, taken):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2401_18022_gb300 import _capi, api
    eng, lib = api.Engine(0), _capi.load()
    wl = W.subset_plan(W.uwb(G=G, n_edges=n_edges), np.arange(200, 200 + n), "block")
    fb, (ch, keep), q = eng.fibre(wl), eng.channels(wl), eng.quad(wl, 0)
    P = torch.tensor(wl.P_W, dtype=torch.float64, device="cuda")
    eta = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
    fn = lib.isrs_gn_eta_noalloc
    fn.argtypes = [ctypes.POINTER(_capi.Fibre), ctypes.POINTER(_capi.Channels), ctypes.c_void_p,
                   ctypes.POINTER(_capi.Quad), ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p]
    rc = fn(ctypes.byref(fb), ctypes.byref(ch), ctypes.c_void_p(P.data_ptr()), ctypes.byref(q),
            ctypes.c_void_p(eta.data_ptr()), None, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    torch.cuda.synchronize()
    assert rc == (0 if taken else 6)
    if taken:
        np.testing.assert_allclose(eta.cpu().numpy(), eng.eta(wl, P)["eta"].cpu().numpy(), rtol=1e-6)
