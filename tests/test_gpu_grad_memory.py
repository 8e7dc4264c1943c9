"""Device memory of a gradient over many pieces: every cell of 250 channels is
5 to 6 million pieces (those with F_c inside the plan; 0.45 GB).  A tile's buckets
take 4 KB: about 39,000 tiles are 0.16 GB of them at most, tiles of 32 pieces
would be 170,000 and 0.7 GB."""
import numpy as np
import pytest

from paper_2401_18022_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_bucket_memory_follows_the_tiles():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2401_18022_gb300 import api
    eng = api.Engine(0)
    wl = W.subset_plan(W.uwb(G=2, n_edges=129, cell_set=W.CELLS_ALL), np.arange(250), "narrow")
    wl = wl.with_(f_THz=190.0 + 0.04 * np.arange(250), B_THz=np.full(250, 0.036))
    eng.grad(wl.with_(G=3, cell_set=W.CELLS_SCI_XCI))          # context, module, the small buffers
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    g = eng.grad(wl)
    torch.cuda.synchronize()
    assert np.all(np.isfinite(g["dT_dP"]))
    grown = free - torch.cuda.mem_get_info()[0]
    assert grown < 0.8e9, grown
    np.testing.assert_allclose(g["eta"], eng.eta(wl)["eta"], rtol=1e-5)
