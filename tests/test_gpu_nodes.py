"""Row sums from nodes (quad_nodes.cuh) at the sizes where they can go wrong:
runs shorter than any rule, just past one, longer than the longest table, rows
in several batches and chunks, rows that turn, many candidates, many spans.

Against the FP64 oracle.  Tolerance 5e-6: the nodes are located to ~3e-7 of a
piece's sum, the rules truncate below 2e-8 and the FP32 z-sums carry ~1e-6."""
import numpy as np
import pytest

from paper_2401_18022_gb300 import workloads as W

pytestmark = pytest.mark.gpu

RTOL = 5e-6


@pytest.fixture(scope="module")
def eng():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2401_18022_gb300 import api
    e = api.Engine(0)
    yield e
    e.set_tile(0, 0)


def _one(G, **kw):
    """Two channels: 7 pieces a CUT, so that large grids stay quick on the CPU."""
    return W.subset_plan(W.tiny(G=G, **kw), np.array([0, 2]), "two")


@pytest.mark.parametrize("G", [1, 2, 3, 4, 5, 8, 13, 47, 48, 49, 96, 97, 255, 256, 257, 300, 513])
def test_grid_sizes(eng, orc, G):
    wl = _one(G, n_edges=9 if G > 100 else 33)
    np.testing.assert_allclose(eng.eta(wl)["sigma"], orc.sigma(wl), rtol=RTOL)


@pytest.mark.parametrize("threads", [32, 96, 256])
@pytest.mark.parametrize("G", [40, 300])
def test_rows_in_batches(eng, orc, threads, G):
    wl = _one(G, n_edges=9)
    eng.set_tile(0, threads)
    got = eng.eta(wl)["sigma"]
    eng.set_tile(0, 0)
    np.testing.assert_allclose(got, orc.sigma(wl), rtol=RTOL)


@pytest.mark.parametrize("spans", [3, 40])
def test_many_spans(eng, orc, spans):
    """The array factor widens the band n-fold: more nodes, parts, then every column."""
    wl = W.subset_plan(W.uwb(G=96, n_edges=17), np.array([0, 1, 300, 588]), "four").with_(n_spans=spans)
    np.testing.assert_allclose(eng.eta(wl)["sigma"], orc.sigma(wl), rtol=RTOL * spans)


def test_wide_channel_and_coarse_rows(eng, orc):
    wl = W.tiny(G=50, n_edges=33).with_(f_THz=np.array([193.2, 193.3, 193.5, 193.7, 193.9]),
                                        B_THz=np.array([.03, .03, .3, .03, .03]), eps_v1=1e-3)
    np.testing.assert_allclose(eng.eta(wl)["sigma"], orc.sigma(wl), rtol=RTOL)


def test_far_cells(eng, orc):
    """Cells 59 THz from the CUT, both signs: points located relative to the cell."""
    wl = W.subset_plan(W.uwb(G=64, n_edges=41), np.array([0, 200, 201, 450, 588]), "far")
    np.testing.assert_allclose(eng.eta(wl)["sigma"], orc.sigma(wl), rtol=RTOL)
