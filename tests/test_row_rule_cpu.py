"""The node counts that ship (gauss_need, block_need of quad_nodes.cuh) against
the sum over every grid point, in 64 bits: Sigma within 1e-7, below the FP32
rounding of the z-sums (2e-7).  A single fast row may be off by more (the count
was fitted to what a row weighs: |S|^2 falls as 1/phi^2); Sigma may not."""
import numpy as np
import pytest

import _row_rule as rr
from paper_2401_18022_gb300 import workloads as W


@pytest.fixture(scope="module")
def counts(tmp_path_factory):
    return rr.shipped_counts(str(tmp_path_factory.mktemp("counts")))


def off(wl, cut, counts):
    ps = list(rr.Fibre(wl).pieces(cut))
    ref = sum(p.full() for p in ps)
    return abs(sum(p.sigma(*counts) for p in ps) / ref - 1.0)


def narrow(lam_nm, n, B, **kw):
    wl = W.subset_plan(W.oband(G=kw.pop("G"), n_edges=kw.pop("n_edges", 41)), np.arange(n), "narrow")
    f = W.thz_from_nm(lam_nm) + 1.04 * B * np.arange(n)
    return wl.with_(f_THz=f, B_THz=np.full(n, B), **{"cell_set": W.CELLS_SCI_XCI, **kw})


@pytest.mark.parametrize("spans", [1, 10, 100])
def test_tiny(counts, spans):
    assert off(W.tiny(G=64, n_edges=57, cell_set=W.CELLS_SCI_XCI).with_(n_spans=spans), 2, counts) < 1e-7


@pytest.mark.parametrize("spans", [1, 10])
def test_uwb_slots_at_zero_dispersion(counts, spans):
    idx = np.array([0, 294, 480, 497, 498, 499, 520, 588])
    assert off(W.subset_plan(W.uwb(G=48, n_edges=41), idx, "slots").with_(n_spans=spans), 4, counts) < 1e-7


@pytest.mark.parametrize("B,G,spans", [(0.096, 256, 20), (0.15, 256, 34), (0.2, 300, 1), (0.032, 200, 1), (0.3, 100, 5)])
def test_own_cell_at_zero_dispersion(counts, B, G, spans):
    """Blocks reach far up, and the bracket of phi vanishes in them."""
    assert off(narrow(1310.0, 1, B, G=G, n_spans=spans), 0, counts) < 1e-7


@pytest.mark.parametrize("lam_nm,n,G,eps", [(1310.13, 3, 33, 1e-3), (1311.19, 1, 16, 1e-3), (1302.46, 1, 16, 1e-3),
                                            (1308.62, 2, 16, 0.05), (1313.4, 1, 200, 1e-3)])
def test_block_of_every_row(counts, lam_nm, n, G, eps):
    assert off(narrow(lam_nm, n, 0.032, G=G, eps_v1=eps), 0, counts) < 1e-7


@pytest.mark.parametrize("G,spans,eps", [(33, 1, 1e-10), (64, 20, 1e-6), (48, 3, 1e-3)])
def test_every_cell(counts, G, spans, eps):
    wl = narrow(1310.3, 3, 0.096, G=G, n_spans=spans, eps_v1=eps, cell_set=W.CELLS_ALL)
    assert off(wl, 1, counts) < 1e-7


@pytest.mark.parametrize("need", [lambda c, A, D: c[0](A, D), lambda c, A, D: c[1](A, D, 0)])
def test_counts_grow(counts, need):
    """Monotone in the swing and in the length; 4096 (every point) past any rule, also for an infinite swing."""
    for D in (0.0, 0.3, 3.0, 11.5):
        n = [need(counts, A, D) for A in (0.0, 0.05, 0.3, 1.0, 10.0, 100.0, 1e4, np.inf)]
        assert n == sorted(n) and n[0] >= 2 and n[-2:] == [4096, 4096]
    n = [need(counts, 1.0, D) for D in (0.0, 0.5, 2.0, 8.0)]
    assert n == sorted(n)
