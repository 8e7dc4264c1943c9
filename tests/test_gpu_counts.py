"""Counts of grid points by phase and of z-sums by form (isrs_last_path_counts,
isrs_last_node_counts) against a count over the grid in 64 bits.

A run of a row counts by its first node, so the share of a class is off by the
runs that cross its border: 5 % of the points; their total by points at a
channel's edge: 1e-3.  Nodes: those of the rule in 64 bits, where a swing at
the step from one rule to the next may round the other way: 2 % (no Raman slope,
which the rule counts as a swing too)."""
import numpy as np
import pytest

import _row_rule as rr
from paper_2401_18022_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eng():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2401_18022_gb300 import api
    return api.Engine(0)


def by_phase(wl, phi):
    """[low, direct, telescoped] points; the longest step decides the form."""
    fib = rr.Fibre(wl)
    low = phi * wl.L_km * wl.n_spans <= 6.0
    direct = phi * fib.dz.max() <= np.pi
    return np.array([low.sum(), (direct & ~low).sum(), (~direct & ~low).sum()])


def check(got, want):
    got = np.array([got[k] for k in ("small", "direct", "telescoped")])
    assert abs(got.sum() / want.sum() - 1.0) < 1e-3
    assert np.abs(got - want).max() < 0.05 * want.sum()


@pytest.mark.parametrize("spans,n_edges", [(1, 33), (10, 33), (1, 2), (3, 3)])
def test_points_and_nodes(eng, spans, n_edges, tmp_path):
    wl = W.tiny(G=40, n_edges=n_edges, cell_set=W.CELLS_SCI_XCI).with_(n_spans=spans, Cr=0.0)
    ps = [p for i in range(wl.n_ch) for p in rr.Fibre(wl).pieces(i)]
    want = by_phase(wl, np.concatenate([p.points() for p in ps]))
    counts = rr.shipped_counts(str(tmp_path))
    for p in ps:
        p.sigma(*counts)
    nodes = sum(p.nodes for p in ps)
    for call in (lambda: eng.eta(wl), lambda: eng.grad(wl), lambda: eng.eta(W.raman(wl))):
        call()
        check(eng.last_path_counts(), want)
        assert abs(sum(eng.last_node_counts().values()) / nodes - 1.0) < 0.02


@pytest.mark.parametrize("spans", [1, 10])
def test_gradient_with_mci_cells(eng, spans):
    """Every MCI point is a z-sum of its own."""
    wl = W.tiny(G=40, n_edges=33).with_(G_mci=12, n_spans=spans)
    every = W.tiny(G=12, n_edges=33).with_(n_spans=spans)                # all cells on the MCI grid
    own = every.with_(cell_set=W.CELLS_SCI_XCI)
    phi = [np.concatenate([p.points() for i in range(wl.n_ch) for p in rr.Fibre(w).pieces(i)])
           for w in (wl.with_(cell_set=W.CELLS_SCI_XCI), every, own)]
    mci = by_phase(wl, phi[1]) - by_phase(wl, phi[2])
    eng.grad(wl)
    got = eng.last_path_counts()
    check(got, by_phase(wl, phi[0]) + mci)
    nodes = sum(eng.last_node_counts().values())
    eng.grad(wl.with_(cell_set=W.CELLS_SCI_XCI, G_mci=0))
    assert abs(nodes - sum(eng.last_node_counts().values()) - mci.sum()) < 0.01 * mci.sum()
