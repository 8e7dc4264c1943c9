"""Start of the thread-block clusters of the Raman ODE and its adjoint: a block
may store into another block's shared memory only after that block has started,
so every path to the first such store passes a cluster barrier."""
import os
import re

import numpy as np
import pytest

from paper_2401_18022_gb300 import workloads as W

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2401_18022_gb300", "csrc",
                   "raman.cu")


def _bodies(text):
    """{name: body} of the functions of a source file without its comments."""
    out = {}
    for m in re.finditer(r"(\w+)\s*\([^;{}]*\)\s*\{", text):
        if m.group(1) in ("if", "for", "while", "switch"):
            continue
        depth, k = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[k], 0)
            k += 1
        out[m.group(1)] = text[m.end():k - 1]
    return out


def test_barrier_before_the_first_remote_store():
    text = re.sub(r"//[^\n]*|__launch_bounds__\([^)]*\)", "", open(SRC).read())
    f = _bodies(text)
    stores = re.compile(r"\bode_(rhs|jt|window)\s*\(")
    assert "map_shared_rank" in f["ode_window"] and not stores.search(f["ode_lane"])
    kernels = [k for k in ("k_raman_ode", "k_raman_adj") if "this_cluster" in f[k]]
    assert kernels == ["k_raman_ode", "k_raman_adj"]
    for k in kernels:
        start = re.sub(r"ode_lane\s*\([^;]*;", lambda m: f["ode_lane"], f[k], count=1)
        first = stores.search(start).start()
        assert re.search(r"\bcl\.sync\(\)", start[:first]), k


@pytest.mark.gpu
def test_many_clusters_equal_single_calls():
    """More clusters than the device places at once: each profile of a batch
    equals its own call bit for bit."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2401_18022_gb300 import api
    eng = api.Engine(0)
    idx = np.sort(np.random.default_rng(5).choice(589, size=300, replace=False))
    wl = W.raman(W.subset_plan(W.uwb(G=2, n_edges=9), idx, "uwb-300"), ode_h_km=5.0)
    bw = W.batched(n_prof=64, G=2, n_edges=9)
    bw.plans, bw.plan_of_profile = [wl], np.zeros(64, dtype=np.int32)
    P = [W.dbm_to_w(np.random.default_rng(p).normal(1, 1.5, wl.n_ch)) for p in range(64)]
    got = eng.eta_batched(bw, np.concatenate(P)).reshape(64, wl.n_ch)
    for p in (0, 13, 63):
        np.testing.assert_array_equal(got[p], eng.eta(wl, P[p])["eta"])
