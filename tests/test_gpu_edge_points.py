"""Which F_c channel a grid point next to a channel's edge belongs to.

On the FP32 path a point's F_c - f_i is the FP32 sum of its f1 and f2: a point within a
few 1e-6 THz of an edge falls on the side where that rounding puts it, and on a plan of
equal slots each such point is worth up to 1e-3 of a channel's eta (5e-5 in the 2-norm).
With every point on its side what is left against the recorded values is the rounding of
phi, up to 1e-7 of tens to hundreds of radians along a row, averaged over a channel's
thousands of points: below 5e-6 in the 2-norm and 1e-4 of any channel."""
import json
import os

import numpy as np
import pytest

from paper_2401_18022_gb300 import workloads as W

pytestmark = pytest.mark.gpu

GOLDEN = json.load(open(os.path.join(os.path.dirname(__file__), "golden", "edge_points_fp32.json")))


@pytest.fixture(scope="module")
def eng():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2401_18022_gb300 import api
    return api.Engine(0)


@pytest.mark.parametrize("profile", ["closed_form", "raman_ode"])
@pytest.mark.parametrize("call", ["eta", "grad"])
def test_recorded_values(eng, profile, call):
    d = GOLDEN
    wl = W.uwb(G=d["G"], n_edges=d["n_edges"], cell_set=W.CELLS_SCI_XCI)
    wl = W.subset_plan(wl, np.arange(d["first_slot"], d["first_slot"] + d["n"]), "zero dispersion")
    P = W.dbm_to_w(np.random.default_rng(d["power_seed"]).normal(1, 1.5, d["n"]))
    eta = np.asarray(getattr(eng, call)(W.raman(wl) if profile == "raman_ode" else wl, P)["eta"])
    ref = np.array(d[profile])
    assert np.linalg.norm(eta - ref) < 5e-6 * np.linalg.norm(ref)
    assert np.abs(eta / ref - 1).max() < 1e-4
