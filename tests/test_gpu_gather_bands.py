"""The separate gather at one node row per band: bands halved until the pupil-edge terms of a
row leave room for two CTAs per SM, terms that do not fit a CTA's shared memory at all, and a
layer with fewer rows than there are bands.  The right-hand side against the FP64 oracle,
relative L2 below 1e-11 as for the other FP64 operator checks.
"""
import numpy as np
import pytest

from gather_systems import many_edge_terms
from host_plan import gather_sizes
from oracle import Tomography

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_tt", [20, 55, 60])
def test_rhs_with_bands_of_one_row(n_tt, tmp_path):
    import torch
    from paper_1302_3734_gb300 import build
    from paper_1302_3734_gb300.binding import Plan
    build.build()
    g = many_edge_terms(n_tt)
    assert gather_sizes(g, 64, 2, tmp_path)[0] == max(l["N"] for l in g["layers"]) > min(l["N"] for l in g["layers"])
    plan = Plan(g, cluster_size=64, transforms=2)
    s = np.random.default_rng(n_tt).standard_normal(plan.n_slopes)
    out = torch.empty(plan.n, dtype=torch.float64, device="cuda")
    plan.rhs(torch.tensor(s, device="cuda"), out)
    ref = Tomography(g).rhs(s)
    assert np.linalg.norm(out.cpu().numpy() - ref) / np.linalg.norm(ref) < 1e-11
