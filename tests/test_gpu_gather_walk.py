"""The separate gather (streamed plans) where its walk down the node rows can go
wrong, against the FP64 oracle: windows that move by zero, one, two or more
corner rows from node to node (subapertures smaller and larger than the layer
cells), sensors with fewer corners than taps, footprints that wrap around the
grid, bands of one row and bands that are halved to fit shared memory, and
spot elongation.

Tolerances (relative L2): right-hand side 1e-5 in FP32 (differences of nearby
values cancel in the slopes' transpose), 1e-11 in FP64, as for the other
operator checks.
"""
import numpy as np
import pytest

from oracle import Tomography
from synth import configs

pytestmark = pytest.mark.gpu

# (n_sub, d_sub, N, layers, bands, precision, extra)
CASES = [(1, 0.6, 16, 2, 8, 0, ""), (2, 0.9, 32, 3, 1, 0, ""), (3, 0.3, 16, 2, 4, 1, ""), (17, 0.3, 32, 3, 16, 0, ""),
         (31, 0.5, 64, 3, 2, 0, "wrap"), (32, 0.75, 128, 3, 64, 0, ""), (33, 1.3, 128, 2, 1, 0, ""),
         (84, 0.5, 128, 5, 1, 0, ""), (20, 0.5, 64, 4, 4, 0, "elong"), (13, 0.4, 32, 3, 2, 1, "elong")]


@pytest.mark.parametrize("n_sub,d_sub,N,layers,bands,precision,extra", CASES)
def test_rhs_through_the_separate_gather(n_sub, d_sub, N, layers, bands, precision, extra):
    import torch
    from paper_1302_3734_gb300 import build
    from paper_1302_3734_gb300.binding import Plan
    build.build()
    g = configs.small_lgs_config(n_sub=n_sub, N=N, n_layers=layers, levels=1, precision=precision, d_sub=d_sub,
                                 obstruction=0.3 if n_sub > 4 else 0.0, wrap=extra == "wrap")
    if extra == "elong":
        g = configs.with_elongation(g)
    plan = Plan(g, cluster_size=bands, transforms=2)
    assert plan.info.streamed and plan.info.gather_separate
    s = np.random.default_rng(5).standard_normal(plan.n_slopes)
    dt = torch.float64 if precision else torch.float32
    sl = torch.tensor(s, dtype=dt, device="cuda")
    out = torch.empty(plan.n, dtype=dt, device="cuda")
    plan.rhs(sl, out)
    ref = Tomography(g).rhs(sl.cpu().numpy().astype(np.float64))
    got = out.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) < (1e-11 if precision else 1e-5)
