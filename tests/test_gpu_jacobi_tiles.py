"""The Jacobi diagonal's CTA tiles at the edges of their ranges, against the FP64
oracle: level blocks narrower than a tile (side 4 and up), a pupil of one
subaperture, row counts that leave a ragged last chunk of 32 subaperture rows,
and a pupil whose prefix sums only fit 8 columns per CTA (n_sub > 360).

Tolerance 1e-12 (relative L2), as for the other Jacobi checks: FP64 on the device.
"""
import math

import numpy as np
import pytest

from oracle import Tomography
from synth import configs

pytestmark = pytest.mark.gpu


def geom(n_sub, d_sub, N, levels, order, altitude=0.0):
    g = configs.small_lgs_config(n_sub=8, N=32, n_layers=1, levels=1, full_ngs=False)
    D = n_sub * d_sub
    w = dict(g["wfs"][0], theta=(0.0, 0.0), n_sub=n_sub, d_sub=d_sub, valid=configs.pupil_mask(n_sub, d_sub, D, 0.2 if n_sub > 4 else 0.0))
    g.update(D_tel=D, wfs=[w], wavelet_order=order, levels=levels,
             layers=[dict(g["layers"][0], altitude=altitude, N=N, dx=0.5)])
    return g


@pytest.mark.parametrize("n_sub,d_sub,N,levels,order,altitude", [
    (1, 0.5, 16, 3, 2, 0.0), (13, 0.5, 16, 4, 1, 2000.0), (33, 0.5, 64, 3, 4, 9000.0), (64, 0.4, 64, 1, 3, 4000.0),
    (361, 0.25, 256, 2, 3, 0.0), (420, 0.25, 256, 5, 4, 0.0)])
def test_jacobi_diagonal_tiles(n_sub, d_sub, N, levels, order, altitude):
    import torch
    from paper_1302_3734_gb300 import build
    from paper_1302_3734_gb300.binding import Plan
    build.build()
    g = geom(n_sub, d_sub, N, levels, order, altitude)
    plan = Plan(g)
    out = torch.empty(plan.n, dtype=torch.float64, device="cuda")
    plan.jacobi_diagonal(out)
    ref = Tomography(g).jacobi_diagonal()
    got = out.cpu().numpy()
    assert math.isfinite(got.sum())
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) < 1e-12
