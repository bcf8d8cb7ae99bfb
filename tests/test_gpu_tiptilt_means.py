"""The two mean slopes of a tip/tilt-only sensor in the noise-free measurement of an
FP32 plan: their sum over the pupil-edge corners is taken in FP64.

The corners of the sensor lie on the nodes of the one layer, so the traced phase is
the grid value itself.  Values of 2^31 (multiples of 2^7) that cancel by symmetry are
mixed with values below 1 (multiples of 2^-17 or 2^-15): every partial sum fits 53
bits, so FP64 gives the exact mean rounded once to FP32, in any order; 48 bits do not.
"""
import math

import numpy as np
import pytest

from synth import configs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_sub,N,bits,seed", [(16, 32, 17, 1), (17, 64, 17, 2), (40, 64, 15, 3)])
def test_mean_slopes_are_summed_in_fp64(n_sub, N, bits, seed):
    import torch
    from paper_1302_3734_gb300 import build
    from paper_1302_3734_gb300.binding import Plan
    build.build()
    d = 1.0 if n_sub % 2 else 0.5     # two cells per subaperture keep an odd sensor's corners on the nodes
    g = configs.small_lgs_config(n_sub=n_sub, N=N, n_layers=1, levels=1, full_ngs=False, d_sub=d)
    g["wfs"] = [w for w in g["wfs"] if w["tt_only"]] + g["wfs"][:1]
    rng = np.random.default_rng(seed)
    # one draw per orbit of the reflections about the pupil's centre (node N / 2)
    q = N // 2
    big = 128.0 * rng.integers(2 ** 23, 2 ** 24, (q + 1, q + 1))
    is_big = rng.random((q + 1, q + 1)) < 0.5
    k = np.abs(np.arange(N) - q)
    phi = np.where(is_big[np.ix_(k, k)], big[np.ix_(k, k)], rng.integers(-2 ** bits, 2 ** bits, (N, N)) / 2.0 ** bits)
    assert np.array_equal(phi, phi.astype(np.float32))
    w = g["wfs"][0]
    n, step = w["n_sub"], int(round(w["d_sub"] / g["layers"][0]["dx"]))
    at = np.arange(n + 1) * step - n * step // 2 + q
    assert (n * step) % 2 == 0 and at.min() >= 0 and at.max() < N
    psi = phi[np.ix_(at, at)]
    v = np.asarray(w["valid"]) != 0
    sx = 0.5 * np.stack([psi[:-1, 1:], psi[1:, 1:], -psi[:-1, :-1], -psi[1:, :-1]])[:, v]
    sy = 0.5 * np.stack([psi[1:, :-1], psi[1:, 1:], -psi[:-1, :-1], -psi[:-1, 1:]])[:, v]
    # what the sum over the edge corners can reach, in units of the smallest term's last bit
    t = np.zeros((2, n + 1, n + 1))
    for d, s in ((0, (-1, 1, -1, 1)), (1, (-1, -1, 1, 1))):
        for c, (dy, dx) in zip(s, ((0, 0), (0, 1), (1, 0), (1, 1))):
            t[d, dy:n + dy, dx:n + dx] += 0.5 * c * v
    assert np.abs(t * psi).sum(axis=(1, 2)).max() * 2.0 ** (bits + 1) < 2.0 ** 53
    ref = [np.float32(math.fsum(s.ravel()) / v.sum()) for s in (sx, sy)]
    plan = Plan(g)
    out = torch.empty(plan.n_slopes, dtype=torch.float32, device="cuda")
    plan.layers_to_slopes(torch.tensor(phi.ravel(), dtype=torch.float32, device="cuda"), out)
    assert out[:2].cpu().numpy().tolist() == ref
