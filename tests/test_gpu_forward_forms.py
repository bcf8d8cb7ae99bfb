"""The two forms of the forward kernel, one corner row per warp in small launches and strips
of rows in big ones: every result is bitwise the same in both.

A batch above the small launches' CTA count (asserted, so that other tiles cannot move it back
below) against the same systems solved alone: elongated spots, FP64, and subapertures larger
than the layers' cells, where a strip skips node rows; cold and warm.  The noise-free
measurement of systems above that count against the FP64 oracle, relative L2 below 1e-5 in
FP32 and 1e-11 in FP64 as for the other operator checks.
"""
import numpy as np
import pytest

from host_plan import forward_ctas
from oracle import Tomography
from synth import configs

pytestmark = pytest.mark.gpu


def system(n_sub, d_sub, N, precision, elong, layers=3):
    g = configs.small_lgs_config(n_sub=n_sub, N=N, n_layers=layers, levels=2, precision=precision, d_sub=d_sub)
    return configs.with_elongation(g) if elong else g


@pytest.mark.parametrize("n_sub,d_sub,N,precision,elong,layers", [
    (61, 0.5, 128, 0, False, 3), (61, 0.5, 128, 0, True, 3), (45, 0.65, 128, 0, False, 5), (45, 0.65, 128, 0, True, 2),
    (31, 0.5, 64, 1, False, 3), (31, 0.5, 64, 1, True, 3), (33, 0.65, 128, 1, False, 2)])
def test_a_big_batch_has_the_bits_of_its_single_solves(n_sub, d_sub, N, precision, elong, layers, tmp_path):
    import torch
    from paper_1302_3734_gb300 import build
    from paper_1302_3734_gb300.binding import Plan, solve_batch
    build.build()
    g = system(n_sub, d_sub, N, precision, elong, layers)
    ctas, small = forward_ctas(g, 0, 1, tmp_path)
    count = small // ctas + 1
    assert ctas <= small < count * ctas and count <= 96
    dt = torch.float64 if precision else torch.float32
    plans = [Plan(g, transforms=1) for _ in range(count)]
    rng = np.random.default_rng(n_sub)
    sl = [torch.tensor(0.3 * rng.standard_normal(p.n_slopes), dtype=dt, device="cuda") for p in plans]
    x0 = [torch.tensor(0.1 * rng.standard_normal(p.n), dtype=dt, device="cuda") for p in plans]
    for warm in (False, True):
        alone = []
        for p, s, x in zip(plans, sl, x0):
            x = x.clone()
            p.solve(s, x, 3, warm=warm)
            alone.append(x.cpu().numpy())
        xs = [x.clone() for x in x0]
        solve_batch(plans, sl, xs, 3, warm=warm)
        for x, ref in zip(xs, alone):
            assert np.array_equal(x.cpu().numpy(), ref)


@pytest.mark.parametrize("n_sub,d_sub,N,precision,sensors", [(100, 0.5, 128, 0, 23), (91, 0.65, 128, 0, 27),
                                                             (64, 0.5, 128, 1, 21), (60, 0.65, 128, 1, 27)])
def test_measurement_of_a_big_system(n_sub, d_sub, N, precision, sensors, tmp_path):
    import torch
    from paper_1302_3734_gb300 import build
    from paper_1302_3734_gb300.binding import Plan
    build.build()
    g = system(n_sub, d_sub, N, precision, False, 2)
    w = g["wfs"]
    g["layers"][1]["altitude"] = 600.0
    g["wfs"] = w[2:3] + [dict(w[k % 2], theta=(1e-4 * np.cos(k), 1e-4 * np.sin(k))) for k in range(sensors)] + w[2:3]
    ctas, small = forward_ctas(g, 16, 2, tmp_path)
    assert ctas > small
    plan, ora = Plan(g, cluster_size=16, transforms=2), Tomography(g)
    dt = torch.float64 if precision else torch.float32
    phi = torch.tensor(np.random.default_rng(sensors).standard_normal(plan.n), dtype=dt, device="cuda")
    out = torch.empty(plan.n_slopes, dtype=dt, device="cuda")
    plan.layers_to_slopes(phi, out)
    grids = [p.reshape(N, N) for p in np.split(phi.cpu().numpy().astype(np.float64), 2)]
    ref = ora.measure(grids)
    got = out.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) < (1e-11 if precision else 1e-5)
    for k in (slice(0, 2), slice(-2, None)):     # the tip/tilt-only sensors' means
        assert np.linalg.norm(got[k] - ref[k]) / np.linalg.norm(ref[k]) < (1e-11 if precision else 1e-4)
