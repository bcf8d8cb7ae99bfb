"""The streamed analysis and synthesis passes at the edges of their column groups
(block sides 128 to 1024), wavelets of 2 to 8 taps, both precisions, and arrays
that do not start on 16 bytes (a caller's tensor may be a slice).

Transforms against the FP64 oracle: relative L2 below 2e-6 in FP32 and 1e-12 in
FP64; a misaligned call against the aligned one: the same bits.
"""
import numpy as np
import pytest

from oracle import Tomography
from synth import configs

pytestmark = pytest.mark.gpu


def one_layer(N, order, levels, precision, precond=1):
    g = configs.small_lgs_config(n_sub=12, N=32, n_layers=1, levels=1, precision=precision, order=order,
                                 precond=precond)
    g["layers"] = [dict(g["layers"][0], N=N)]
    g["levels"] = levels
    return g


@pytest.mark.parametrize("N,order,levels,precision", [(128, 1, 1, 0), (128, 3, 4, 0), (256, 2, 2, 0), (256, 4, 5, 0),
                                                      (512, 3, 6, 0), (1024, 4, 7, 0), (128, 2, 3, 1), (256, 4, 4, 1)])
def test_passes_and_misaligned_arrays(N, order, levels, precision):
    import torch
    from paper_1302_3734_gb300 import build
    from paper_1302_3734_gb300.binding import Plan
    build.build()
    g = one_layer(N, order, levels, precision)
    plan = Plan(g, cluster_size=64 if N > 512 else 16, transforms=2)
    ora = Tomography(g)
    rng = np.random.default_rng(N + order)
    dt = torch.float64 if precision else torch.float32
    n = plan.n
    x = torch.tensor(rng.standard_normal(n), dtype=dt, device="cuda")
    s = torch.tensor(rng.standard_normal(plan.n_slopes), dtype=dt, device="cuda")
    tol = 1e-12 if precision else 2e-6

    def runs(shift):
        buf = [torch.zeros(n + 4, dtype=dt, device="cuda") for _ in range(4)]
        a, b, c, d = (t[shift:shift + n] for t in buf)
        xs = torch.zeros(n + 4, dtype=dt, device="cuda")[shift:shift + n]
        xs.copy_(x)
        plan.layers_to_coeffs(xs, a)
        plan.coeffs_to_layers(xs, b)
        plan.apply_normal(xs, c)
        d.copy_(xs)
        plan.solve(s, d, 2, warm=True)
        return [t.cpu().numpy().astype(np.float64) for t in (a, b, c, d)]

    plain, shifted = runs(0), runs(1)
    for p, q in zip(plain, shifted):
        assert np.array_equal(p, q)
    xh = x.cpu().numpy().astype(np.float64)
    w, phi = ora.analysis([xh.reshape(N, N)]), ora.join(ora.synthesis(xh))
    assert np.linalg.norm(plain[0] - w) / np.linalg.norm(w) < tol
    assert np.linalg.norm(plain[1] - phi) / np.linalg.norm(phi) < tol


@pytest.mark.parametrize("N,C,order,levels,precision", [(16, 4, 2, 3, 0), (32, 4, 3, 3, 0), (32, 1, 1, 5, 0),
                                                        (64, 8, 3, 2, 0), (64, 2, 4, 4, 1), (128, 16, 3, 5, 0),
                                                        (128, 4, 2, 1, 0), (256, 16, 4, 6, 0)])
def test_coarse_block_of_the_cluster_transforms(N, C, order, levels, precision):
    """CTA 0's block (larger than one row per CTA, not reached, or a single level): the same
    bits as the streamed transforms."""
    import torch
    from paper_1302_3734_gb300 import build
    from paper_1302_3734_gb300.binding import Plan
    build.build()
    g = one_layer(N, order, levels, precision)
    if N == 16:
        g = dict(configs.small_lgs_config(n_sub=6, N=16, n_layers=2, levels=levels, precision=precision, order=order))
    dt = torch.float64 if precision else torch.float32
    out = []
    for tf, c in ((1, C), (2, C)):
        plan = Plan(g, cluster_size=c, transforms=tf)
        x = torch.tensor(np.random.default_rng(1).standard_normal(plan.n), dtype=dt, device="cuda")
        res = [torch.empty_like(x) for _ in range(3)]
        plan.layers_to_coeffs(x, res[0])
        plan.coeffs_to_layers(x, res[1])
        plan.apply_normal(x, res[2])
        out.append([r.cpu().numpy() for r in res])
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_big_batch_forms_alpha_once():
    """More update CTAs than one wave: alpha comes from its own kernel.  Every instance gets the
    bits of its single solve, and one whose data are NaN breaks down alone."""
    import torch
    from paper_1302_3734_gb300 import build
    from paper_1302_3734_gb300.binding import Plan, TomoError, solve_batch
    build.build()
    g = configs.config1()
    plans = [Plan(g, cluster_size=2, transforms=2) for _ in range(5)]
    rng = np.random.default_rng(3)
    sl = [torch.tensor(0.3 * rng.standard_normal(p.n_slopes), dtype=torch.float32, device="cuda") for p in plans]
    single = []
    for p, s in zip(plans, sl):
        x = torch.zeros(p.n, dtype=torch.float32, device="cuda")
        p.solve(s, x, 3, warm=False)
        single.append(x.cpu().numpy())
    xs = [torch.zeros(p.n, dtype=torch.float32, device="cuda") for p in plans]
    solve_batch(plans, sl, xs, 3, warm=False)
    for x, ref in zip(xs, single):
        assert np.array_equal(x.cpu().numpy(), ref)
    sl[2].fill_(float("nan"))
    xs = [torch.zeros(p.n, dtype=torch.float32, device="cuda") for p in plans]
    solve_batch(plans, sl, xs, 3, warm=True)
    torch.cuda.synchronize()
    assert plans[2]._info().breakdown_pending == 1 and plans[1]._info().breakdown_pending == 0
    assert np.array_equal(xs[2].cpu().numpy(), np.zeros(plans[2].n, dtype=np.float32))
    for i in (0, 1, 3, 4):
        assert np.array_equal(xs[i].cpu().numpy(), single[i])
    with pytest.raises(TomoError):
        plans[2].solve(sl[2], xs[2], 1)
