"""Systems at the limits of the separate gather kernel."""
import numpy as np

from synth import configs


def many_edge_terms(n_tt):
    """n_tt tip/tilt-only sensors whose valid subapertures stand alone in two rows of 250: on a
    512 x 512 layer (FP64) each adds a pupil-edge term to 501 nodes of eight rows.  A second layer
    has half the rows (twice the pitch)."""
    g = configs.small_lgs_config(n_sub=12, N=512, n_layers=2, levels=4, precision=1, order=1, d_sub=1.0)
    n, dx = 250, g["layers"][0]["dx"]
    valid = np.zeros((n, n), dtype=np.uint8)
    valid[124:128:2, ::2] = 1
    tt = next(w for w in g["wfs"] if w["tt_only"])
    rng = np.random.default_rng(n_tt)
    g["layers"][0]["altitude"] = 1000.0
    g["layers"][1].update(altitude=0.0, N=256, dx=2 * dx)
    # footprints between a quarter and three quarters of a cell off the nodes
    g["wfs"] = g["wfs"][:1] + [dict(tt, n_sub=n, d_sub=2 * dx, valid=valid, sigma=0.1 + 0.01 * k,
                                    theta=tuple(rng.uniform(0.25, 0.75, 2) * dx / 1000.0)) for k in range(n_tt)]
    g["D_tel"] = n * 2 * dx
    return g
