"""The work this framework is measured on, through its public entry points.

Each listed case is one thing a user's program has the library do; `draw` gives
more of the same kinds over the sizes, wavelets, precisions and options the
library takes.  The inputs are seeded von Karman screens (Sec. 3 of the paper),
their slopes with white noise, and the previous frame's solution as the warm
start; they are made here in 64 bits, and `exact` solves the same problems in
64 bits with dense interpolation and wavelet matrices, sharing no code with the
library.
"""
import math

import numpy as np
import torch

import paper_1302_3734_gb300 as tomo

ARCMIN = math.pi / (180.0 * 60.0)
SODIUM = 90e3                     # laser guide star altitude (m)
R0, L0 = 0.15, 25.0               # Fried parameter at 500 nm and outer scale (m)
FRAME_S = 0.002                   # 500 Hz
ELT_HEIGHTS = [0.0, 600.0, 1200.0, 2500.0, 5000.0, 7500.0, 10000.0, 15000.0, 20000.0]
ELT_CN2 = [0.5, 0.1, 0.1, 0.07, 0.06, 0.05, 0.05, 0.04, 0.03]
FIT_DMS = [(0.0, 0.5), (4000.0, 0.72), (12700.0, 1.0)]   # mirror altitude and pitch (m)

# One adaptive-optics system (see `geometry`): the E-ELT-sized MCAO system of Sec. 5.1.
EELT = {"n_sub": 84, "d_sub": 0.5, "obstruction": math.sqrt(0.28), "lgs": 6, "lgs_ring": 1.0, "tt": 3, "ngs": 0,
        "layers": 9, "profile": "elt", "N": 128, "order": 3, "levels": 4, "precision": 0, "precond": 1,
        "elong": False}
# The 8 m system: three full-resolution natural guide stars, two layers.
VLT = {"n_sub": 16, "d_sub": 0.5, "obstruction": 0.0, "lgs": 0, "lgs_ring": 0.0, "tt": 0, "ngs": 3,
       "layers": 2, "profile": "two", "N": 32, "order": 3, "levels": 3, "precision": 0, "precond": 1, "elong": False}
# The 100 m system: 9 LGS, 35 layers of 512^2, db4.
OWL = {"n_sub": 200, "d_sub": 0.5, "obstruction": 0.0, "lgs": 9, "lgs_ring": 0.75, "tt": 3, "ngs": 0,
       "layers": 35, "profile": "dense", "N": 512, "order": 4, "levels": 5, "precision": 0, "precond": 1,
       "elong": False}


def listed():
    return [
        # The smallest telescope of the served mix, one frame from the previous one: launches and latency.
        {"name": "frame_8m", "kind": "frame", **VLT, "iters": 10, "warm": True},
        # The same telescope in the FP64 build with plain CG, cold: the reference-accuracy configuration.
        {"name": "frame_8m_fp64", "kind": "frame", **dict(VLT, precision=1, precond=0), "iters": 30, "warm": False},
        # The headline: one E-ELT frame, 10 PCG iterations from the previous frame's solution.
        {"name": "frame_eelt", "kind": "frame", **EELT, "iters": 10, "warm": True},
        # The normal operator alone, with spot-elongated laser guide stars (a caller's own Krylov solver).
        {"name": "normal_eelt_elong", "kind": "normal", **dict(EELT, elong=True)},
        # Sixteen E-ELT systems per launch, at the launch shape the autotuner picks for them.
        {"name": "batch16_eelt", "kind": "batch", "set": "eelt", "count": 16, "cluster": 2, "transforms": 2,
         "iters": 10},
        # Sixty-four systems of uneven size per launch (16..84 subapertures, 2..9 layers, 32..256 grids).
        {"name": "batch64_uneven", "kind": "batch", "set": "uneven", "sizes": 2000, "count": 64, "cluster": 4,
         "transforms": 2, "iters": 10},
        # The largest system, cold: 9.2 M unknowns.  10 iterations, the count up to which FP32 runs of this
        # system are comparable (its own 20 amplify any rounding far beyond FP32).
        {"name": "frame_100m", "kind": "frame", **OWL, "iters": 10, "warm": False},
        # One closed-loop control step, slopes to mirror commands (Algorithm 4.1): solve, fitting, integrator.
        {"name": "control_eelt", "kind": "control", **EELT, "iters": 10, "fit_iters": 4, "gain": 0.4},
        # The fitting step alone, layers to commands of three mirrors over 5 x 5 directions.
        {"name": "fit_eelt", "kind": "fit", **EELT, "fit_iters": 4},
        # The plant of a closed-loop simulation: the sensors' slopes of the true layers, minus what the
        # mirrors take away, and the residual wavefront error per direction.
        {"name": "plant_eelt", "kind": "plant", **EELT},
        # A real-time thread retuning alpha: the Jacobi diagonal again, without allocating.
        {"name": "jacobi_eelt", "kind": "jacobi", **EELT},
        # One frame from each of 16 telescopes (8 m, E-ELT and uneven ones) through the server, host to host.
        {"name": "serve16", "kind": "serve", "telescopes": 16, "cluster": 4, "transforms": 2, "iters": 10},
    ]


def _grid_need(n_sub, d_sub, profile_top, ring):
    return 2.0 * (ring * ARCMIN * profile_top + n_sub * d_sub / 2.0) / 0.5 + 4.0


def draw(rng):
    """One more case: any kind, sizes over the listed range (odd ones among them)."""
    kind = rng.choice(["frame", "frame", "frame", "normal", "normal", "batch", "control", "fit", "plant", "jacobi"])
    if kind == "batch":
        if rng.random() < 0.5:
            tf = rng.choice([1, 2])
            return {"kind": "batch", "set": "uneven", "sizes": rng.randrange(1, 10 ** 6), "count": rng.randint(2, 40),
                    "cluster": 8 if tf == 1 else rng.choice([2, 4, 8]), "transforms": tf, "iters": rng.randint(5, 10)}
        return {"kind": "batch", "set": "eelt", "count": rng.randint(2, 15), "cluster": rng.choice([2, 4]),
                "transforms": rng.choice([1, 2]), "iters": rng.randint(5, 10)}
    top = 120 if kind in ("frame", "normal") else 84
    n_sub = int(round(math.exp(rng.uniform(math.log(9), math.log(top)))))
    d_sub = rng.choice([0.4, 0.5, 0.5, 0.625])
    layers = rng.randint(1, 9)
    lgs, tt, ngs = rng.choice([(0, 0, 3), (0, 0, 4), (3, 3, 0), (4, 3, 0), (5, 3, 1), (6, 3, 0), (6, 2, 1)])
    need = _grid_need(n_sub, d_sub, ELT_HEIGHTS[layers - 1], 1.0)
    N = next(g for g in (16, 32, 64, 128, 256, 512) if g >= need)
    order = rng.choice([2, 3, 3, 4])
    levels = rng.randint(1, min(5, int(math.log2(N // (2 * order))) + 1))
    c = {"kind": kind, "n_sub": n_sub, "d_sub": d_sub, "obstruction": rng.choice([0.0, 0.3]), "lgs": lgs,
         "lgs_ring": 1.0, "tt": tt, "ngs": ngs, "layers": layers, "profile": "elt", "N": N, "order": order,
         "levels": levels, "precision": int(N <= 128 and rng.random() < 0.15), "precond": 1 if lgs else int(rng.random() < 0.5),
         "elong": bool(lgs and rng.random() < 0.25)}
    if kind == "frame":
        c.update(iters=rng.randint(3, 10), warm=rng.random() < 0.7)
    elif kind == "control":
        c.update(iters=rng.randint(3, 10), fit_iters=rng.randint(2, 5), gain=0.4)
    elif kind == "fit":
        c.update(fit_iters=rng.randint(2, 6))
    return c


# ------------------------------------------------------------------ geometries

def _pupil(n, d, D, obs):
    c = (np.arange(n) + 0.5 - n / 2.0) * d
    r = np.hypot(*np.meshgrid(c, c))
    return ((r <= D / 2.0) & (r >= obs * D / 2.0)).astype(np.uint8)


def _ring(n, arcmin, start):
    a = [math.radians(start + 360.0 * k / n) for k in range(n)]
    return [(arcmin * ARCMIN * math.cos(t), arcmin * ARCMIN * math.sin(t)) for t in a]


def _profile(case):
    L = case["layers"]
    if case["profile"] == "two":
        return [0.0, 6000.0], [0.7, 0.3]
    if case["profile"] == "dense":
        h = [0.0] + sorted(float(x) for x in np.random.default_rng(4000).uniform(0.0, 25e3, L - 1))
        return h, [math.exp(-x / 5e3) for x in h]
    return ELT_HEIGHTS[:L], ELT_CN2[:L]


def geometry(case):
    """The library's geometry dict of a case."""
    n, d, obs, dx = case["n_sub"], case["d_sub"], case["obstruction"], 0.5
    D = n * d
    valid = _pupil(n, d, D, obs)

    def sensor(theta, height, sigma, **kw):
        return {"theta": theta, "height": height, "n_sub": n, "d_sub": d, "valid": valid, "sigma": sigma,
                "tt_only": False, "remove_tt": False, **kw}

    wfs = [sensor(t, SODIUM, 0.3, remove_tt=True) for t in _ring(case["lgs"], case["lgs_ring"], 0.0)]
    if case["elong"]:
        for w in wfs:      # 10 km of sodium seen from a launch at the pupil's edge, in units of a 1" spot
            az = math.atan2(w["theta"][1], w["theta"][0])
            w.update(elong_tau=0.8, elong_scale=10e3 / SODIUM ** 2 / (ARCMIN / 60.0),
                     llt=(D / 2.0 * math.cos(az), D / 2.0 * math.sin(az)))
    wfs += [sensor(t, math.inf, 0.1, tt_only=True) for t in _ring(case["tt"], 1.0, 90.0)]
    wfs += [sensor(t, math.inf, 0.1) for t in _ring(case["ngs"], 0.5, 90.0)]
    heights, cn2 = _profile(case)
    tot = sum(cn2)
    lay = [{"altitude": h, "dx": dx, "N": case["N"],
            "prior_weight": 1.0 / (f / tot * 0.9 * (dx / R0) ** (5 / 3) * (2 * dx) ** (11 / 3))}
           for h, f in zip(heights, cn2)]
    g = {"D_tel": D, "obstruction": obs, "wfs": wfs, "layers": lay, "wavelet_order": case["order"],
         "levels": case["levels"], "alpha": 1.0, "L0": L0, "precond": case["precond"],
         "precision": case["precision"], "cn2": [f / tot for f in cn2]}
    if case["kind"] in ("control", "fit", "plant"):
        half = ARCMIN
        ts = np.linspace(-half, half, 5)
        g["fitting"] = {"dms": [{"altitude": h, "pitch": p, "n": 2 * int(math.ceil((D / 2.0 + h * half) / p)) + 3}
                                for h, p in FIT_DMS],
                        "directions": [(float(x), float(y)) for y in ts for x in ts], "n_sub": n, "d_sub": d,
                        "valid": valid}
    return g


def _members(case):
    """The systems of a batch or of the served mix, as single cases."""
    if case.get("set") == "eelt":
        return [dict(EELT, kind="frame") for _ in range(case["count"])]
    rng = np.random.default_rng(case.get("sizes", 2000))
    out = []
    for _ in range(case.get("count", 16)):
        n = int(rng.choice([16, 32, 40, 64, 84]))
        L, lgs = int(rng.integers(2, 10)), int(rng.integers(3, 7))
        need = _grid_need(n, 0.5, ELT_HEIGHTS[L - 1], 1.0)
        N = int(rng.choice([g for g in (32, 64, 128, 256) if g >= need]))
        out.append(dict(EELT, kind="frame", n_sub=n, obstruction=0.0, lgs=lgs, layers=L, N=N,
                        levels=min(4, int(round(math.log2(N))) - 2)))
    if case["kind"] == "serve":
        out = [dict(VLT, kind="frame") if i % 3 == 0 else dict(EELT, kind="frame") if i % 3 == 1 else out[i]
               for i in range(case["telescopes"])]
    return out


# ------------------------------------------- the same problems in 64 bits

def _dev():
    return torch.device("cuda")


def _taps(order):
    """Daubechies low-pass taps with `order` vanishing moments, minimum phase (spectral factorisation)."""
    y = np.roots([math.comb(order - 1 + k, k) for k in range(order - 1, -1, -1)])
    h = np.poly1d([1.0])
    for _ in range(order):
        h = h * np.poly1d([1.0, 1.0])
    for r in y:
        z = np.roots([1.0, -(2.0 - 4.0 * r), 1.0])
        h = h * np.poly1d([1.0, -z[np.argmin(np.abs(z))]])
    h = np.real(h.coeffs)
    return h * math.sqrt(2.0) / h.sum()


def _linear(coord, n, periodic):
    """Interpolation matrices [..., points, n] of the coordinates on n nodes (zero outside unless periodic)."""
    i0 = torch.floor(coord)
    f = coord - i0
    A = torch.zeros(*coord.shape, n, dtype=torch.float64, device=coord.device)
    for i, w in ((i0.long(), 1.0 - f), (i0.long() + 1, f)):
        if not periodic:
            w = torch.where((i >= 0) & (i < n), w, torch.zeros_like(w))
        A.scatter_add_(-1, (i % n).unsqueeze(-1), w.unsqueeze(-1))
    return A


class Model:
    """Normal equations, right-hand side, Jacobi diagonal, fitting and control of one geometry."""

    def __init__(self, g):
        dev = _dev()
        self.g, self.J = g, g["levels"]
        self.N, self.L = g["layers"][0]["N"], len(g["layers"])
        N, dx = self.N, g["layers"][0]["dx"]
        self.alt = torch.tensor([l["altitude"] for l in g["layers"]], dtype=torch.float64, device=dev)
        h = _taps(g["wavelet_order"])
        gg = np.array([(-1) ** k * h[len(h) - 1 - k] for k in range(len(h))])
        self.W = []                                     # analysis matrix of each level
        for k in range(self.J):
            M = N >> k
            A = np.zeros((M, M))
            for i in range(M // 2):
                for t in range(len(h)):
                    A[i, (2 * i + t) % M] += h[t]
                    A[M // 2 + i, (2 * i + t) % M] += gg[t]
            self.W.append(torch.tensor(A, device=dev))
        lev = np.full((N, N), self.J)
        for k in range(self.J, 0, -1):
            H = N >> k
            m = np.maximum(*np.indices((N, N)))
            lev[(m >= H) & (m < 2 * H)] = k
        self.lev = torch.tensor(lev, device=dev)
        pw = torch.tensor([l["prior_weight"] for l in g["layers"]], dtype=torch.float64, device=dev)
        D = L0 ** (-11 / 3) + torch.pow(dx * torch.pow(2.0, self.lev.double()), -11 / 3)
        self.D = pw[:, None, None] * D[None]
        self.sens = []
        for w in g["wfs"]:
            n, d = w["n_sub"], w["d_sub"]
            r = (torch.arange(n + 1, dtype=torch.float64, device=dev) - n / 2.0) * d
            lgs = math.isfinite(w["height"])
            cone = 1.0 - self.alt / w["height"] if lgs else torch.ones_like(self.alt)
            ax, ay = [_linear((cone[:, None] * r[None] + th * self.alt[:, None]) / dx + N / 2.0, N, True)
                      for th in w["theta"]]
            v = torch.tensor(w["valid"], dtype=torch.float64, device=dev)
            s = {"w": w, "ax": ax, "ay": ay, "v": v, "S": float(v.sum()), "lgs": lgs, "el": None,
                 "idx": v.flatten().nonzero()[:, 0], "r": r}
            act = torch.zeros(n + 1, n + 1, dtype=torch.float64, device=dev)
            for b in (0, 1):
                for a in (0, 1):
                    act[b:b + n, a:a + n] += v
            s["act"] = (act > 0).double()
            if lgs and w.get("elong_tau", 0.0) > 0.0 and not w["tt_only"]:
                c = r[:-1] + d / 2.0
                gx = (w["elong_scale"] * (c - w["llt"][0]))[None, :].expand(n, n)
                gy = (w["elong_scale"] * (c - w["llt"][1]))[:, None].expand(n, n)
                t = w["elong_tau"]
                s["el"] = (gx, gy, t / (1.0 + t * (gx * gx + gy * gy)))
            self.sens.append(s)
        self.n_meas = [2 if s["w"]["tt_only"] else 2 * len(s["idx"]) for s in self.sens]
        self._fit = None

    # wavelets
    def synthesis(self, c):
        x = c.reshape(self.L, self.N, self.N).clone()
        for A in reversed(self.W):
            M = A.shape[0]
            x[:, :M, :M] = A.T @ x[:, :M, :M] @ A
        return x

    def analysis(self, phi):
        x = phi.clone()
        for A in self.W:
            M = A.shape[0]
            x[:, :M, :M] = A @ x[:, :M, :M] @ A.T
        return x.flatten()

    # sensors
    @staticmethod
    def fried(s, psi):
        a, b, c, e = psi[:-1, :-1], psi[:-1, 1:], psi[1:, :-1], psi[1:, 1:]
        return 0.5 * (b + e - a - c) * s["v"], 0.5 * (c + e - a - b) * s["v"]

    @staticmethod
    def fried_t(s, x, y):
        x, y = 0.5 * x * s["v"], 0.5 * y * s["v"]
        f = torch.zeros_like(s["act"])
        f[:-1, 1:] += x - y
        f[1:, 1:] += x + y
        f[:-1, :-1] -= x + y
        f[1:, :-1] += y - x
        return f

    def see(self, s, phi):
        return self.fried(s, (s["ay"] @ phi @ s["ax"].transpose(1, 2)).sum(0) * s["act"])

    def noise(self, s, x, y):
        if s["el"] is not None:
            gx, gy, c = s["el"]
            t = c * (gx * x + gy * y)
            x, y = x - gx * t, y - gy * t
        return x / s["w"]["sigma"] ** 2, y / s["w"]["sigma"] ** 2

    def weight(self, s, x, y, means=None):
        """C^-1 of model slopes (or, for a tip/tilt-only sensor's data, of its two means)."""
        v, S = s["v"], s["S"]
        if s["w"]["tt_only"]:
            mx, my = means if means is not None else (x.sum() / S, y.sum() / S)
            k = 1.0 / (s["w"]["sigma"] ** 2 * S)
            return mx * k * v, my * k * v
        if s["w"]["remove_tt"]:
            x, y = self.noise(s, (x - x.sum() / S) * v, (y - y.sum() / S) * v)
            x, y = x * v, y * v
            return (x - x.sum() / S) * v, (y - y.sum() / S) * v
        return self.noise(s, x, y)

    def pack(self, s, x, y):
        if s["w"]["tt_only"]:
            return torch.stack([x.sum() / s["S"], y.sum() / s["S"]])
        return torch.cat([x.flatten()[s["idx"]], y.flatten()[s["idx"]]])

    def measure(self, phi):
        return torch.cat([self.pack(s, *self.see(s, phi)) for s in self.sens])

    def back(self, g, s, x, y):
        g += s["ay"].transpose(1, 2) @ (self.fried_t(s, x, y) * s["act"]) @ s["ax"]

    def normal(self, c):
        phi = self.synthesis(c)
        g = torch.zeros_like(phi)
        for s in self.sens:
            self.back(g, s, *self.weight(s, *self.see(s, phi)))
        return self.analysis(g) + self.g["alpha"] * self.D.flatten() * c

    def rhs(self, slopes):
        g = torch.zeros(self.L, self.N, self.N, dtype=torch.float64, device=slopes.device)
        for s, z in zip(self.sens, slopes.split(self.n_meas)):
            if s["w"]["tt_only"]:
                x, y = self.weight(s, None, None, means=(z[0], z[1]))
            else:
                k = len(s["idx"])
                x, y = torch.zeros_like(s["v"]).flatten(), torch.zeros_like(s["v"]).flatten()
                x[s["idx"]], y[s["idx"]] = z[:k], z[k:]
                x, y = self.weight(s, x.view_as(s["v"]), y.view_as(s["v"]))
            self.back(g, s, x, y)
        return self.analysis(g)

    def jacobi(self, alpha):
        N, out = self.N, torch.zeros(self.L, self.N, self.N, dtype=torch.float64, device=_dev())
        for k in range(1, self.J + 1):
            M = N >> (k - 1)
            P = torch.eye(M, dtype=torch.float64, device=_dev())
            for A in reversed(self.W[:k]):            # basis functions of level k: synthesis of unit vectors
                m = A.shape[0]
                P = P @ A if P.shape[1] == m else torch.nn.functional.pad(P, (0, m - P.shape[1])) @ A
            acc = torch.zeros(self.L, M, M, dtype=torch.float64, device=_dev())
            for s in self.sens:
                if not s["lgs"]:
                    continue
                U, V = P @ s["ax"].transpose(1, 2), P @ s["ay"].transpose(1, 2)
                dU, mU = U[..., 1:] - U[..., :-1], 0.5 * (U[..., 1:] + U[..., :-1])
                dV, mV = V[..., 1:] - V[..., :-1], 0.5 * (V[..., 1:] + V[..., :-1])
                acc += ((mV ** 2) @ s["v"] @ (dU ** 2).transpose(1, 2)
                        + (dV ** 2) @ s["v"] @ (mU ** 2).transpose(1, 2)) / s["w"]["sigma"] ** 2
            sel = self.lev[:M, :M] == k
            out[:, :M, :M] = torch.where(sel[None], acc, out[:, :M, :M])
        return (out + alpha * self.D).flatten()

    @staticmethod
    def cg(op, b, x, iters, jac=None):
        """Hestenes-Stiefel (P)CG, exactly `iters` iterations."""
        r = b - op(x)
        z = r / jac if jac is not None else r
        p, rz = z, r @ z
        for _ in range(iters):
            q = op(p)
            a = torch.where(rz == 0, torch.zeros_like(rz), rz / (p @ q))
            x, r = x + a * p, r - a * q
            z = r / jac if jac is not None else r
            new = r @ z
            p, rz = z + torch.where(rz == 0, torch.zeros_like(rz), new / rz) * p, new
        return x

    def solve(self, slopes, x0, iters):
        jac = self.jacobi(self.g["alpha"]) if self.g["precond"] else None
        return self.cg(self.normal, self.rhs(slopes), x0, iters, jac)

    # mirrors
    def fit(self):
        if self._fit is None:
            f, dev = self.g["fitting"], _dev()
            n, d, dx = f["n_sub"], f["d_sub"], self.g["layers"][0]["dx"]
            th = torch.tensor(f["directions"], dtype=torch.float64, device=dev)
            r = (torch.arange(n + 1, dtype=torch.float64, device=dev) - n / 2.0) * d
            act = next(s["act"] for s in self.sens if s["w"]["n_sub"] == n)
            mir = [[_linear((r[None] + m["altitude"] * th[:, a:a + 1]) / m["pitch"] + (m["n"] - 1) / 2.0, m["n"], False)
                    for a in (0, 1)] for m in f["dms"]]
            lay = [[_linear((r[None] + h * th[:, a:a + 1]) / dx + self.N / 2.0, self.N, True) for a in (0, 1)]
                   for h in self.alt.tolist()]
            self._fit = (mir, lay, act, [m["n"] for m in f["dms"]])
        return self._fit

    def _split(self, a):
        ns = self.fit()[3]
        return [x.view(n, n) for x, n in zip(a.split([n * n for n in ns]), ns)]

    def mirror(self, a):
        mir, _, act, _ = self.fit()
        return sum(by @ A @ bx.transpose(1, 2) for (bx, by), A in zip(mir, self._split(a))) * act

    def mirror_t(self, u):
        mir, _, act, _ = self.fit()
        return torch.cat([(by.transpose(1, 2) @ (u * act) @ bx).sum(0).flatten() for bx, by in mir])

    def project(self, phi):
        _, lay, act, _ = self.fit()
        return sum(by @ p @ bx.transpose(1, 2) for (bx, by), p in zip(lay, phi)) * act

    def fitting(self, phi, a0, iters):
        return self.cg(lambda a: self.mirror_t(self.mirror(a)), self.mirror_t(self.project(phi)), a0, iters)

    def mirror_slopes(self, a):
        out = []
        for s in self.sens:
            w, psi = s["w"], 0.0
            for m, A in zip(self.g["fitting"]["dms"], self._split(a)):
                cone = 1.0 - m["altitude"] / w["height"] if s["lgs"] else 1.0
                bx, by = [_linear((cone * s["r"] + t * m["altitude"]) / m["pitch"] + (m["n"] - 1) / 2.0, m["n"], False)
                          for t in w["theta"]]
                psi = psi + by @ A @ bx.T
            out.append(self.pack(s, *self.fried(s, psi * s["act"])))
        return torch.cat(out)

    def residual_rms(self, phi, a):
        act = self.fit()[2]
        u = (self.project(phi) - self.mirror(a)).flatten(1)[:, act.flatten() > 0]
        return (u - u.mean(1, keepdim=True)).square().mean(1).sqrt()

    # inputs
    def screens(self, gen, times):
        """Frozen-flow von Karman layers [L, N, N] at each time."""
        N, dx, dev = self.N, self.g["layers"][0]["dx"], _dev()
        f = torch.fft.fftfreq(N, d=dx, dtype=torch.float64, device=dev)
        fy, fx = f[:, None], f[None, :]
        k2 = fx ** 2 + fy ** 2 + L0 ** -2.0
        cn2 = torch.tensor(self.g["cn2"], dtype=torch.float64, device=dev)
        amp = torch.sqrt(0.023 * R0 ** (-5 / 3) * cn2[:, None, None] * k2 ** (-11 / 6)) / (N * dx)
        amp[:, 0, 0] = 0.0
        F = amp * torch.complex(*[torch.randn(self.L, N, N, dtype=torch.float64, device=dev, generator=gen)
                                  for _ in range(2)])
        wind = torch.rand(2, self.L, dtype=torch.float64, device=dev, generator=gen)
        speed, ang = 5.0 + 15.0 * wind[0], 2.0 * math.pi * wind[1]
        vx, vy = (speed * torch.cos(ang))[:, None, None], (speed * torch.sin(ang))[:, None, None]
        return [torch.fft.ifft2(F * torch.exp(-2j * math.pi * (fx * vx + fy * vy) * t)).real * N * N for t in times]

    def noisy(self, gen, slopes):
        sig = torch.cat([torch.full((m,), s["w"]["sigma"], dtype=torch.float64, device=slopes.device)
                         for m, s in zip(self.n_meas, self.sens)])
        return slopes + sig * torch.randn(len(sig), dtype=torch.float64, device=slopes.device, generator=gen)


def _gen(seed, member=0):
    return torch.Generator(device=_dev()).manual_seed(1_000_003 * (int(seed) % (1 << 40)) + member)


def _frame_inputs(case, seed, member=0):
    """(model, slopes, x0) of one frame: x0 the previous frame's cold solution, or zero."""
    m = Model(geometry(case))
    gen, dt = _gen(seed, member), torch.float64 if case["precision"] else torch.float32
    prev, now = m.screens(gen, (0.0, FRAME_S))
    s0, s1 = m.noisy(gen, m.measure(prev)), m.noisy(gen, m.measure(now)).to(dt)
    x0 = torch.zeros(m.L * m.N * m.N, dtype=torch.float64, device=_dev())
    if case.get("warm", True):
        x0 = m.solve(s0, x0, case["iters"])
    return m, s1, x0.to(dt)


def _control_inputs(case, seed):
    """(model, slopes, x0, a_rec, a_tm2, a_tm1): a loop that has followed the turbulence for a while."""
    m = Model(geometry(case))
    gen, dt = _gen(seed), torch.float64 if case["precision"] else torch.float32
    prev, now = m.screens(gen, (0.0, FRAME_S))
    x0 = m.solve(m.noisy(gen, m.measure(prev)), torch.zeros(m.L * m.N * m.N, dtype=torch.float64, device=_dev()),
                 case["iters"])
    a = m.fitting(m.synthesis(x0), torch.zeros(sum(n * n for n in m.fit()[3]), dtype=torch.float64, device=_dev()),
                  case["fit_iters"])
    a2, a1 = (0.9 * a).to(dt), (0.95 * a).to(dt)
    s = m.noisy(gen, m.measure(now) - m.mirror_slopes(a2.double())).to(dt)
    return m, s, x0.to(dt), a.to(dt), a2, a1


def _plant_inputs(case, seed):
    """(model, layers, commands): true layers and the commands that fit them roughly."""
    m = Model(geometry(case))
    gen, dt = _gen(seed), torch.float64 if case["precision"] else torch.float32
    prev, now = m.screens(gen, (0.0, FRAME_S))
    a = m.fitting(prev, torch.zeros(sum(n * n for n in m.fit()[3]), dtype=torch.float64, device=_dev()), 3)
    return m, now.flatten().to(dt), a.to(dt)


def _serve_frames(case, seed):
    """Per telescope (model, frames): host slopes of 8 consecutive frames."""
    out = []
    for i, c in enumerate(_members(case)):
        m, gen = Model(geometry(c)), _gen(seed, i)
        scr = m.screens(gen, [FRAME_S * k for k in range(8)])
        out.append((m, [m.noisy(gen, m.measure(p)).float().cpu().numpy() for p in scr]))
    return out


def _alpha(seed):
    return float(0.5 * 4.0 ** np.random.default_rng(int(seed) % (1 << 40)).random())


# ---------------------------------------------------------------- the cases

def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        flat, plans, slopes, x0 = 0, [], [], []
        for i, c in enumerate(_members(case)):
            c = dict(c, iters=case["iters"])
            plans.append(tomo.Plan(geometry(c), cluster_size=case["cluster"], transforms=case["transforms"]))
            _, s, x = _frame_inputs(c, seed, i)
            slopes.append(s)
            x0.append(x)
        start = torch.cat(x0)
        x = torch.empty_like(start)
        return {"kind": kind, "plans": plans, "slopes": slopes, "start": start, "x": x,
                "xs": list(x.split([p.n for p in plans])), "iters": case["iters"]}
    if kind == "serve":
        srv = tomo.Server(iters=case["iters"], max_in_flight=4, queue_depth=64, result_slots=2)
        ids = [srv.admit(geometry(c), cluster_size=case["cluster"], transforms=case["transforms"])
               for c in _members(case)]
        return {"kind": kind, "server": srv, "ids": ids, "frames": [f for _, f in _serve_frames(case, seed)], "k": 0}
    plan = tomo.Plan(geometry(case))
    st = {"kind": kind, "plan": plan}
    if kind == "frame":
        _, slopes, x0 = _frame_inputs(case, seed)
        st.update(slopes=slopes, start=x0, x=torch.empty_like(x0), iters=case["iters"], warm=case["warm"])
    elif kind == "normal":
        x = _frame_inputs(dict(case, iters=3, warm=True), seed)[2]
        st.update(x=x, out=torch.empty_like(x))
    elif kind == "jacobi":
        st.update(out=torch.empty(plan.n, dtype=torch.float64, device=_dev()), alpha=_alpha(seed))
    else:
        fit = tomo.Fit(plan, geometry(case)["fitting"])
        st.update(fit=fit)
        if kind == "control":
            _, slopes, x0, a_rec, a2, a1 = _control_inputs(case, seed)
            start = torch.cat([x0, a_rec])
            cur = torch.empty_like(start)
            st.update(slopes=slopes, start=start, cur=cur, x=cur[:plan.n], a_rec=cur[plan.n:], a2=a2, a1=a1,
                      a=torch.empty_like(a1), gain=case["gain"], iters=case["iters"], fit_iters=case["fit_iters"])
        else:
            _, layers, a = _plant_inputs(case, seed)
            if kind == "fit":
                st.update(layers=layers, start=a, a=torch.empty_like(a), fit_iters=case["fit_iters"])
            else:
                st.update(layers=layers, a=a, s=torch.empty(plan.n_slopes, dtype=plan.dtype, device=_dev()),
                          out=torch.empty(plan.n_slopes, dtype=plan.dtype, device=_dev()),
                          rms=torch.empty(25, dtype=torch.float64, device=_dev()))
    return st


def run(st):
    """One pass.  A warm start is copied from the kept previous solution, so that a pass can be repeated."""
    kind = st["kind"]
    if kind == "frame":
        if st["warm"]:
            st["x"].copy_(st["start"])
        st["plan"].solve(st["slopes"], st["x"], st["iters"], warm=st["warm"])
        return st["x"]
    if kind == "normal":
        st["plan"].apply_normal(st["x"], st["out"])
        return st["out"]
    if kind == "batch":
        st["x"].copy_(st["start"])
        tomo.solve_batch(st["plans"], st["slopes"], st["xs"], st["iters"])
        return st["xs"]
    if kind == "control":
        st["cur"].copy_(st["start"])
        st["fit"].polc_step(st["slopes"], st["x"], st["a_rec"], st["a2"], st["a1"], st["a"], st["gain"], st["iters"],
                            st["fit_iters"])
        return [st["x"], st["a_rec"], st["a"]]
    if kind == "fit":
        st["a"].copy_(st["start"])
        st["fit"].solve(st["layers"], st["a"], st["fit_iters"])
        return st["a"]
    if kind == "plant":
        st["plan"].layers_to_slopes(st["layers"], st["s"])
        st["fit"].mirror_slopes(st["a"], st["out"], slopes_in=st["s"], scale=-1.0)
        st["fit"].residual_rms(st["layers"], st["a"], st["rms"])
        return [st["out"], st["rms"]]
    if kind == "jacobi":
        st["plan"].jacobi_diagonal_noalloc(st["out"], st["alpha"])
        return st["out"]
    srv, k = st["server"], st["k"]
    st["k"] = k + 1
    for t, f in zip(st["ids"], st["frames"]):
        srv.submit(t, f[k % len(f)], k)
    srv.drain()
    done = {r["telescope"]: r for r in srv.poll()}
    return [srv.result(t, done[t]["result_slot"], k) for t in st["ids"]]


def exact(case, seed):
    kind = case["kind"]
    if kind == "frame":
        m, s, x0 = _frame_inputs(case, seed)
        return m.solve(s.double(), x0.double(), case["iters"])
    if kind == "normal":
        m, _, x = _frame_inputs(dict(case, iters=3, warm=True), seed)
        return m.normal(x.double())
    if kind == "batch":
        out = []
        for i, c in enumerate(_members(case)):
            m, s, x0 = _frame_inputs(dict(c, iters=case["iters"]), seed, i)
            out.append(m.solve(s.double(), x0.double(), case["iters"]))
        return out
    if kind == "control":
        m, s, x0, a_rec, a2, a1 = _control_inputs(case, seed)
        x = m.solve(s.double() + m.mirror_slopes(a2.double()), x0.double(), case["iters"])
        a = m.fitting(m.synthesis(x), a_rec.double(), case["fit_iters"])
        return [x, a, a1.double() + case["gain"] * (a - a2.double())]
    if kind in ("fit", "plant"):
        m, layers, a = _plant_inputs(case, seed)
        phi = layers.double().view(m.L, m.N, m.N)
        if kind == "fit":
            return m.fitting(phi, a.double(), case["fit_iters"])
        return [m.measure(phi) - m.mirror_slopes(a.double()), m.residual_rms(phi, a.double())]
    if kind == "jacobi":
        return Model(geometry(case)).jacobi(_alpha(seed))
    out = []
    for m, f in _serve_frames(case, seed):
        s = torch.from_numpy(f[0]).to(_dev()).double()
        out.append(m.solve(s, torch.zeros(m.L * m.N * m.N, dtype=torch.float64, device=_dev()), case["iters"]))
    return out


def _sizes(case):
    """(element bytes, coefficients, slopes, corner values traced per operator, sensors, layers)."""
    e, n = 8 if case["precision"] else 4, case["layers"] * case["N"] ** 2
    S = float(_pupil(case["n_sub"], case["d_sub"], case["n_sub"] * case["d_sub"], case["obstruction"]).sum())
    full = case["lgs"] + case["ngs"]
    return e, n, 2 * S * full + 2 * case["tt"], S, full, case["layers"]


def _operator_flops(case):
    """Bilinear trace and its transpose per (sensor, layer, point), slopes, and both 2-D transforms."""
    _, n, _, S, full, L = _sizes(case)
    lf = 2 * case["order"]
    return full * S * (L * (2 * 11) + 30) + 2 * (4 * lf * n * (1 - 0.25 ** case["levels"]) / 0.75)


def _solve_work(case, iters, warm):
    """Inputs and outputs once; per iteration x, r, p read and written and J^-1 read (CG's own recurrences)."""
    e, n, ns, *_ = _sizes(case)
    per = (7 if case["precond"] else 6) * n
    return (e * (ns + n * (2 if warm else 1) + iters * per), (iters + 1) * _operator_flops(case) + iters * 14 * n)


def work(case):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        parts = [_solve_work(c, case["iters"], True) for c in _members(case)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    e, n, ns, S, full, L = _sizes(case)
    if kind == "frame":
        b, f = _solve_work(case, case["iters"], case["warm"])
    elif kind == "normal":
        b, f = 2 * e * n, _operator_flops(case)
    elif kind == "jacobi":
        # per coefficient and laser guide star: products over the support's rows and columns of the pupil
        b, f = 8 * n, n * case["lgs"] * 8 * case["n_sub"] * 0.5
    else:
        acts = sum((2 * int(math.ceil((case["n_sub"] * case["d_sub"] / 2 + h * ARCMIN) / p)) + 3) ** 2
                   for h, p in FIT_DMS)
        trace = 25 * S * (11 * L + 11 * len(FIT_DMS))
        if kind == "plant":
            b, f = e * (n + acts + ns), full * S * 11 * (L + len(FIT_DMS)) + trace
        else:
            fb, ff = e * (n + 2 * acts), 2 * trace + case["fit_iters"] * acts * 2 * 200
            if kind == "fit":
                b, f = fb, ff
            else:
                sb, sf = _solve_work(case, case["iters"], True)
                b, f = sb + e * 5 * acts, sf + ff
    return {"bytes": b, "flops": f}
