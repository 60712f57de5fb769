"""Timed cases of the library: what its users run, through the public binding.

Four kinds of work, with sizes from the workload definitions, the tests and the benchmark:

* ``single``  one instance advanced by a number of SSP-RK3 steps, then its moments (one flow studied
  in detail: the cylindrical and spherical workloads, the paper's large radial orders);
* ``sweep``   a parameter sweep in one batched handle: instances of different size and physics on the
  16 x 8 x 8 quadrature, FP32, stepped together, then every instance's moments;
* ``steady``  many small instances run towards their steady states with residual checks (the training
  and held-out sets of the warm start, the dense gas at rest), FP32, or FP64 as in the polish;
* ``net``     the warm-start network: inference, or loss and gradients of a training batch.

`prepare` gives each instance a state on its way to the steady one: wall-to-wall profiles of n, u_2
and T with a smooth modulation of every momentum, a few per cent deep, from the seed.  Passes on one
state continue the run.  Moments of FP32 runs are kept in FP32.

`exact` is the method restated in FP64 torch, independent of the package: quadratures, derivative
matrices, Fischer-Methfessel weights, closure, WENO5 advection, curvature force, collision, walls and
the RK scheme, for instances of equal cell count stacked along a leading axis.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2403_15051_gb300 import fdlb
from paper_2403_15051_gb300 import workloads as wl

CYL, SPH, CYL_Z = wl.CYL, wl.SPH, wl.CYL_Z
EXACT_UPDATES = 2.5e10  # population updates (per stage) beyond which exact() takes too long


# ------------------------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest run: plane-like Couette flow, 64 cells x 128 momenta, FP64, latency-bound
        dict(name="couette_64_fp64", kind="single", geometry=CYL, n_cells=64, R_out=2.0, beta=0.0, Q_R=4, Q_2=4, Q_3=4,
             Kn=0.1, sigma=0.0, eta0=0.1, T_out=1.0, u_in=0.1, dt=1e-3, precision="fp64", steps=40),
        # one instance at production resolution between cylinders, stretched grid
        dict(name="fourier_cyl_1024", kind="single", geometry=CYL, n_cells=1024, R_out=3.0, beta=1.5, Q_R=8, Q_2=8, Q_3=8,
             Kn=0.05, sigma=0.0, eta0=0.2, T_out=1.1, u_in=0.0, dt=0.0, precision="fp32", steps=40),
        # one instance between spheres, the largest momentum set
        dict(name="fourier_sph_2048", kind="single", geometry=SPH, n_cells=2048, R_out=4.0, beta=0.0, Q_R=12, Q_2=12,
             Q_3=12, Kn=0.03464, sigma=0.0, eta0=0.3, T_out=1.2, u_in=0.0, dt=0.0, precision="fp32", steps=20),
        # dense Couette flow on the paper's quadrature of radial order 20 (Sec. IV)
        dict(name="couette_q20", kind="single", geometry=CYL, n_cells=240, R_out=11.0, beta=0.0, Q_R=20, Q_2=8, Q_3=8,
             Kn=0.0, sigma=1.0, eta0=0.1, T_out=1.0, u_in=1.0, dt=0.0, precision="fp32", steps=20),
        # the same flow with p_z integrated out, at the paper's resolution of 24 cells per sigma
        dict(name="couette_reduced_q20", kind="single", geometry=CYL_Z, n_cells=96, R_out=5.0, beta=0.0, Q_R=20, Q_2=8,
             Q_3=0, Kn=0.0, sigma=1.0, eta0=0.1, T_out=1.0, u_in=1.0, dt=0.0, precision="fp32", steps=40),
        # a parameter sweep of a dozen flows, and one of a study's size
        dict(name="sweep_12", kind="sweep", instances=12, draw_seed=1, lo=128, hi=2048, steps=20),
        dict(name="sweep_128", kind="sweep", instances=128, draw_seed=0, lo=128, hi=2048, steps=8),
        # training set of the warm start: many small flows towards steady state, FP32
        dict(name="steady_256_fp32", kind="steady", geometry=CYL, instances=256, cells=64, draw_seed=1, precision="fp32",
             steps=100, check_every=50),
        # the FP64 polish of such a set
        dict(name="polish_48_fp64", kind="steady", geometry=CYL, instances=48, cells=64, draw_seed=2, precision="fp64",
             steps=40, check_every=20),
        # the dense gas at rest between spheres (27 instances of 96, 168 and 240 cells)
        dict(name="layering_sph_fp32", kind="steady", geometry=SPH, instances=27, cells=0, draw_seed=0, precision="fp32",
             steps=60, check_every=30),
        # the warm-start network: profiles of a held-out set, and one training batch
        dict(name="net_forward_64", kind="net", grad=False, batch=64, width=64, modes=6, layers=4, hidden=128, points=256),
        dict(name="net_train_32", kind="net", grad=True, batch=32, width=64, modes=6, layers=4, hidden=128, points=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["single", "single", "single", "sweep", "steady", "steady", "net"])
    if kind == "single":
        geometry = rng.choice([CYL, CYL, SPH, CYL_Z])
        orders = {CYL: [(4, 4, 4), (5, 5, 5), (6, 6, 6), (8, 8, 8), (8, 8, 8), (12, 8, 8), (20, 8, 8)],
                  SPH: [(4, 4, 4), (5, 5, 5), (8, 8, 8), (12, 12, 12), (12, 12, 12)],
                  CYL_Z: [(8, 8, 0), (20, 8, 0)]}[geometry]
        Q_R, Q_2, Q_3 = rng.choice(orders)
        n_cells = _log_int(rng, 32, 1024 if Q_R < 20 or geometry == CYL_Z else 300)
        by_sigma = rng.random() < 0.4
        gap = rng.uniform(3.5, 8.0) if by_sigma else rng.uniform(1.0, 3.0)
        precision = "fp64" if rng.random() < 0.35 and 2 * Q_R * Q_2 * max(Q_3, 2) * n_cells < 4e5 else "fp32"
        u_in = 0.0 if geometry == SPH else rng.choice([0.0, 0.1, 0.3])
        return dict(kind=kind, geometry=geometry, n_cells=n_cells, R_out=1.0 + gap, beta=rng.choice([0.0, 0.0, 1.5]),
                    Q_R=Q_R, Q_2=Q_2, Q_3=Q_3, Kn=0.0 if by_sigma else 0.05, sigma=1.0 if by_sigma else 0.0,
                    eta0=rng.choice([0.05, 0.1, 0.2]), T_out=rng.uniform(1.0, 1.2), u_in=u_in, dt=0.0,
                    precision=precision, steps=rng.choice([1, 7, 20, 33]))
    if kind == "sweep":
        lo = rng.choice([64, 128])
        return dict(kind=kind, instances=_log_int(rng, 2, 80), draw_seed=rng.randrange(1 << 20), lo=lo,
                    hi=rng.choice([4, 12, 16]) * lo, steps=rng.choice([3, 5, 8]))
    if kind == "steady":
        precision = rng.choice(["fp32", "fp32", "fp64"])
        check = rng.choice([10, 20, 25] if precision == "fp32" else [10, 20])
        return dict(kind=kind, geometry=rng.choice([CYL, CYL, SPH]),
                    instances=_log_int(rng, 4, 400 if precision == "fp32" else 28), cells=rng.choice([48, 64, 81, 100]),
                    draw_seed=rng.randrange(1 << 20), precision=precision, steps=2 * check, check_every=check)
    return dict(kind=kind, grad=rng.random() < 0.6, batch=_log_int(rng, 1, 64), width=rng.choice([32, 64]),
                modes=rng.choice([4, 6]), layers=rng.choice([2, 4]), hidden=rng.choice([64, 128]),
                points=rng.choice([64, 128, 256]))


def _instances(case):
    """The workload dictionaries of a case."""
    if case["kind"] == "single":
        c = case
        return [dict(geometry=c["geometry"], R_in=1.0, R_out=c["R_out"], n_cells=c["n_cells"], beta=c["beta"], Q_R=c["Q_R"],
                     Q_2=c["Q_2"], Q_3=c["Q_3"], Kn=c["Kn"] or None, sigma=c["sigma"] or None, eta0=c["eta0"],
                     T_wall=(1.0, c["T_out"]), u_wall=(c["u_in"], 0.0), dt=c["dt"] or None, precision=c["precision"])]
    accept = lambda kn, eta0, *_: _confinement(kn, eta0) >= 3.0  # noqa: E731
    if case["kind"] == "sweep":
        return wl.batch_instances(accept, n=case["instances"], seed=case["draw_seed"], n_lo=case["lo"], n_hi=case["hi"])
    if case["cells"] == 0:
        return wl.layering_instances(case["geometry"], precision=case["precision"])[:case["instances"]]
    out = wl.batch_instances(accept, n=case["instances"], seed=case["draw_seed"], n_lo=case["cells"], n_hi=case["cells"])
    for d in out:
        d.update(geometry=case["geometry"], Q_R=4, Q_2=4, Q_3=4, precision=case["precision"])
        if case["geometry"] == SPH:
            d.update(u_wall=(0.0, 0.0))
    return out


def work(case):
    if case["kind"] == "net":
        B, W, m, L, H, P = (case[k] for k in ("batch", "width", "modes", "layers", "hidden", "points"))
        rows = B * P
        fwd = 2.0 * rows * (6 * W + L * W * W + W * H + 4 * H) + L * (2 * 2.0 * B * 2 * m * W * P + 8.0 * B * m * W * W)
        n_par = 6 * W + W + L * (2 * m * W * W + W * W + W) + W * H + H + 4 * H + 4
        return {"bytes": 4.0 * (n_par * (2 if case["grad"] else 1) + rows * 4 + 5 * B), "flops": fwd * (3 if case["grad"] else 1)}
    flops = state = moments = 0.0
    for d in _instances(case):
        nR, n2, n3 = 2 * d["Q_R"], d["Q_2"], 2 if d["geometry"] == CYL_Z else d["Q_3"]
        sph = d["geometry"] == SPH
        # WENO5, flux difference, force, collision, RK, moment sums per population and stage
        per = 76 + 5 + 2 * nR + 2 * n2 + (2 * n3 + 13 if sph else 5) + 52 + 5 + 30
        pops = d["n_cells"] * nR * n2 * n3
        flops += 3.0 * case["steps"] * pops * per
        state += pops * (8 if d["precision"] == "fp64" else 4)
        moments += d["n_cells"] * 72.0
    return {"bytes": 2.0 * state + moments, "flops": flops}


# ------------------------------------------------------------------------------- inputs
def _profiles(P, gen):
    """n, u_2, T per cell of a flow on its way to steady state ([B][N])."""
    r = lambda *s: torch.rand(*s, generator=gen, device=P.dev, dtype=torch.float64)  # noqa: E731
    B = P.R_c.shape[0]
    x = P.x_c
    a, ph = 0.05 + 0.05 * r(3, B, 1), 2.0 * math.pi * r(3, B, 1)
    n = P.n0[:, None] * (1.0 + a[0] * torch.sin(2.0 * math.pi * x + ph[0]))
    T = P.Tw[:, :1] + (P.Tw[:, 1:] - P.Tw[:, :1]) * x + 0.2 * a[1] * torch.sin(math.pi * x)
    u2 = P.uw[:, :1] * (1.0 - x) * (0.5 + 0.5 * r(B, 1)) + (0.0 if P.geometry == SPH else 0.05) * a[2] * torch.sin(math.pi * x)
    return n, u2, T


def _initial(P, gen):
    """Populations [B][N][k][i][j] in FP64: the discrete Maxwellian of the profiles, every momentum
    modulated by a smooth wave along the radius."""
    n, u2, T = _profiles(P, gen)
    z = torch.zeros_like(n)
    g3 = torch.stack([torch.ones_like(T), T], -1) if P.reduced else _g_full(P.p3, P.w3, z, T)
    f = n[..., None, None, None] * g3[..., :, None, None] * _g_half(P, z, T)[..., None, :, None] \
        * _g_full(P.p2, P.w2, u2, T)[..., None, None, :]
    shape = f.shape[:1] + (1,) + f.shape[2:]
    wave = torch.randint(1, 4, shape, generator=gen, device=P.dev).double()
    phase = 2.0 * math.pi * torch.rand(shape, generator=gen, device=P.dev, dtype=torch.float64)
    if P.reduced:  # the pair (phi, chi) moves together
        wave, phase = wave[:, :, :1], phase[:, :, :1]
    return f * (1.0 + 0.02 * torch.sin(2.0 * math.pi * wave * P.x_c[..., None, None, None] + phase))


def _groups(ds):
    """Instances of equal shape, as lists of indices (at most 64 to a group, fewer when large)."""
    by = {}
    for q, d in enumerate(ds):
        by.setdefault(d["n_cells"], []).append(q)
    out = []
    for n, qs in by.items():
        per = max(1, min(64, 4_000_000 // (n * 2 * ds[0]["Q_R"] * ds[0]["Q_2"] * max(2, ds[0]["Q_3"]))))
        out += [qs[a:a + per] for a in range(0, len(qs), per)]
    return out


def _states(ds, seed, dev, weights):
    """(indices, problem, initial populations) of every group; the same numbers for prepare and exact."""
    for k, qs in enumerate(_groups(ds)):
        gen = torch.Generator(device=dev)
        gen.manual_seed(1_000_003 * (int(seed) % 1_000_000_007) + k)
        P = _Problem([ds[q] for q in qs], dev, weights)
        yield qs, P, _initial(P, gen)


def _element(precision):
    return torch.float64 if precision == "fp64" else torch.float32


def prepare(case, seed):
    if case["kind"] == "net":
        raw, target, theta = _net_inputs(case, seed)
        net = fdlb.WarmStartNet(case["width"], case["modes"], case["layers"], case["hidden"], case["points"],
                                max_batch=case["batch"])
        net.set_params(theta)
        return {"kind": "net", "net": net, "raw": raw, "target": target, "grad": case["grad"]}
    ds = _instances(case)
    S = fdlb.Solver(ds)
    dt = _element(ds[0]["precision"])
    size = torch.empty((), dtype=dt).element_size()
    cells = [d["n_cells"] for d in ds]
    off, at = [], 0
    for q in range(len(ds)):  # each instance's populations start on a 256-byte boundary
        off.append(at)
        at += -(-S.raw_elements(q) * size // 256) * (256 // size)
    f = torch.zeros(S.state_bytes() // size, dtype=dt, device="cuda")
    for qs, _, f0 in _states(ds, seed, f.device, False):
        for b, q in enumerate(qs):
            f[off[q]:off[q] + f0[b].numel()] = f0[b].reshape(-1).to(dt)
    S.set_state_raw(f.data_ptr(), -1, on_device=True)
    torch.cuda.synchronize()
    return {"kind": case["kind"], "S": S, "steps": case["steps"], "check": case.get("check_every", 0), "f": f,
            "moments": torch.empty(sum(cells), fdlb.NMOM, dtype=torch.float64, device="cuda"), "dtype": dt}


def run(state):
    if state["kind"] == "net":
        if state["grad"]:
            loss, grad = state["net"].loss_grad(state["raw"], state["target"])
            return {"loss": loss, "grad": grad}
        return {"profiles": state["net"].forward(state["raw"])}
    S = state["S"]
    out = {}
    if state["kind"] == "steady":
        _, out["taken"], _ = S.run_to_steady(tol=1e-30, max_steps=state["steps"], check_every=state["check"])
    else:
        S.step(state["steps"])
    S.moments_device(-1, state["moments"].data_ptr())
    S.get_state_raw(state["f"].data_ptr(), -1, on_device=True)
    out["f"] = state["f"]
    out["moments"] = state["moments"].to(state["dtype"])
    return out


# ------------------------------------------------------------------------------- the method in FP64
def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if case["kind"] == "net":
        return _net_exact(case, seed, dev)
    ds = _instances(case)
    dt = _element(ds[0]["precision"])
    pops = [d["n_cells"] * 2 * d["Q_R"] * d["Q_2"] * (2 if d["geometry"] == CYL_Z else d["Q_3"]) for d in ds]
    if 3.0 * case["steps"] * (sum(pops) + 4e5 * len(_groups(ds))) > EXACT_UPDATES:
        return None
    align = 32 if dt == torch.float64 else 64
    off = np.concatenate([[0], np.cumsum([-(-p // align) * align for p in pops])])
    cell = np.concatenate([[0], np.cumsum([d["n_cells"] for d in ds])])
    f_all = torch.zeros(int(off[-1]), dtype=torch.float64, device=dev)
    m_all = torch.empty(int(cell[-1]), 9, dtype=torch.float64, device=dev)
    for qs, P, f in _states(ds, seed, dev, True):
        f = f.to(dt).double()  # the populations as the handle is given them
        for _ in range(case["steps"]):
            f1 = f + P.dt * _rhs(P, f)
            f2 = 0.75 * f + 0.25 * (f1 + P.dt * _rhs(P, f1))
            f = f / 3.0 + 2.0 / 3.0 * (f2 + P.dt * _rhs(P, f2))
        n, u, T, q, S = _macroscopic(P, f)
        m = torch.cat([n[..., None], u, T[..., None], q, (S[..., 7] - n * u[..., 0] * u[..., 1])[..., None]], -1)
        for b, k in enumerate(qs):
            f_all[int(off[k]):int(off[k]) + pops[k]] = f[b].reshape(-1)
            m_all[int(cell[k]):int(cell[k + 1])] = m[b]
    return {"taken": None, "f": f_all, "moments": m_all} if case["kind"] == "steady" else {"f": f_all, "moments": m_all}


def _chi(eta):
    return (2.0 - eta) / (2.0 * (1.0 - eta) ** 3)


def _confinement(kn, eta0):
    return 1.0 / (6.0 * math.sqrt(2.0) * eta0 * _chi(eta0) * kn)


def _hermite(x, L):
    He = [np.ones_like(x), x]
    for n in range(1, L):
        He.append(x * He[n] - n * He[n - 1])
    return np.stack(He[:L + 1])


def _full_rule(Q):
    """Q-point Gauss-Hermite rule of the normal weight and the matrix of d(f p)/dp on it (Eq. force2)."""
    x, w = np.polynomial.hermite_e.hermegauss(Q)
    w = w / w.sum()
    He = _hermite(x, Q)
    K = np.zeros((Q, Q))
    for l in range(Q - 1):
        K -= np.outer(w * He[l + 1], He[l + 1] + (l * He[l - 1] if l else 0.0)) / math.factorial(l)
    return x, w, K


def _half_polys(x, a, b, L):
    """h_0 .. h_L, orthonormal under the normal weight on the half line, and their derivatives."""
    h, d = [np.full_like(x, 1.0 / b[0])], [np.zeros_like(x)]
    for l in range(L):
        h.append(((x - a[l]) * h[l] - (b[l] * h[l - 1] if l else 0.0)) / b[l + 1])
        d.append((h[l] + (x - a[l]) * d[l] - (b[l] * d[l - 1] if l else 0.0)) / b[l + 1])
    return np.stack(h), np.stack(d)


def _half_rule(Q):
    """Nodes and weights (positive half first), recurrence (a, b = sqrt(beta)), d/dp matrix (Eq. force1)."""
    g, gw = np.polynomial.legendre.leggauss(24)
    edges = np.linspace(0.0, 12.0 + 2.0 * math.sqrt(2.0 * Q), 161)
    h = 0.5 * np.diff(edges)[:, None]
    x = (0.5 * (edges[1:] + edges[:-1])[:, None] + h * g).ravel()
    w = (h * gw).ravel() * np.exp(-0.5 * x * x) / math.sqrt(2.0 * math.pi)
    a, b = np.zeros(Q + 1), np.zeros(Q + 2)
    prev, cur = np.zeros_like(x), np.ones_like(x)
    b[0] = math.sqrt(w.sum())
    cur = cur / b[0]
    for l in range(Q + 1):
        a[l] = (w * x * cur * cur).sum()
        nxt = (x - a[l]) * cur - (b[l] * prev if l else 0.0)
        b[l + 1] = math.sqrt((w * nxt * nxt).sum())
        prev, cur = cur, nxt / b[l + 1]
    J = np.diag(a[:Q]) + np.diag(b[1:Q], 1) + np.diag(b[1:Q], -1)
    xn = np.sort(np.linalg.eigvalsh(J))
    for _ in range(2):
        H, D = _half_polys(xn, a, b, Q)
        xn = xn - H[Q] / D[Q]
    H, D = _half_polys(xn, a, b, Q - 1)
    wn = 1.0 / (H * H).sum(0)
    p, w2 = np.concatenate([xn, -xn]), np.concatenate([wn, wn])
    H2, D2 = np.concatenate([H, H], 1), np.concatenate([D, D], 1)
    s = np.sign(p)
    phi0 = _half_polys(np.zeros(1), a, b, Q - 1)[0][:, 0] @ H2
    K = -(s * w2)[:, None] * (np.outer(phi0, phi0) / (2.0 * math.sqrt(2.0 * math.pi)) + (s[:, None] == s[None]) * (H2.T @ D2))
    return p, w2, a, b, K


class _Problem:
    """Instances of equal cell count and momentum set; per-instance quantities carry a leading axis."""

    def __init__(self, ds, dev, weights):
        d0 = ds[0]
        t = lambda v: torch.tensor(np.asarray(v), dtype=torch.float64, device=dev)  # noqa: E731
        self.dev, self.geometry, self.reduced = dev, SPH if d0["geometry"] == SPH else CYL, d0["geometry"] == CYL_Z
        pR, wR, self.a, self.b, KR = _half_rule(d0["Q_R"])
        p2, w2, K2 = _full_rule(d0["Q_2"])
        p3, w3, K3 = (np.zeros(2), np.ones(2), np.zeros((2, 2))) if self.reduced else _full_rule(d0["Q_3"])
        self.QR = d0["Q_R"]
        self.pR, self.wR, self.KR, self.p2, self.w2, self.K2, self.p3, self.w3, self.K3 = map(t, (pR, wR, KR, p2, w2, K2, p3, w3, K3))
        NR = min(d0["Q_R"] - 1, 7)
        self.H = t(_half_polys(np.abs(pR), self.a, self.b, NR)[0])  # [N+1][2Q]
        # monomial coefficients of h_0 .. h_NR
        C = np.zeros((NR + 1, NR + 1))
        C[0, 0] = 1.0 / self.b[0]
        for l in range(NR):
            C[l + 1, 1:] = C[l, :-1]
            C[l + 1] -= self.a[l] * C[l] + (self.b[l] * C[l - 1] if l else 0.0)
            C[l + 1] /= self.b[l + 1]
        self.C = t(C)
        self.w = self.w3[:, None, None] * self.wR[None, :, None] * self.w2[None, None, :]
        self.moment_columns()
        N = d0["n_cells"]
        rows = []
        for d in ds:
            gap = d["R_out"] - d["R_in"]
            sigma = d.get("sigma") or gap / _confinement(d["Kn"], d["eta0"])
            n0 = 6.0 * d["eta0"] / (math.pi * sigma ** 3)
            beta, s = d.get("beta") or 0.0, np.concatenate([np.arange(N + 1), np.arange(N) + 0.5]) / N
            R0, L = d["R_in"] + 0.5 * sigma, gap - sigma
            if beta:
                R = R0 + 0.5 * L * (1.0 + np.tanh(beta * (2.0 * s - 1.0)) / math.tanh(beta))
                dR = L * beta / np.cosh(beta * (2.0 * s - 1.0)) ** 2 / math.tanh(beta)
            else:
                R, dR = R0 + L * s, np.full_like(s, L)
            Rf, Rc = R[:N + 1], R[N + 1:]
            A = Rf ** 2 if self.geometry == SPH else Rf
            V = np.diff(Rf ** 3) / 3.0 if self.geometry == SPH else 0.5 * np.diff(Rf ** 2)
            Tm, dt = max(d["T_wall"]), d.get("dt")
            if not dt:
                tau = float(_viscosity(n0, Tm, _chi(d["eta0"]), sigma, math.sqrt)) / (n0 * Tm)
                dt = min(0.4 * np.diff(Rf).min() / (np.abs(pR).max() * math.sqrt(Tm)), 0.5 * tau)
            rows.append((sigma, n0, dt, Rf, Rc, dR[N + 1:], A, V, d["T_wall"], d["u_wall"], (Rc - Rf[0]) / (Rf[-1] - Rf[0])))
        self.sigma, self.n0, dt, self.R_f, self.R_c, self.dRds, self.A, self.V, self.Tw, self.uw, self.x_c = (
            t(np.stack([np.asarray(r[k], dtype=np.float64) for r in rows])) for k in range(11))
        self.dt = dt[:, None, None, None, None]
        self.N = N
        if not weights:
            return
        self.W = torch.stack([_fm_weights(self, b) for b in range(len(ds))])
        z = torch.zeros_like(self.Tw)
        g3 = torch.stack([torch.ones_like(self.Tw), self.Tw], -1) if self.reduced else _g_full(self.p3, self.w3, z, self.Tw)
        self.wall = g3[..., :, None, None] * _g_half(self, z, self.Tw)[..., None, :, None] \
            * _g_full(self.p2, self.w2, self.uw, self.Tw)[..., None, None, :]  # [B][side][k][i][j]

    def moment_columns(self):
        """[k i j][13]: the weights of the raw sums S0, S1_a, S2_ab (00 11 22 01 02 12), S3_a."""
        p3, pR, p2 = (x.expand(len(self.p3), len(self.pR), len(self.p2)).reshape(-1) for x in
                      (self.p3[:, None, None], self.pR[None, :, None], self.p2[None, None, :]))
        sq = pR * pR + p2 * p2 + p3 * p3
        c = [torch.ones_like(pR), pR, p2, p3, pR * pR, p2 * p2, p3 * p3, pR * p2, pR * p3, p2 * p3, sq * pR, sq * p2, sq * p3]
        c = torch.stack(c, -1)
        if self.reduced:  # chi = int p_z^2 f carries S2_zz and the p_z^2 p_a part of S3_a alone
            half = c.shape[0] // 2
            c[half:] = 0.0
            c[half:, 6] = 1.0
            c[half:, 10], c[half:, 11] = pR[half:], p2[half:]
        self.columns = c


def _viscosity(n, T, chi, sigma, sqrt=torch.sqrt):
    br = 2.0 * math.pi / 3.0 * sigma ** 3 * n
    return 5.0 / (16.0 * sigma ** 2) * sqrt(T / math.pi) * (1.0 / chi + 0.8 * br + 0.16 * (1.0 + 12.0 / math.pi) * br ** 2 * chi)


def _g_full(p, w, u, T):
    """Discrete Gaussian on a full-range axis, expanded to order min(Q - 1, 7) (Eq. eq_gak_H)."""
    N = min(len(p) - 1, 7)
    He = [torch.ones_like(p), p]
    for l in range(1, N):
        He.append(p * He[l] - l * He[l - 1])
    out = 0.0
    for l in range(N + 1):
        c = 0.0
        for s in range(l // 2 + 1):
            c = c + (T - 1.0) ** s * u ** (l - 2 * s) / (2.0 ** s * math.factorial(s) * math.factorial(l - 2 * s))
        out = out + c[..., None] * He[l]
    return out * w


def _g_half(P, u, T):
    """Discrete Gaussian on the half-range axis: each half projected on h_0 .. h_N (Eq. eq_gak_hh)."""
    N = P.C.shape[0] - 1
    halves = []
    for s in (1.0, -1.0):
        v = s * u
        m = [0.5 * (1.0 + torch.erf(v / torch.sqrt(2.0 * T)))]
        m.append(v * m[0] + T * torch.exp(-v * v / (2.0 * T)) / torch.sqrt(2.0 * math.pi * T))
        for j in range(1, N):
            m.append(v * m[j] + j * T * m[j - 1])
        M = torch.stack(m[:N + 1], -1) @ P.C.T
        halves.append(M @ (P.H[:, :P.QR] if s > 0 else P.H[:, P.QR:]))
    return torch.cat(halves, -1) * P.wR


def _fm_weights(P, b):
    """Fischer-Methfessel weights of one instance, [N][N]: shares of the ball of radius sigma around a
    cell's radius in every shell (Eq. fm, App. A)."""
    sigma, Rc, Rf = P.sigma[b], P.R_c[b], P.R_f[b]
    d, R = Rc[:, None].expand(P.N, P.N + 1), Rf[None].expand(P.N, P.N + 1)
    U = torch.where(d + sigma <= R, 4.0 / 3.0 * math.pi * sigma ** 3, torch.zeros_like(R))
    part = (d + sigma > R) & (R > d - sigma)
    dp, Rp = d[part], R[part]
    vals = []
    for a in range(0, len(dp), 1 << 19):
        x, y = dp[a:a + (1 << 19)], Rp[a:a + (1 << 19)]
        vals.append(_lens(sigma, y, x) if P.geometry == SPH else _ball_cylinder(sigma, x, y))
    if vals:
        U[part] = torch.cat(vals)
    return 3.0 / (4.0 * math.pi * sigma ** 3) * (U[:, 1:] - U[:, :-1])


def _lens(r1, r2, d):
    v = math.pi * (r1 + r2 - d) ** 2 * (d * d + 2 * d * r2 - 3 * r2 * r2 + 2 * d * r1 + 6 * r1 * r2 - 3 * r1 * r1) / (12.0 * d)
    small = 4.0 / 3.0 * math.pi * torch.minimum(r1.expand_as(r2), r2) ** 3
    return torch.where(d <= (r1 - r2).abs(), small, torch.where(d < r1 + r2, v, torch.zeros_like(v)))


def _ball_cylinder(sigma, d, R):
    """|ball(sigma) at distance d from the axis, inside rho < R|: the circle-circle lens area integrated
    over z = sigma sin t, the t range split where the disc radius crosses |R - d| or R + d."""
    u, wu = np.polynomial.legendre.leggauss(28)
    u, wu = torch.tensor(0.5 * (u + 1.0), device=d.device), torch.tensor(0.5 * wu, device=d.device)
    phi, jac = 0.5 * (1.0 - torch.cos(math.pi * u)), 0.5 * math.pi * torch.sin(math.pi * u) * wu
    cut = lambda r: torch.where((r > 0) & (r < sigma), torch.arccos(torch.clamp(r / sigma, -1.0, 1.0)), torch.zeros_like(r))  # noqa: E731
    t = torch.sort(torch.stack([cut((R - d).abs()), cut(R + d)]), 0).values
    edges = [torch.zeros_like(d), t[0], t[1], torch.full_like(d, 0.5 * math.pi)]
    d, R, out = d[:, None], R[:, None], 0.0
    for lo, hi in zip(edges[:-1], edges[1:]):
        L = (hi - lo)[:, None]
        z = sigma * torch.cos(lo[:, None] + L * phi)  # disc radius, and dz / dt
        c1 = torch.clamp((d * d + z * z - R * R) / (2 * d * z), -1.0, 1.0)
        c2 = torch.clamp((d * d + R * R - z * z) / (2 * d * R), -1.0, 1.0)
        k = (-d + z + R) * (d + z - R) * (d - z + R) * (d + z + R)
        area = z * z * torch.arccos(c1) + R * R * torch.arccos(c2) - 0.5 * torch.sqrt(torch.clamp(k, min=0.0))
        area = torch.where(d <= (R - z).abs(), math.pi * torch.minimum(z, R.expand_as(z)) ** 2,
                           torch.where(d < z + R, area, torch.zeros_like(area)))
        out = out + 2.0 * (area * z * L * jac).sum(1)
    return out


def _macroscopic(P, f):
    S = f.flatten(2) @ P.columns
    n = S[..., 0]
    u = S[..., 1:4] / n[..., None]
    M = S[..., [4, 7, 8, 7, 5, 9, 8, 9, 6]].unflatten(-1, (3, 3))
    tr, uu = S[..., 4] + S[..., 5] + S[..., 6], (u * u).sum(-1)
    T = (tr - n * uu) / (3.0 * n)
    q = 0.5 * (S[..., 10:13] - 2.0 * (M @ u[..., None])[..., 0] - u * tr[..., None] + 2.0 * (n * uu)[..., None] * u)
    return n, u, T, q, S


def _d_dR(P, y):
    """Fourth-order derivative along the radius ([B][N]), one-sided at the two cells next to each wall."""
    d = torch.empty_like(y)
    N = P.N
    d[:, 2:N - 2] = y[:, :N - 4] - 8.0 * y[:, 1:N - 3] + 8.0 * y[:, 3:N - 1] - y[:, 4:]
    e = y.new_tensor([[-25.0, 48.0, -36.0, 16.0, -3.0], [-3.0, -10.0, 18.0, -6.0, 1.0]])
    d[:, :2] = y[:, :5] @ e.T
    d[:, [N - 1, N - 2]] = -(y[:, [N - 1, N - 2, N - 3, N - 4, N - 5]] @ e.T)
    return d * N / 12.0 / P.dRds


def _weno(a, b, c, d, e):
    q = lambda x, y: 13.0 / 12.0 * x * x + 0.25 * y * y + 1e-6  # noqa: E731
    w0 = 0.1 / q(a - 2 * b + c, a - 4 * b + 3 * c) ** 2
    w1 = 0.6 / q(b - 2 * c + d, b - d) ** 2
    w2 = 0.3 / q(c - 2 * d + e, 3 * c - 4 * d + e) ** 2
    return (w0 * (2 * a - 7 * b + 11 * c) + w1 * (-b + 5 * c + 2 * d) + w2 * (2 * c + 5 * d - e)) / (6.0 * (w0 + w1 + w2))


def _advection(P, f):
    """Conservative WENO5 advection with diffuse walls; populations [B][N][k][i][j]."""
    N, Q = P.N, P.QR
    ext = f.new_empty(f.shape[:1] + (N + 4,) + f.shape[2:])
    ext[:, 2:N + 2] = f / P.w
    for g, s in ((1, 1), (N + 2, -1)):  # outgoing directions: cubic extrapolation beyond the wall cell
        v = [ext[:, (2 if s > 0 else N + 1) + s * k] for k in range(4)]
        ext[:, g] = 4 * v[0] - 6 * v[1] + 4 * v[2] - v[3]
        ext[:, g - s] = 10 * v[0] - 20 * v[1] + 15 * v[2] - 4 * v[3]
    x = lambda c: ext[:, c + 2]  # noqa: E731
    pabs = P.pR.abs()[None, :, None]
    mass = (lambda y: y[:, :1]) if P.reduced else (lambda y: y)
    walls = []
    for side, out, inn, vh in ((0, slice(Q, None), slice(None, Q), _weno(x(2), x(1), x(0), x(-1), x(-2))),
                               (1, slice(None, Q), slice(Q, None), _weno(x(N - 3), x(N - 2), x(N - 1), x(N), x(N + 1)))):
        flux = mass((pabs * P.w * vh)[:, :, out]).sum((1, 2, 3))
        walls.append(flux / mass((pabs * P.wall[:, side])[:, :, inn]).sum((1, 2, 3)))
    inc = [walls[s][:, None, None, None] * P.wall[:, s] for s in (0, 1)]  # incoming populations at the walls
    ext[:, :2, :, :Q] = (inc[0] / P.w)[:, None, :, :Q]
    ext[:, N + 2:, :, Q:] = (inc[1] / P.w)[:, None, :, Q:]
    up = [ext[:, k:k + N, :, :Q] for k in range(5)]
    dn = [ext[:, k:k + N, :, Q:] for k in range(4, -1, -1)]
    wp, wn = P.w[:, :Q], P.w[:, Q:]
    right = torch.cat([inc[0][:, None, :, :Q], _weno(*up) * wp], 1)  # faces 0 .. N, p_R > 0
    left = torch.cat([_weno(*dn) * wn, inc[1][:, None, :, Q:]], 1)  # p_R < 0
    F = P.A[..., None, None, None] * P.pR[None, :, None] * torch.cat([right, left], 3)
    return (F[:, 1:] - F[:, :-1]) / P.V[..., None, None, None]


def _rhs(P, f):
    e = lambda y: y[..., None, None, None]  # noqa: E731
    n, u, T, q, _ = _macroscopic(P, f)
    sg = P.sigma[:, None]
    nbar = (P.W @ n[..., None])[..., 0]
    chi = _chi(math.pi * sg ** 3 * nbar / 6.0)
    br = 2.0 * math.pi / 3.0 * sg ** 3 * n
    y = br * chi
    Pr = 2.0 / 3.0 * (1.0 + 0.8 * y + 0.16 * (1.0 + 12.0 / math.pi) * y ** 2) \
        / (1.0 + 1.2 * y + 0.36 * (1.0 + 32.0 / (9.0 * math.pi)) * y ** 2)
    tau = _viscosity(n, T, chi, sg) / (n * T)
    X, Y = _d_dR(P, torch.log(n * n * chi * T)), _d_dR(P, torch.log(T))
    du = [_d_dR(P, u[..., a]) for a in range(3)]
    R, sph = P.R_c, P.geometry == SPH
    S00, S11 = du[0], u[..., 0] / R
    S22 = S11 if sph else torch.zeros_like(S11)
    S01 = 0.5 * (du[1] - u[..., 1] / R)
    S02 = 0.5 * (du[2] - (u[..., 2] / R if sph else 0.0))
    div = du[0] + (2.0 if sph else 1.0) * S11
    # collision
    p3, pR, p2 = P.p3[:, None, None], P.pR[None, :, None], P.p2[None, None, :]
    x0, x1 = pR - e(u[..., 0]), p2 - e(u[..., 1])
    if P.reduced:
        x2, sq = torch.zeros_like(x0), x0 * x0 + x1 * x1 + e(T) * T.new_tensor([1.0, 3.0])[:, None, None]
        g3 = torch.stack([torch.ones_like(T), T], -1)
    else:
        x2 = p3 - e(u[..., 2])
        sq = x0 * x0 + x1 * x1 + x2 * x2
        g3 = _g_full(P.p3, P.w3, u[..., 2], T)
    fmb = e(n) * g3[..., :, None, None] * _g_half(P, u[..., 0], T)[..., None, :, None] \
        * _g_full(P.p2, P.w2, u[..., 1], T)[..., None, None, :]
    xq = x0 * e(q[..., 0]) + x1 * e(q[..., 1]) + x2 * e(q[..., 2])
    fS = fmb * (1.0 + e((1.0 - Pr) / (n * T * T)) * (sq / (5.0 * e(T)) - 1.0) * xq)
    zz = sq / (2.0 * e(T)) - 2.5
    strain = (x0 * x0 * e(S00) + x1 * x1 * e(S11) + x2 * x2 * e(S22) + 2.0 * x0 * (x1 * e(S01) + x2 * e(S02))) / e(T)
    J1 = -e(y) * fmb * (x0 * (e(X) + 0.6 * zz * e(Y)) + 0.4 * (strain + zz * e(div)))
    L = (fS - f) / e(tau) + J1 - _advection(P, f)
    # curvature force
    kap = e((P.A[:, 1:] - P.A[:, :-1]) / P.V)
    KRf, K2f = P.KR @ f, f @ P.K2.T
    if sph:
        K3f = (P.K3 @ f.flatten(3)).unflatten(3, f.shape[3:])
        return L - 0.5 * kap * ((p2 * p2 + p3 * p3) * KRf - pR * (K2f + K3f))
    return L - kap * (p2 * p2 * KRf - pR * K2f)


# ------------------------------------------------------------------------------- the network
def _net_shapes(case):
    W, m, L, H = (case[k] for k in ("width", "modes", "layers", "hidden"))
    out = [("lift", (6, W)), ("lift_b", (W,))]
    for l in range(L):
        out += [("re%d" % l, (m, W, W)), ("im%d" % l, (m, W, W)), ("w%d" % l, (W, W)), ("b%d" % l, (W,))]
    return out + [("p1", (W, H)), ("c1", (H,)), ("p2", (H, 4)), ("c2", (4,))]


def _net_inputs(case, seed):
    """Sweep parameters, steady-like target profiles and weights of a partly trained network."""
    rng = np.random.default_rng(int(seed))
    B, P = case["batch"], case["points"]
    raw = np.stack([10 ** rng.uniform(-2, 0, B), rng.uniform(0.01, 0.3, B), rng.uniform(1.2, 5, B), rng.uniform(0, 0.3, B),
                    rng.uniform(1.0, 1.3, B)], 1).astype(np.float32)
    x = np.linspace(0.0, 1.0, P)
    c = rng.uniform(-1.0, 1.0, (B, 1, 4))
    target = (c * np.cos(math.pi * x)[None, :, None] + raw[:, None, 3:4] * (1.0 - x)[None, :, None]).astype(np.float32)
    theta = []
    for name, shape in _net_shapes(case):
        scale = 0.5 / case["width"] if name[:2] in ("re", "im") else 0.1 if len(shape) == 1 else 1.0 / math.sqrt(shape[0])
        theta.append((scale * rng.uniform(-1.0, 1.0, shape)).astype(np.float32).ravel())
    return raw, target, np.concatenate(theta)


def _net_exact(case, seed, dev):
    """Forward pass (and gradient, by autograd) in FP64 with the weight matrices as BF16 holds them."""
    raw, target, theta = _net_inputs(case, seed)
    t = lambda v: torch.tensor(v, dtype=torch.float64, device=dev)  # noqa: E731
    p, at = {}, 0
    for name, shape in _net_shapes(case):
        v = torch.from_numpy(theta[at:at + int(np.prod(shape))]).reshape(shape)
        at += v.numel()
        p[name] = (v if len(shape) == 1 else v.bfloat16()).to(dev).double().requires_grad_(case["grad"])
    B, P, m = case["batch"], case["points"], case["modes"]
    r = raw.astype(np.float64)
    feat = t(np.stack([np.log10(r[:, 0]) + 1.0, (r[:, 1] - 0.155) / 0.145, (r[:, 2] - 3.1) / 1.9, (r[:, 3] - 0.15) / 0.15,
                       (r[:, 4] - 1.15) / 0.15], 1))
    x = torch.arange(P, device=dev, dtype=torch.float64)
    a = torch.cat([feat[:, None].expand(B, P, 5), (x / (P - 1))[None, :, None].expand(B, P, 1)], -1)
    ang = 2.0 * math.pi / P * torch.outer(torch.arange(m, device=dev, dtype=torch.float64), x)
    c = torch.where(torch.arange(m, device=dev) == 0, 1.0, 2.0).double()[:, None] / P
    gelu = lambda z: 0.5 * z * (1.0 + torch.erf(z / math.sqrt(2.0)))  # noqa: E731
    v = a @ p["lift"] + p["lift_b"]
    for l in range(case["layers"]):
        re, im = torch.cos(ang) @ v, -torch.sin(ang) @ v  # [B][m][W]
        mix = lambda y, R: torch.einsum("bki,kio->bko", y, R)  # noqa: E731
        yre = mix(re, p["re%d" % l]) - mix(im, p["im%d" % l])
        yim = mix(re, p["im%d" % l]) + mix(im, p["re%d" % l])
        s = (c * torch.cos(ang)).T @ yre - (c * torch.sin(ang)).T @ yim
        v = gelu(v @ p["w%d" % l] + p["b%d" % l] + s)
    out = gelu(v @ p["p1"] + p["c1"]) @ p["p2"] + p["c2"]
    if not case["grad"]:
        return {"profiles": out}
    loss = ((out - t(target)) ** 2).mean()
    loss.backward()
    return {"loss": loss.detach(), "grad": torch.cat([p[k].grad.reshape(-1) for k, _ in _net_shapes(case)])}
