"""The work a user of this framework has it do, as cases that can be timed and compared.

Every case goes through the Python binding (``paper_2301_05780_gb300.pdds``), the calls that the
README, the three-phase pipeline (``calibrated.py``) and the control-variate study (``cv.py``) make.
The kinds of work:

  assemble    Problem.assemble() [+ solve()]: Monte Carlo assembly of G and b, every coefficient
              set, naive (EM) or Gobet-Menozzi (GM) exits, linear or RBF stencils, without a
              control variate, with a tabulated one, or with the in-path network; uniform budgets
              or per-knot budgets and steps
  host        the end-to-end call on host buffers (pdds_assemble_solve_host)
  batch       several problems in one launch, host buffers (pdds_assemble_solve_batch_host)
  calibrate   the mixed GM/EM calibration run and the plan (pdds_calibrate, pdds_plan)
  train       the fit of v_theta (pdds_mlp_train)
  eval        v_theta and its gradient at the nodes of the look-up table (pdds_mlp_eval_tc)

``exact`` restates each of them in torch float64: Philox4x32-10 and Box-Muller from their
published definitions, the estimator path by path, the solve as a dense one.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2301_05780_gb300 import pdds
from paper_2301_05780_gb300 import workloads as W

DEV = "cuda"
R2 = math.sqrt(2.0)

# domain [lo, hi]^2, bounds of s, and the counted FP32 operations of one path-step (random
# normals, exit test, update and coefficients; an FMA counts two, a transcendental one)
SETS = {
    "laplace": dict(id=W.COEF_LAPLACE_EXPSIN, lo=0.0, hi=1.0, s=(R2, R2), flops=27),
    "manufactured": dict(id=W.COEF_MANUFACTURED, lo=0.0, hi=1.0, s=(R2, R2), flops=77),
    "varsigma": dict(id=W.COEF_VARSIGMA, lo=0.0, hi=4.0, s=(0.7 * R2, 1.3 * R2), flops=70),
    "table": dict(id=W.COEF_TABLE, lo=0.0, hi=1.0, s=(R2 - 0.3, R2 + 0.3), flops=64),
    "e1": dict(id=W.COEF_POISSON_E1, lo=-100.0, hi=100.0, s=(R2, R2), flops=89),
}
NET_FLOPS = 4 * 64 * 64 + 64 * 24    # grad v_theta at one point: two 64 x 64 products, the SiLUs
NPARAM = pdds.MLP_NPARAM


def listed():
    return [
        # the first problem a new user runs, and the smallest: 29 knots, 1e4 paths each, assembled
        # and solved (the package's config 1); launches and the longest path are what it waits for
        dict(name="laplace_2x2", kind="assemble", coef="laplace", H=2, m=8, N=10_000, dt=1e-4,
             solve=True),
        # one mid-size problem with drift and potential, end to end on host buffers (config 2)
        dict(name="manufactured_8x8_host", kind="host", coef="manufactured", H=8, m=8, N=100_000,
             dt=1e-5),
        # the headline: 16 boundary-value problems of mixed sizes in one launch, per-knot budgets
        # log-uniform (config 3 at a tenth of its budgets, so that a pass stays below a second)
        dict(name="varsigma_batch16", kind="batch", coef="varsigma", count=16, H_lo=4, H_hi=32, m=8,
             N_lo=1_000, N_hi=10_000, dt=1e-5),
        # measured coefficient fields: 1025 x 1025 tables, 16 knot intervals per edge (config 4's
        # spacing of tables and knots on a quarter of its subdomains, same steps per path)
        dict(name="table_32x32", kind="assemble", coef="table", H=32, m=16, N=1_000, dt=4e-7,
             solve=False),
        # the warm-up of the control-variate study: many knots, paths of about ten steps, then a
        # large sparse solve (config 5 with n0 = 1000)
        dict(name="short_paths_128x128", kind="assemble", coef="manufactured", H=128, m=4, N=1_000,
             dt=1e-6, solve=True),
        # its production run with the in-path network (config 5 with a small budget)
        dict(name="network_cv_128x128", kind="assemble", coef="manufactured", H=128, m=4, N=100,
             dt=1e-6, cv="network", solve=False),
        # the paper's problem, Phase I: warm-up with Gobet-Menozzi exits, solved
        dict(name="paper_phase1_gm", kind="assemble", coef="e1", H=10, m=63, N=1_000, dt=0.08,
             scheme="gm", launch=True, solve=True),
        # Phase I on the paper's own RBF stencils (Sec. 2.1), a smaller budget
        dict(name="paper_rbf_gm", kind="assemble", coef="e1", H=10, m=63, N=200, dt=0.08,
             scheme="gm", rbf=True, launch=True, solve=False),
        # Phase II: mixed GM/EM calibration with the tabulated control variate, and the plan
        dict(name="paper_phase2_calibrate", kind="calibrate", coef="e1", H=10, m=63, N=1_000, dt=0.08,
             cv="table", launch=True),
        # Phase III: production with per-knot steps and budgets, GM exits and the table
        dict(name="paper_phase3_production", kind="assemble", coef="e1", H=10, m=63, N=1_300, dt=0.08,
             scheme="gm", cv="table", ragged=True, knot_steps=True, launch=True, solve=True),
        # the fit between Phases I and II: full-batch Adam on the paper's 11,241 nodal values
        dict(name="fit_11241", kind="train", points=11_241, steps=100, engine="tc"),
        # the look-up table of grad u0 at half the paper's knot spacing: 1261 x 1261 nodes
        dict(name="eval_table_1261", kind="eval", points=1_261 * 1_261),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["assemble"] * 6 + ["host", "batch", "calibrate", "train", "eval"])
    if kind == "train":
        return dict(kind=kind, points=_log(rng, 1_000, 40_000), steps=_log(rng, 20, 200),
                    engine=rng.choice(["tc", "tc", "fp32"]))
    if kind == "eval":
        return dict(kind=kind, points=_log(rng, 1_000, 2_000_000))
    if kind == "batch":
        return dict(kind=kind, coef="varsigma", count=rng.randint(2, 8), H_lo=3,
                    H_hi=rng.randint(5, 24), m=rng.choice([5, 8, 11]), N_lo=200,
                    N_hi=_log(rng, 500, 10_000), dt=1e-5)
    coef = rng.choice(["e1", "e1", "manufactured"]) if kind == "calibrate" else \
        rng.choice(["laplace", "manufactured", "varsigma", "table", "e1"])
    H = _log(rng, 2, {"e1": 12, "varsigma": 24}.get(coef, 48))
    m = rng.choice([3, 4, 7, 8, 16]) if coef != "e1" else rng.choice([15, 33, 63])
    L = (SETS[coef]["hi"] - SETS[coef]["lo"]) / H
    steps = math.exp(rng.uniform(math.log(10.0), math.log(800.0)))   # per path, about
    dt = 0.25 * L * L / (SETS[coef]["s"][1] ** 2 * steps)
    n = 2 * (H - 1) * (H * m - 1) - (H - 1) ** 2
    top = min(100_000.0, 8e9 / (n * steps))
    if kind == "calibrate":
        top = min(top, 1.2e7 / n)
    N = _log(rng, max(1.0, min(200.0, top / 20)), max(2.0, top))
    c = dict(kind=kind, coef=coef, H=H, m=m, N=N, dt=dt)
    if kind == "host":
        return c
    cv = rng.choice(["none", "none", "table"] + (["network"] if coef in ("manufactured", "e1")
                                                 and n * steps * N < 4e8 else []))
    c.update(cv=cv, ragged=rng.random() < 0.3, knot_steps=rng.random() < 0.2)
    if kind == "calibrate":
        return c
    c.update(scheme=rng.choice(["em", "em", "gm"]), rbf=coef != "table" and rng.random() < 0.15,
             solve=rng.random() < 0.4)
    return c


# ------------------------------------------------------------------ preparation
def _grid(case, H=None):
    s = SETS[case["coef"]]
    H = H if H is not None else case["H"]
    return dict(x0=s["lo"], x1=s["hi"], y0=s["lo"], y1=s["hi"], Hx=H, Hy=H, m=case["m"], ext=0)


def _workload(case, seed, H=None):
    """The workload of a case: the stencil extension and step cap the package's own rules give."""
    s = SETS[case["coef"]]
    g = _grid(case, H)
    g["ext"] = W.stencil_extension(g, s["s"][1], case["dt"])
    if case.get("rbf"):
        g["ext"] = max(g["ext"], min(case["m"] // 2, 9))
    w = W.Workload(case.get("name", "drawn"), g, s["id"], n_paths=int(case.get("N", 0)),
                   dt=case["dt"], seed=_key(seed), sigma_bounds=s["s"])
    w.k_max = W.step_cap(g, s["s"][0], case["dt"])
    if case["coef"] == "table":
        w.params = (1.0, 0.0)
        w.tables = _tables(seed, g["Hx"])
    return w


def _key(seed):
    return (2_301_057_800 + 7_919 * int(seed)) % (1 << 63)


def _modes(seed):
    r = np.random.default_rng([int(seed), 4])
    return (r.integers(1, 5, (2, 32)), r.uniform(0, 1, 32), r.uniform(0, 2 * math.pi, 32))


def _field(seed, nx, ny):
    """Smooth random field on the unit square with values in [-1, 1] (32 low Fourier modes)."""
    (kx, ky), a, ph = _modes(seed)
    x, y = np.linspace(0, 1, nx), np.linspace(0, 1, ny)
    ex = np.exp(2j * math.pi * kx[:, None] * x[None, :] + 1j * ph[:, None]) * a[:, None]
    ey = np.exp(2j * math.pi * ky[:, None] * y[None, :])
    F = (ey.T @ ex).real
    return F / np.abs(F).max()


def _tables(seed, H):
    n = min(1025, 32 * H + 1)   # nodes a side: a patch's tile has to fit its stage
    return ((R2 + 0.3 * _field(seed, n, n)).astype(np.float32),
            (-1.25 + 0.75 * _field(int(seed) + 1_000_003, n, n)).astype(np.float32))


def _knots(g):
    """Lattice coordinates of the knots, ordered by (y, x)."""
    LX, LY, m = g["Hx"] * g["m"], g["Hy"] * g["m"], g["m"]
    j, i = np.meshgrid(np.arange(1, LY), np.arange(1, LX), indexing="ij")
    on = (i % m == 0) | (j % m == 0)
    return i[on].astype(np.int64), j[on].astype(np.int64)


def _budgets(case, seed, n):
    """Per-knot budgets as Eq. 41 gives them: multiples of a job size, unevenly spread."""
    r = np.random.default_rng([int(seed), 11])
    job = 200 if case["N"] >= 1_000 else 32 if case["N"] >= 100 else 1
    k = np.maximum(1, np.rint(case["N"] / job * np.exp(r.normal(-0.2, 0.6, n))))
    return np.minimum(k, np.ceil(4.0 * case["N"] / job)).astype(np.int64) * job


def _steps(case, seed, n):
    """Per-knot steps as Eq. 40 gives them: h0 at most knots, down to a fourth at the others."""
    r = np.random.default_rng([int(seed), 12])
    return case["dt"] * np.clip(np.exp(r.normal(0.4, 0.6, n)), 0.25, 1.0)


def _grad_u(coef, x, y):
    """Gradient of the closed-form solution of each set (of a smooth stand-in for the table set)."""
    if coef == "laplace":
        return torch.exp(x) * torch.sin(y), torch.exp(x) * torch.cos(y)
    if coef == "manufactured":
        return (math.pi * torch.cos(math.pi * x) * torch.cos(math.pi * y) + y,
                -math.pi * torch.sin(math.pi * x) * torch.sin(math.pi * y) + x)
    if coef == "varsigma":
        return (0.25 * torch.exp(x / 4) * torch.cos(y / 2), -0.5 * torch.exp(x / 4) * torch.sin(y / 2))
    if coef == "table":
        return 0.2 * torch.cos(3 * x) * torch.sin(3 * y), 0.2 * torch.sin(3 * x) * torch.cos(3 * y)
    r = torch.sqrt(1 + x * x / 100 + y * y / 50)
    a, b = 3 * x / 25 + y / 20, x / 20 - 3 * y / 25
    t = 1 - torch.tanh(torch.sin(a) + torch.sin(b)) ** 2
    return ((torch.cos(r) * x / 100 / r + t * (0.12 * torch.cos(a) + 0.05 * torch.cos(b))) / 3,
            (torch.cos(r) * y / 50 / r + t * (0.05 * torch.cos(a) - 0.12 * torch.cos(b))) / 3)


def _cv_table(case, seed, g):
    """The look-up table of grad u0 (Sec. 4.2), two nodes per knot spacing: the gradient of the
    solution with the smooth error that a warm-up fit leaves."""
    n = 2 * g["Hx"] * g["m"] + 1
    t = torch.linspace(g["x0"], g["x1"], n, dtype=torch.float64, device=DEV)
    y, x = torch.meshgrid(t, t, indexing="ij")
    gx, gy = _grad_u(case["coef"], x, y)
    r = np.random.default_rng([int(seed), 13])
    L = g["x1"] - g["x0"]
    scale = 0.2 * float(torch.sqrt((gx * gx + gy * gy).mean()))
    kx, ky, p, q = r.integers(2, 9), r.integers(2, 9), *r.uniform(0, 6.28, 2)
    e = scale * torch.sin(kx * math.pi * x / L + p) * torch.cos(ky * math.pi * y / L + q)
    return torch.stack([gx + e, gy - e], dim=-1).to(torch.float32).contiguous()


def _theta(seed, coef, lo, hi):
    """A network fitted to the solution of its set: seeded hidden layers on inputs scaled to
    [-1, 1]^2, the last layer by least squares (float64), the input scaling folded into layer 1."""
    r = np.random.default_rng([int(seed), 14])
    W1, b1 = r.normal(0, 1.0, (64, 2)) * 2.0, r.uniform(-2, 2, 64)
    W2, b2 = r.normal(0, 1.0, (64, 64)) / 8 * 1.5, r.uniform(-0.5, 0.5, 64)
    x = r.uniform(-1, 1, (4096, 2))
    silu = lambda a: a / (1 + np.exp(-a))  # noqa: E731
    F = np.concatenate([silu(silu(x @ W1.T + b1) @ W2.T + b2), np.ones((4096, 1))], axis=1)
    c, s = (lo + hi) / 2, (hi - lo) / 2
    u = _u_exact(coef, x[:, 0] * s + c, x[:, 1] * s + c)
    A = F.T @ F + 1e-6 * np.eye(65) * 4096
    w3 = np.linalg.solve(A, F.T @ u)
    W1s = W1 / s
    return np.concatenate([W1s.ravel(), b1 - W1s.sum(axis=1) * c, W2.ravel(), b2,
                           w3]).astype(np.float32)


def _u_exact(coef, x, y):
    if coef == "manufactured":
        return np.sin(math.pi * x) * np.cos(math.pi * y) + x * y
    if coef == "laplace":
        return np.exp(x) * np.sin(y)
    r, q = np.sqrt(1 + x * x / 100 + y * y / 50), np.sin(.12 * x + .05 * y) + np.sin(.05 * x - .12 * y)
    return 3 + np.sin(r) / 3 + np.tanh(q) / 3


def _setup(P, case, seed):
    """What a context keeps between calls: exit scheme, stencils, control variate, per-knot data."""
    g = P.w.grid
    if case.get("launch"):     # the launch shape of the three-phase pipeline (calibrated.run)
        pdds.pdds_set_launch(P.ctx, 128, 0, 1024, 4)
    if case.get("scheme") == "gm":
        pdds.pdds_set_scheme(P.ctx, pdds.PDDS_SCHEME_GM)
    if case.get("rbf"):
        pdds.pdds_set_interpolation(P.ctx, pdds.PDDS_INTERP_RBF, RBF_C * (g["x1"] - g["x0"]) /
                                    (g["Hx"] * g["m"]))
    if case.get("cv") == "table":
        pdds.pdds_set_control_variate_grid(P.ctx, _cv_table(case, seed, g))
    elif case.get("cv") == "network":
        theta = torch.tensor(_theta(seed, case["coef"], g["x0"], g["x1"]), device=DEV)
        pdds.pdds_set_control_variate(P.ctx, theta)
    if case.get("knot_steps"):
        pdds.pdds_set_knot_steps(P.ctx, torch.tensor(_steps(case, seed, P.n), device=DEV))
    if case.get("ragged"):
        P.n_per_knot = torch.tensor(_budgets(case, seed, P.n), device=DEV)


RBF_C = 2.0    # shape parameter of the RBF stencils in knot spacings


class _Batch:
    def __init__(self, case, seed):
        r = np.random.default_rng([21, case["count"], case["H_hi"]])   # the sizes are the case's own
        Hs = r.integers(case["H_lo"], case["H_hi"] + 1, case["count"])
        b = np.random.default_rng([int(seed), 22])
        self.P, self.N, self.out = [], [], []
        for H in Hs:
            P = pdds.Problem(_workload(case, seed, int(H)))
            pdds.pdds_set_launch(P.ctx, 128, 0, 2048, 4)   # as the headline benchmark sets it
            e = b.uniform(math.log10(case["N_lo"]), math.log10(case["N_hi"]), P.n)
            self.P.append(P)
            self.N.append(torch.from_numpy((np.round(10.0 ** e / 32) * 32).clip(32).astype(np.int64))
                          .pin_memory())
            self.out.append(_host_out(P))


def _host_out(P):
    i = lambda n: torch.empty(n, dtype=torch.int32, pin_memory=True)     # noqa: E731
    d = lambda n: torch.empty(n, dtype=torch.float64, pin_memory=True)   # noqa: E731
    return dict(row_ptr=i(P.n + 1), col=i(P.nnz), val=d(P.nnz), b=d(P.n), u=d(P.n))


def _points(seed, n):
    r = torch.Generator(device=DEV).manual_seed(int(seed) + 31)
    return torch.rand(n, 2, generator=r, device=DEV, dtype=torch.float32) * 2 - 1


def _fit_data(case, seed):
    """Nodal values of a warm-up: a smooth solution with Monte Carlo noise, standardised."""
    xy = _points(seed, case["points"])
    r = torch.Generator(device=DEV).manual_seed(int(seed) + 32)
    x, y = xy[:, 0].double(), xy[:, 1].double()
    u = torch.sin(3 * x) * torch.cos(2 * y) + torch.tanh(2 * torch.sin(3 * y - x))
    u = u + 0.02 * torch.randn(u.shape, generator=r, device=DEV, dtype=torch.float64)
    return xy, ((u - u.mean()) / u.std()).float()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        xy, t = _fit_data(case, seed)
        return dict(case=case, xy=xy, t=t, theta0=torch.tensor(W.mlp_init(int(seed) + 55), device=DEV,
                                                               dtype=torch.float32))
    if kind == "eval":
        theta = torch.tensor(_theta(seed, "manufactured", -1.0, 1.0), device=DEV)
        return dict(case=case, xy=_points(seed, case["points"]), theta=theta)
    if kind == "batch":
        return dict(case=case, B=_Batch(case, seed))
    P = pdds.Problem(_workload(case, seed))
    _setup(P, case, seed)
    st = dict(case=case, P=P)
    if kind == "host":
        st["out"] = _host_out(P)
    if kind == "calibrate":
        ki, kj = _knots(P.w.grid)
        st.update(u0=_u0(case, seed, P.w.grid, ki, kj), mom=torch.empty(P.n, 8, dtype=torch.float64,
                  device=DEV), h=torch.empty(P.n, dtype=torch.float64, device=DEV),
                  n=torch.empty(P.n, dtype=torch.int64, device=DEV),
                  diag=torch.empty(P.n, 3, dtype=torch.float64, device=DEV))
    return st


def _u0(case, seed, g, ki, kj):
    """Nodal values of a warm-up solve: the solution with Monte Carlo noise."""
    L = g["x1"] - g["x0"]
    x, y = g["x0"] + ki * (L / (g["Hx"] * g["m"])), g["y0"] + kj * (L / (g["Hy"] * g["m"]))
    r = np.random.default_rng([int(seed), 15])
    return torch.tensor(_u_exact(case["coef"], x, y) + 0.01 * r.normal(0, 1, len(x)), device=DEV)


# ------------------------------------------------------------------------- run
RTOL = 1e-12


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "train":
        theta = st["theta0"].clone()
        loss = pdds.pdds_mlp_train(theta, st["xy"], st["t"], steps=case["steps"], lr=3e-3,
                                   engine=case["engine"])
        return dict(theta=theta, loss=loss)
    if kind == "eval":
        v, g = pdds.pdds_mlp_eval_tc(st["theta"], st["xy"])
        return dict(v=v, grad=g)
    if kind == "batch":
        B = st["B"]
        w = B.P[0].w
        pick = lambda k: [o[k] for o in B.out]   # noqa: E731
        pdds.pdds_assemble_solve_batch_host([P.ctx for P in B.P], 0, w.dt, w.seed, RTOL, 5000,
                                            pick("row_ptr"), pick("col"), pick("val"), pick("b"),
                                            pick("u"), n_per_knot=B.N)
        return dict(row_ptr=pick("row_ptr")[:2], col=pick("col")[:2], val=pick("val"), b=pick("b"),
                    u=pick("u"))
    P = st["P"]
    if kind == "host":
        o = st["out"]
        pdds.pdds_assemble_solve_host(P.ctx, P.w.n_paths, P.w.dt, P.w.seed, RTOL, 5000,
                                      o["row_ptr"], o["col"], o["val"], o["b"], o["u"])
        return dict(o)
    if kind == "calibrate":
        pdds.pdds_calibrate(P.ctx, st["u0"], st["mom"], P.w.n_paths, P.n_per_knot, P.w.dt, P.w.seed)
        pdds.pdds_plan(st["mom"], 0.01, P.w.dt, P.w.dt, 200, st["h"], st["n"], st["diag"])
        return dict(mom=st["mom"], h=st["h"], n=st["n"], diag=st["diag"])
    P.assemble()
    out = dict(row_ptr=P.row_ptr, col=P.col, val=P.val, b=P.b)
    if case.get("solve"):
        P.solve(rtol=RTOL)
        out["u"] = P.u
    return out


# ------------------------------------------------------------------------ work
def _mean_steps(case, dt=None):
    """Mean steps of a path, about: the mean exit time of a patch of two subdomains from the knots
    along their shared edge, over the step (short paths add the overshoot of the last step)."""
    s = SETS[case["coef"]]
    L = (s["hi"] - s["lo"]) / case["H"]
    return 0.2 * L * L / (s["s"][0] * s["s"][1] * (dt or case["dt"])) + 3.0


def work(case):
    kind = case["kind"]
    if kind == "train":
        n = case["points"]
        return dict(bytes=12.0 * n * case["steps"], flops=float(n) * case["steps"] * 3 * 2 * (64 * 64 + 192))
    if kind == "eval":
        return dict(bytes=20.0 * case["points"], flops=float(case["points"]) * NET_FLOPS)
    if kind == "batch":
        one = [dict(case, H=int(H)) for H in np.linspace(case["H_lo"], case["H_hi"], case["count"])]
        mean_n = (case["N_hi"] - case["N_lo"]) / math.log(case["N_hi"] / case["N_lo"])
        w = [_assembly_work(dict(c, N=mean_n)) for c in one]
        return dict(bytes=sum(x[0] for x in w), flops=sum(x[1] for x in w))
    b, f = _assembly_work(case)
    return dict(bytes=b, flops=f)


def _assembly_work(case):
    H, m, N = case["H"], case["m"], case["N"]
    n = 2.0 * (H - 1) * (H * m - 1) - (H - 1) ** 2
    steps = _mean_steps(case)
    flops = SETS[case["coef"]]["flops"] + {"table": 30, "network": NET_FLOPS}.get(case.get("cv"), 0)
    nnz = n * (6.0 * m + 6)
    return 12.0 * nnz + 8 * n * 2 + 128 * n, n * N * steps * flops


# ----------------------------------------------------------------------- exact
MOST_STEPS = 1.3e9   # path-steps that the float64 restatement does within about twenty seconds


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "eval":
        xy = _points(seed, case["points"]).double()
        th = torch.tensor(_theta(seed, "manufactured", -1.0, 1.0), device=DEV).double()
        v, gx, gy = _net(th, xy[:, 0], xy[:, 1])
        return dict(v=v, grad=torch.stack([gx, gy], dim=1))
    if kind == "batch":
        return None
    g = _workload(case, seed).grid
    ki, kj = _knots(g)
    n = len(ki)
    total = _mean_steps(case) * n * case["N"] * (2 if kind == "calibrate" else 1) * \
        (2 if case.get("knot_steps") else 1) * (8 if case.get("cv") == "network" else 1)
    if total > MOST_STEPS:
        return None
    S = _Sim(case, seed, g, ki, kj)
    if kind == "calibrate":
        return S.calibrate(_u0(case, seed, g, ki, kj))
    val, b, row_ptr, col = S.assemble()
    out = dict(row_ptr=None, col=None, val=val, b=b)
    if case.get("solve") or kind == "host":
        out["u"] = None
        if n <= 12_000:
            A = torch.zeros(n, n, dtype=torch.float64, device=DEV)
            rows = torch.repeat_interleave(torch.arange(n, device=DEV), row_ptr[1:] - row_ptr[:-1])
            A[rows, col] = val
            out["u"] = torch.linalg.solve(A, b)
    return out


def _exact_train(case, seed):
    xy, t = _fit_data(case, seed)
    x, y, t = xy[:, 0].double(), xy[:, 1].double(), t.double()
    th = torch.tensor(W.mlp_init(int(seed) + 55), device=DEV, dtype=torch.float32).double()
    m, v, loss = torch.zeros_like(th), torch.zeros_like(th), []
    X = torch.stack([x, y], dim=1)
    for k in range(1, case["steps"] + 1):
        W1, b1, W2, b2, w3, b3 = _split(th)
        a1 = X @ W1.T + b1
        s1 = torch.sigmoid(a1)
        h1 = a1 * s1
        a2 = h1 @ W2.T + b2
        s2 = torch.sigmoid(a2)
        h2 = a2 * s2
        r = h2 @ w3 + b3 - t
        loss.append((r * r).mean())
        dv = 2 * r / len(t)
        g2 = dv[:, None] * w3 * (s2 * (1 + a2 * (1 - s2)))
        g1 = (g2 @ W2) * (s1 * (1 + a1 * (1 - s1)))
        g = torch.cat([(g1.T @ X).reshape(-1), g1.sum(0), (g2.T @ h1).reshape(-1), g2.sum(0), h2.T @ dv,
                       dv.sum()[None]])
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        th = th - 3e-3 * (m / (1 - 0.9 ** k)) / (torch.sqrt(v / (1 - 0.999 ** k)) + 1e-8)
    return dict(theta=th, loss=torch.stack(loss).cpu().numpy())


def _split(th):
    return (th[:128].view(64, 2), th[128:192], th[192:4288].view(64, 64), th[4288:4352],
            th[4352:4416], th[4416])


def _net(th, x, y, chunk=1 << 19):
    W1, b1, W2, b2, w3, b3 = _split(th)
    out = []
    for i in range(0, len(x), chunk):
        a1 = torch.stack([x[i:i + chunk], y[i:i + chunk]], dim=1) @ W1.T + b1
        s1 = torch.sigmoid(a1)
        a2 = (a1 * s1) @ W2.T + b2
        s2 = torch.sigmoid(a2)
        d1 = ((w3 * s2 * (1 + a2 * (1 - s2))) @ W2) * (s1 * (1 + a1 * (1 - s1)))
        out.append(torch.cat([((a2 * s2) @ w3 + b3)[:, None], d1 @ W1], dim=1))
    o = torch.cat(out)
    return o[:, 0], o[:, 1], o[:, 2]


MASK = 0xFFFFFFFF


def _philox(c, key):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors holding 32-bit words."""
    k0, k1 = key & MASK, (key >> 32) & MASK
    for r in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & MASK) ^ c[1] ^ k0, p1 & MASK, ((p0 >> 32) & MASK) ^ c[3] ^ k1, p0 & MASK]
        k0, k1 = (k0 + 0x9E3779B9) & MASK, (k1 + 0xBB67AE85) & MASK
    return c


def _normals(a, b):
    rho = torch.sqrt(-2 * torch.log((a.double() + 0.5) * 2.0 ** -32))
    th = (2 * math.pi) * ((b.double() + 0.5) * 2.0 ** -32)
    return rho * torch.cos(th), rho * torch.sin(th)


def _bilinear(T, fx, fy):
    """Bilinear interpolation of T [ny, nx, ...] at node coordinates."""
    ny, nx = T.shape[:2]
    i, j = fx.floor().long().clamp(0, nx - 2), fy.floor().long().clamp(0, ny - 2)
    tx, ty = (fx - i).clamp(0, 1), (fy - j).clamp(0, 1)
    F = T.reshape(nx * ny, -1)
    a, b, c, d = (F[(j + q) * nx + i + p].double() for q in (0, 1) for p in (0, 1))
    tx, ty = tx[:, None], ty[:, None]
    return (1 - ty) * ((1 - tx) * a + tx * b) + ty * ((1 - tx) * c + tx * d)


class _Sim:
    """The estimator of Sec. 2-3 of the paper path by path in float64: Euler-Maruyama steps from the
    knot, naive or Gobet-Menozzi exit from its patch, exits interpolated on the side's stencil."""

    def __init__(self, case, seed, g, ki, kj):
        self.case, self.g, self.coef = case, g, case["coef"]
        self.m, self.L = g["m"], g["Hx"] * g["m"]
        self.dx = (g["x1"] - g["x0"]) / self.L
        self.key = _key(seed)
        n = self.n = len(ki)
        t = lambda a: torch.tensor(a, device=DEV)   # noqa: E731
        self.i, self.j = t(ki), t(kj)
        m = self.m
        lo = lambda a: torch.where(a % m == 0, a - m, a // m * m)           # noqa: E731
        hi = lambda a: torch.where(a % m == 0, a + m, a // m * m + m)       # noqa: E731
        xl, xh, yl, yh = lo(self.i), hi(self.i), lo(self.j), hi(self.j)
        self.line = torch.stack([xh, yh, xl, yl], dim=1)                    # sides E, N, W, S
        self.a = (torch.stack([yl, xl, yl, xl], dim=1) - g["ext"]).clamp(min=0)
        self.b = (torch.stack([yh, xh, yh, xh], dim=1) + g["ext"]).clamp(max=self.L)
        self.index = torch.full((self.L + 1, self.L + 1), -1, dtype=torch.int64, device=DEV)
        self.index[self.j, self.i] = torch.arange(n, device=DEV)
        self.N = t(_budgets(case, seed, n)) if case.get("ragged") else \
            torch.full((n,), int(case["N"]), device=DEV)
        self.h = t(_steps(case, seed, n)) if case.get("knot_steps") else \
            torch.full((n,), case["dt"], dtype=torch.float64, device=DEV)
        cap = W.step_cap(g, SETS[self.coef]["s"][0], case["dt"])
        self.cap = torch.where(self.h == case["dt"], torch.full_like(self.h, cap),
                               torch.ceil(cap * case["dt"] / self.h).clamp(min=1)).long()
        self.tabs = None
        if self.coef == "table":
            self.tabs = torch.stack([t(T) for T in _tables(seed, g["Hx"])], dim=-1)
        self.cvt = _cv_table(case, seed, g) if case.get("cv") == "table" else None
        self.net = None
        if case.get("cv") == "network":
            self.net = t(_theta(seed, self.coef, g["x0"], g["x1"])).double()

    def u(self, x, y):
        c = self.coef
        if c == "laplace":
            return torch.exp(x) * torch.sin(y)
        if c == "manufactured":
            return torch.sin(math.pi * x) * torch.cos(math.pi * y) + x * y
        if c == "varsigma":
            return torch.exp(x / 4) * torch.cos(y / 2)
        if c == "table":
            return torch.zeros_like(x)
        r = torch.sqrt(1 + x * x / 100 + y * y / 50)
        q = torch.sin(.12 * x + .05 * y) + torch.sin(.05 * x - .12 * y)
        return 3 + torch.sin(r) / 3 + torch.tanh(q) / 3

    def at(self, x, y):
        """s, d, c, f at a point (None: zero)."""
        pi, c = math.pi, self.coef
        if c == "laplace":
            return R2, None, None, None, None
        if c == "manufactured":
            sx, cx, sy, cy = torch.sin(pi * x), torch.cos(pi * x), torch.sin(pi * y), torch.cos(pi * y)
            dx, dy, cc = 2 * sy * cy, 1 - 2 * sx * sx, -(1 + x * x)
            f = -2 * pi * pi * sx * cy + dx * (pi * cx * cy + y) + dy * (x - pi * sx * sy) + \
                cc * (sx * cy + x * y)
            return R2, dx, dy, cc, f
        if c == "varsigma":
            s = R2 * (1 + 0.3 * torch.sin(2 * pi * x) * torch.sin(2 * pi * y))
            u = self.u(x, y)
            return s, None, None, -torch.ones_like(x), -u * (1 + 3 * s * s / 32)
        if c == "table":
            T = _bilinear(self.tabs, x * (self.tabs.shape[1] - 1), y * (self.tabs.shape[0] - 1))
            return T[:, 0], None, None, T[:, 1], torch.ones_like(x)
        r2 = 1 + x * x / 100 + y * y / 50
        r = torch.sqrt(r2)
        G = (x * x / 1e4 + y * y / 2.5e3) / r2
        a, b = .12 * x + .05 * y, .05 * x - .12 * y
        q = torch.sin(a) + torch.sin(b)
        qx, qy = .12 * torch.cos(a) + .05 * torch.cos(b), .05 * torch.cos(a) - .12 * torch.cos(b)
        T = torch.tanh(q)
        f = torch.cos(r) * (0.03 - G) / r - torch.sin(r) * G + \
            (1 - T * T) * (-0.0169 * q - 2 * T * (qx * qx + qy * qy))
        return R2, None, None, None, f / 3

    def shifts(self, X, Y, box, x0, y0, h):
        """Gobet-Menozzi shifts of the sides E, N, W, S for the point (X, Y)."""
        c = 0.5826 * torch.sqrt(h)
        if self.coef not in ("varsigma", "table"):
            return (c * R2)[:, None].expand(-1, 4)
        cx, cy = X.clamp(box[:, 0], box[:, 1]), Y.clamp(box[:, 2], box[:, 3])
        pts = [(box[:, 1], cy), (cx, box[:, 3]), (box[:, 0], cy), (cx, box[:, 2])]
        return torch.stack([c * self.at(x0 + px, y0 + py)[0].abs() for px, py in pts], dim=1)

    def paths(self, gm, chunk=3_000_000):
        """Every path of every knot: (knot, X, Y, S, Z, xi, side) of its exit, chunk by chunk."""
        first = torch.zeros(self.n + 1, dtype=torch.int64, device=DEV)
        first[1:] = torch.cumsum(self.N, 0)
        k0 = 0
        while k0 < self.n:
            k1 = int(torch.searchsorted(first, first[k0] + chunk))
            k1 = min(self.n, max(k0 + 1, k1))
            yield self._chunk(k0, k1, first, gm)
            k0 = k1

    def _chunk(self, k0, k1, first, gm):
        k = torch.repeat_interleave(torch.arange(k0, k1, device=DEV), self.N[k0:k1])
        p = torch.arange(len(k), device=DEV) - (first[k] - first[k0])
        total = len(k)
        out = torch.zeros(6, total, dtype=torch.float64, device=DEV)   # X, Y, S, Z, xi, side
        kk = k.clone()
        who = torch.arange(total, device=DEV)
        z = lambda: torch.zeros(total, dtype=torch.float64, device=DEV)   # noqa: E731
        X, Y, S, Z, XI = z(), z(), z(), z(), z()
        alive = torch.ones(total, dtype=torch.bool, device=DEV)
        x0, y0 = self.g["x0"] + self.i[k] * self.dx, self.g["y0"] + self.j[k] * self.dx
        ln = self.line[k]
        box = torch.stack([ln[:, 2] - self.i[k], ln[:, 0] - self.i[k], ln[:, 3] - self.j[k],
                           ln[:, 1] - self.j[k]], dim=1) * self.dx
        h, cap, step = self.h[k], self.cap[k], 0
        ahead = []                                          # normals of the next steps of `who`
        while len(who):
            if not ahead:    # few paths left: the words of several Philox calls at once
                calls = max(1, min(32, 1_000_000 // len(who)))
                q = torch.arange(step // 2, step // 2 + calls, device=DEV)[:, None].expand(-1, len(who))
                w = _philox([q, p.expand_as(q), k.expand_as(q), torch.zeros_like(q)], self.key)
                one, two = _normals(w[0], w[1]), _normals(w[2], w[3])
                ahead = [v for c in range(calls) for v in ((one[0][c], one[1][c]), (two[0][c], two[1][c]))]
            for _ in range(2):
                zx, zy = ahead.pop(0)
                x, y = x0 + X, y0 + Y
                s, dx, dy, c, f = self.at(x, y)
                Yw = torch.exp(S) if c is not None else 1.0
                sq = torch.sqrt(h)
                if self.cvt is not None or self.net is not None:
                    if self.net is not None:
                        _, gx, gy = _net(self.net, x, y)
                    else:
                        q = (self.cvt.shape[0] - 1) / (self.g["x1"] - self.g["x0"])
                        gx, gy = _bilinear(self.cvt, (x - self.g["x0"]) * q, (y - self.g["y0"]) * q).T
                    XI = XI - Yw * s * sq * (gx * zx + gy * zy)
                if f is not None:
                    Z = Z - f * Yw * h
                if c is not None:
                    S = S + c * h
                X = X + s * sq * zx + (dx * h if dx is not None else 0)
                Y = Y + s * sq * zy + (dy * h if dy is not None else 0)
                step += 1
                sh = self.shifts(X, Y, box, x0, y0, h) if gm else 0.0
                over = torch.stack([X - box[:, 1], Y - box[:, 3], box[:, 0] - X, box[:, 2] - Y], dim=1) + sh
                ex = alive & ((over > 0).any(dim=1) | (step >= cap))
                e = ex.nonzero()[:, 0]
                if len(e):
                    o = over[e]
                    pos = torch.where(o > 0, o, torch.full_like(o, math.inf))
                    side = torch.where((o > 0).any(dim=1), pos.argmin(dim=1), o.argmax(dim=1))
                    out[:, who[e]] = torch.stack([X[e], Y[e], S[e], Z[e], XI[e], side.double()])
                    alive = alive & ~ex
            keep = alive.nonzero()[:, 0]
            if len(keep) < 0.9 * len(who):
                who, k, p, X, Y, S, Z, XI, alive, x0, y0, box, h, cap = (
                    v[keep] for v in (who, k, p, X, Y, S, Z, XI, alive, x0, y0, box, h, cap))
                ahead = [(a[keep], b[keep]) for a, b in ahead]
        return kk, out[0], out[1], out[2], out[3], out[4], out[5].long()

    def scores(self, k, X, Y, S, Z, side):
        """b share without xi, and the (stencil point, weight) pairs of each path's exit."""
        vert = (side % 2) == 0
        ln = self.line[k, side]
        a, b = self.a[k, side], self.b[k, side]
        w = torch.exp(S) if self.coef in ("manufactured", "varsigma", "table") else torch.ones_like(S)
        along = torch.where(vert, self.j[k] + Y / self.dx, self.i[k] + X / self.dx)
        x0, y0 = self.g["x0"], self.g["y0"]
        on = (ln == 0) | (ln == self.L)
        al = along.clamp(0, self.L)
        gb = self.u(x0 + self.dx * torch.where(vert, ln.double(), al),
                    y0 + self.dx * torch.where(vert, al, ln.double()))
        bc = Z + torch.where(on, w * gb, torch.zeros_like(w))
        sl = torch.minimum((along - a).clamp(min=0), (b - a).double())
        return vert, ln, a, b, w, on, sl, bc

    def point(self, vert, ln, t):
        """Knot index (-1 on the boundary) and g of the lattice point t along a side's line."""
        i, j = torch.where(vert, ln, t), torch.where(vert, t, ln)
        return self.index[j, i], self.u(self.g["x0"] + self.dx * i.double(),
                                        self.g["y0"] + self.dx * j.double())

    def weights(self, sc):
        """[(path, lattice point, weight)] of the exits on interfaces."""
        vert, ln, a, b, w, on, sl, bc = sc
        q = (~on).nonzero()[:, 0]
        if not self.case.get("rbf"):
            t = torch.minimum(sl[q].floor().long(), b[q] - a[q] - 1)
            lam = sl[q] - t
            yield q, a[q] + t, w[q] * (1 - lam)
            yield q, a[q] + t + 1, w[q] * lam
            return
        for n in torch.unique(b[q] - a[q] + 1).tolist():      # inverse multiquadrics (Sec. 2.1)
            z = torch.arange(n, dtype=torch.float64, device=DEV)
            inv = torch.linalg.inv(1 / torch.sqrt((z[:, None] - z[None, :]) ** 2 + RBF_C ** 2))
            same = q[(b[q] - a[q] + 1) == n]
            for part in same.split(400_000):
                H = (1 / torch.sqrt((sl[part][:, None] - z[None, :]) ** 2 + RBF_C ** 2)) @ inv
                t = a[part][:, None] + torch.arange(n, device=DEV)[None, :]
                yield part[:, None].expand(-1, n).reshape(-1), t.reshape(-1), (w[part][:, None] * H).reshape(-1)

    def pattern(self):
        """CSR keys row * n + col of the stencils, sorted (the diagonal included)."""
        keys = [torch.arange(self.n, device=DEV) * (self.n + 1)]
        span = int((self.b - self.a).max()) + 1
        t = torch.arange(span, device=DEV)
        for side in range(4):
            ln, a, b = self.line[:, side], self.a[:, side], self.b[:, side]
            p = a[:, None] + t[None, :]
            ok = (p <= b[:, None]) & (ln > 0)[:, None] & (ln < self.L)[:, None]
            i, j = (ln[:, None].expand_as(p), p) if side % 2 == 0 else (p, ln[:, None].expand_as(p))
            c = self.index[j.clamp(0, self.L), i.clamp(0, self.L)]
            row = torch.arange(self.n, device=DEV)[:, None].expand_as(p)
            ok = ok & (c >= 0)
            keys.append(row[ok] * self.n + c[ok])
        return torch.unique(torch.cat(keys))

    def assemble(self):
        keys = self.pattern()
        val = torch.zeros(len(keys), dtype=torch.float64, device=DEV)
        b = torch.zeros(self.n, dtype=torch.float64, device=DEV)
        for k, X, Y, S, Z, XI, side in self.paths(self.case.get("scheme") == "gm"):
            sc = self.scores(k, X, Y, S, Z, side)
            bc = sc[7] + XI
            for q, t, wt in self.weights(sc):
                c, gv = self.point(sc[0][q], sc[1][q], t)
                inside = c >= 0
                val.index_add_(0, torch.searchsorted(keys, k[q][inside] * self.n + c[inside]), wt[inside])
                bc.index_add_(0, q[~inside], (wt * gv)[~inside])
            b.index_add_(0, k, bc)
        row, col = keys // self.n, keys % self.n
        val = torch.where(row == col, torch.ones_like(val), -val / self.N[row])
        row_ptr = torch.searchsorted(keys, torch.arange(self.n + 1, device=DEV) * self.n)
        return val, b / self.N, row_ptr, col

    def calibrate(self, u0):
        """Moments of the mixed GM/EM scores and Eq. 40-41."""
        mom = torch.zeros(self.n, 8, dtype=torch.float64, device=DEV)
        for one, two in zip(self.paths(False), self.paths(True)):
            phi = []
            for k, X, Y, S, Z, XI, side in (one, two):
                sc = self.scores(k, X, Y, S, Z, side)
                f = sc[7].clone()
                for q, t, wt in self.weights(sc):
                    c, gv = self.point(sc[0][q], sc[1][q], t)
                    f.index_add_(0, q, wt * torch.where(c >= 0, u0[c.clamp(min=0)], gv))
                phi.append(f)
            k, xi, (pe, pg) = two[0], two[5], phi
            d = pe - pg
            mom.index_add_(0, k, torch.stack([torch.ones_like(d), d, d * d, pg, pg * pg, xi, xi * xi,
                                              pg * xi], dim=1))
        N, eps, h0 = mom[:, 0], 0.01, self.case["dt"]
        gap = mom[:, 1] / N
        cen = lambda ab, a, b: ((ab - a * b / N) / (N - 1).clamp(min=1)) * (N > 1)   # noqa: E731
        var = cen(mom[:, 4], mom[:, 3], mom[:, 3]).clamp(min=0)
        vx, cov = cen(mom[:, 6], mom[:, 5], mom[:, 5]), cen(mom[:, 7], mom[:, 3], mom[:, 5])
        rho2 = torch.where((var > 0) & (vx > 0), cov * cov / (var * vx), torch.zeros_like(var)).clamp(max=1)
        h = torch.where(gap != 0, torch.clamp(2 * h0 * eps / (3 * gap.abs()), max=h0),
                        torch.full_like(gap, h0))
        return dict(mom=mom, h=h, n=None, diag=torch.stack([gap, var, rho2], dim=1))
