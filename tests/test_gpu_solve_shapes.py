"""The fused BiCGSTAB solve over the shapes its launch rule distinguishes: one
CTA or a team of them, every lanes-per-row variant, ragged and empty-ish rows,
sizes around the CTA's 1024 threads.  Reference: a dense FP64 solve."""
import numpy as np
import pytest

from paper_2301_05780_gb300 import pdds

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _system(n, per_row, seed):
    """Row-substochastic system like Eq. 23's: unit diagonal, negative
    off-diagonals summing to 0.9 per row, ragged row lengths up to per_row."""
    r = np.random.default_rng(seed)
    rows, A = [], np.eye(n)
    for k in range(n):
        m = min(n - 1, int(r.integers(0, per_row + 1)))
        c = r.choice(n - 1, size=m, replace=False)
        c[c >= k] += 1
        w = r.uniform(0.1, 1.0, m)
        A[k, c] = -0.9 * w / max(w.sum(), 1e-300)
        rows.append(np.sort(np.append(c, k)))
    rp = np.concatenate([[0], np.cumsum([len(c) for c in rows])]).astype(np.int32)
    col = np.concatenate(rows).astype(np.int32)
    val = np.concatenate([A[k, c] for k, c in enumerate(rows)])
    return A, rp, col, val, r.normal(size=n)


@pytest.mark.parametrize("n,per_row", [(1, 0), (2, 1), (31, 12), (255, 40), (1023, 60), (1024, 150),
                                       (1025, 260), (2047, 700), (3001, 120)])
def test_solve_matches_a_dense_solve(n, per_row):
    A, rp, col, val, b = _system(n, per_row, n)
    dev = lambda a: torch.tensor(a, device="cuda")
    G, bd = (dev(rp), dev(col), dev(val)), dev(b)
    u = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
    it = pdds.pdds_solve_noalloc(G, bd, u, rtol=1e-12, maxit=1000)
    got = u.cpu().numpy()
    assert it >= 1
    # the recurrence stops at 1e-12 ||b||; FP64 rounding of its ~100 updates stays below that
    assert np.linalg.norm(b - A @ got) <= 1e-11 * np.linalg.norm(b)
    # ||A^-1||_inf <= 1 / (1 - 0.9)
    assert np.abs(got - np.linalg.solve(A, b)).max() <= 10 * 1e-11 * np.linalg.norm(b)
    # repeats bit for bit, also with the solution taking the place of b
    alias = bd.clone()
    pdds.pdds_solve_noalloc(G, alias, alias, rtol=1e-12, maxit=1000)
    assert torch.equal(alias, u)


def test_zero_right_hand_side_and_maxit():
    A, rp, col, val, b = _system(300, 20, 5)
    dev = lambda a: torch.tensor(a, device="cuda")
    G = (dev(rp), dev(col), dev(val))
    u = torch.full((300,), float("nan"), dtype=torch.float64, device="cuda")
    assert pdds.pdds_solve_noalloc(G, torch.zeros_like(u), u) == 0
    assert torch.equal(u, torch.zeros_like(u))
    with pytest.raises(pdds.PddsError) as e:
        pdds.pdds_solve_noalloc(G, dev(b), u, rtol=1e-14, maxit=2)
    assert e.value.status == pdds.PDDS_ENOCONV and "after 2 iterations" in str(e.value)


def test_solves_and_fits_from_several_threads():
    """The solve and the tensor-core fit are cooperative launches whose CTAs wait
    for one another: several of them at once, on streams of their own next to
    assemblies, all finish, and every solve gives the serial result bit for bit."""
    import threading

    from paper_2301_05780_gb300 import workloads as W

    ws = [W.config1(), W.config2().scaled(n_paths=300), W.paper_e1().scaled(n_paths=20)]
    probs = [pdds.Problem(w) for w in ws]
    want = []
    for P in probs:
        P.assemble()
        P.solve()
        want.append(P.u.clone())
    busy = pdds.Problem(W.config2().scaled(n_paths=2000))
    xy = torch.rand(11_000, 2, device="cuda") * 2 - 1
    t = torch.sin(3 * xy[:, 0]) * xy[:, 1]
    torch.cuda.synchronize()
    bad = []

    def solve(i):
        s = torch.cuda.Stream()
        for _ in range(25):
            u = torch.full_like(want[i], float("nan"))
            torch.cuda.current_stream().synchronize()
            pdds.pdds_solve(probs[i].ctx, probs[i].G, probs[i].b, u, 1e-12, 5000, stream=s)
            if not torch.equal(u, want[i]):
                bad.append(("solve", i))

    def fit():
        s = torch.cuda.Stream()
        for _ in range(10):
            th = torch.tensor(W.mlp_init(), dtype=torch.float32, device="cuda")
            torch.cuda.current_stream().synchronize()
            loss = pdds.pdds_mlp_train(th, xy, t, steps=20, stream=s, engine="tc")
            if not (np.isfinite(loss).all() and loss[-1] < loss[0]):
                bad.append(("fit", loss))

    def assemble():
        s = torch.cuda.Stream()
        for _ in range(10):
            busy.assemble(stream=s)
            s.synchronize()

    def guard(f, *a):
        def run():
            try:
                f(*a)
            except Exception as e:   # a wait that ran out comes back as an error
                bad.append((f.__name__, repr(e)))
        return run

    ts = [threading.Thread(target=guard(solve, i)) for i in range(3)] + \
         [threading.Thread(target=guard(f)) for f in (fit, fit, assemble)]
    [x.start() for x in ts]
    [x.join() for x in ts]
    assert not bad, bad[:3]
