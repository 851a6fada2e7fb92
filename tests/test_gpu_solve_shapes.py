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
