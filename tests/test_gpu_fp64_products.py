"""FP64 products against numpy at the edges of the small-tile kernel (rows per tile
1, 2, 4, 8; 32 columns; 64 of K; split-K) and of the 64 x 64 tiles.

Tolerance: a sum of n products in any order, FMA or not, is within
n 2^-53 sum |r||x| (1 + small) of the exact sum; both sides obey it, so their
difference is held to 2 n 2^-53 sum |r||x| with the slack of 1 + 2^-20."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2605_22188_gb300 import kglm, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p,m", [
    (1, 1, 1), (63, 31, 1), (64, 32, 2), (65, 33, 3), (200, 30, 1), (200, 30, 8), (129, 33, 9), (2000, 30, 5),
    (5000, 31, 1), (200, 200, 64), (640, 97, 65), (1000, 300, 17), (3001, 65, 129),
])
def test_fp64_xtr_sizes(n, p, m):
    rng = np.random.default_rng(n * 1000 + p * 10 + m)
    X = rng.standard_normal((n, p)) * np.exp(rng.uniform(-3, 3, (1, p)))
    y = rng.standard_normal(n)
    R = rng.standard_normal((m, n))
    with kglm.Engine(X, y, 1, 1e-2, 2.0, synth.LSQ, prec="fp64", max_batch=m) as eng:
        r = torch.from_numpy(R).cuda()
        g = torch.full((m, p), float("nan"), device="cuda", dtype=torch.float64)
        for _ in range(2):                    # the second call finds the tile counters at 0 again
            kglm.kglm_xtr(eng.ctx, m, r.data_ptr(), g.data_ptr())
    tol = 2.0 * n * 2.0 ** -53 * (1 + 2.0 ** -20) * (np.abs(R) @ np.abs(X)) + 1e-300
    assert np.all(np.abs(g.cpu().numpy() - R @ X) <= tol)


@pytest.mark.parametrize("n,p", [(40, 1), (64, 8), (200, 30), (700, 257)])
def test_step_size_from_power_iteration(n, p):
    """The engine's step size against LAPACK's norm: a first FISTA step from 0 on the root
    with the budget open (k = p, kbar >= pf) is beta = clip(2 eta X^T y / (1 + c)), so the
    iterate gives eta.  The power iteration ends within its own stopping rule (1e-13 per
    step, at most 500 steps); on a spectrum with one dominant eigenvalue, a ratio of at
    most 0.9 in 500 steps, that is below 1e-10 relative, plus the engine's 1e-6 margin."""
    rng = np.random.default_rng(p)
    X = rng.standard_normal((n, p))
    X += 4.0 * np.outer(rng.standard_normal(n), np.ones(p))      # one dominant direction
    y = rng.standard_normal(n)
    k = min(p, kglm.MAX_K)
    lam2, M = 1e-2, 1e6
    J0 = list(range(k, p))                                       # all coordinates past k fixed out
    csr = synth.sets_to_csr([(J0, [])])
    with kglm.Engine(X, y, k, lam2, M, synth.LSQ, prec="fp64", max_batch=1) as eng:
        eng.push(*csr)
        eng.evaluate(1)
        B, _ = eng.read_batch(zeta=False)
    L = 2.0 * np.linalg.norm(X, 2) ** 2 * (1.0 + 1e-6)
    eta = 1.0 / L
    want = (2.0 * eta * (X.T @ y) / (1.0 + 2.0 * eta * lam2))[:k]
    assert np.linalg.norm(B[0, :k] - want) <= 1e-9 * np.linalg.norm(want)
