"""Instance set-up by digit products: the Gram matrix through least-squares re-optimization.

v(S) and its coefficients come from the Gram block and X^T y alone, so they are compared
with LAPACK solves of the same normal equations: 1e-11 relative (a Gram matrix of
rho = 0.5 columns with condition below 100 and FP64 entries, a 5 x 5 Cholesky)."""

import numpy as np
import pytest

pytest.importorskip("torch")

from paper_2605_22188_gb300 import kglm, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "bf16", "fp32"])
@pytest.mark.parametrize("n,p,spread", [(2000, 320, 0.0), (1999, 257, 0.0), (1601, 513, 6.0), (2000, 320, 1e9)])
def test_gram_block_solutions(prec, n, p, spread):
    """spread: columns on scales e^(+-spread), or (1e9) one outlier, whose instance takes the FP64 pipe."""
    X, y, _ = synth.instance(n, p, 5, synth.LSQ, rho=0.5, seed=4)
    rng = np.random.default_rng(1)
    if spread > 100.0:
        X[3, 200] = spread
    elif spread:
        X *= np.exp(rng.uniform(-spread, spread, (1, p)))
    M = 1e9
    lam2 = 1e-3
    csr = synth.random_nodes(12, p, 5, rng, max_out=p // 2, max_in=5)
    with kglm.Engine(X, y, 5, lam2, M, synth.LSQ, prec=prec, max_batch=12) as eng:
        eng.push(*csr)
        res = eng.evaluate(3)
    for b in range(12):
        S = [j for j in res["support"][b] if j >= 0]
        if not S or 200 in S and spread > 100.0:
            continue
        A = X[:, S].T @ X[:, S] + lam2 * np.eye(len(S))
        d = 1.0 / np.sqrt(np.diag(A))                       # scaled, so that the columns' sizes drop out
        c = X[:, S].T @ y
        beta = d * np.linalg.solve(A * d[:, None] * d[None, :], d * c)
        assert np.linalg.norm((res["beta_re"][b, :len(S)] - beta) / d) <= 1e-11 * np.linalg.norm(beta / d)
        v = float(y @ y - c @ beta)
        assert abs(res["ub"][b] - v) <= 1e-11 * float(y @ y)
