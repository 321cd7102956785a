"""The FP64 mode's v(S) of the logistic loss (one logarithm of a running product per thread
and 512 samples) against the sum over the samples in extended precision, at the returned
coefficients: margins from 1e-9 to past the exponential's range, and sample counts around
one, two and three chunks of 512 per thread.

Tolerance: the predictor's k products and sums carry (k + 2) 2^-53 sum |x_j b_j| per sample
into a term of slope at most 1; a term and its share of the thread's sum are within 8 units
of 2^-53 of max(term, the thread's sum), and the block's and the ridge's additions within
16 units of the total."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2605_22188_gb300 import kglm, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [31, 257, 2000, 131072, 131073, 300000])
@pytest.mark.parametrize("scale", [1e-9, 1.0, 30.0, 2000.0])
def test_objective(n, scale):
    p, k, m, M, lam2 = 12, 3, 9, 1.0, 1e-3
    X, y, _ = synth.instance(n, p, k, synth.LOGISTIC, seed=3)
    X = X * scale
    with kglm.Engine(X, y, k, lam2, M, synth.LOGISTIC, prec="fp64", max_batch=m) as eng:
        eng.push(*synth.random_nodes(m, p, k, np.random.default_rng(1)))
        res = eng.evaluate(5)
    Xl, yl = X.astype(np.longdouble), y.astype(np.longdouble)
    for b in range(m):
        S = res["support"][b]
        use = S >= 0
        x, beta = Xl[:, S[use]], res["beta_re"][b][use].astype(np.longdouble)
        t = -yl * (x @ beta)
        want = np.sum(np.maximum(t, 0) + np.log1p(np.exp(-np.abs(t)))) + lam2 * np.sum(beta * beta)
        unit = np.longdouble(2.0) ** -53
        tol = (k + 2) * unit * np.sum(np.abs(x) @ np.abs(beta)) + (8 * max(1.0, n / 256) + 16) * unit * want
        assert abs(np.longdouble(res["ub"][b]) - want) <= tol, (b, res["ub"][b], float(want))
