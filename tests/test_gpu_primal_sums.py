"""The primal value Phi of the reduced-precision modes at given FP32 coefficients, with the
ridge weight so large that only the sum of squares of Theorem 4.1 counts (at most k nonzeros,
no fixings: G = lambda2 sum beta^2).  Up to 512 coordinates the sum is an FP64 one.

Bound: a square of an FP32 value is exact in FP64; at most 4 terms per thread, 5 steps in a
warp, 4 warps and the loss are added with one rounding each, all terms non-negative: 14 2^-53
of the result, the losses' own error below 2^-53 of it; 2 lambda2 is a power of two."""

import math

import numpy as np
import pytest

pytest.importorskip("torch")

from paper_2605_22188_gb300 import kglm, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["bf16", "tf32x3"])
@pytest.mark.parametrize("p,k", [(30, 30), (64, 33), (128, 40), (129, 60), (200, 60), (512, 64)])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** 70])
def test_sum_of_squares(prec, p, k, scale):
    n, m, lam2 = 96, 200, 2.0 ** 27
    rng = np.random.default_rng(p + k)
    X = 1e-4 * rng.standard_normal((n, p))
    y = 1e-3 * rng.standard_normal(n)
    B = np.zeros((m, p), dtype=np.float32)
    for b in range(m):
        at = rng.choice(p, size=rng.integers(k // 2, k + 1), replace=False)
        B[b, at] = rng.standard_normal(at.size) * np.exp(rng.uniform(-2, 1, at.size))
    B = np.clip(B, -30, 30).astype(np.float64) * scale
    csr = (np.zeros(m + 1, np.int32), np.zeros(0, np.int32)) * 2
    with kglm.Engine(X, y, k, lam2, 64.0 * scale, synth.LSQ, prec=prec, max_batch=m) as eng:
        eng.push(*csr, warm_B=B)
        primal = eng.evaluate(0)["primal"]
        assert np.array_equal(eng.read_batch(zeta=False)[0], B)
    want = np.array([lam2 * math.fsum(v * v for v in row) for row in B])
    loss = ((B @ X.T - y) ** 2).sum(1)
    assert np.all(loss * 2.0 ** -18 < 2.0 ** -53 * want)          # (its FP32 terms' error)
    err = np.abs(primal - (want + loss)) / want
    assert np.all(err <= 15 * 2.0 ** -53), float(err.max() * 2 ** 53)
