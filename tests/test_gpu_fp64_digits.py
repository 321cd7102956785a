"""The FP64 digit products on the device: their error against the CUDA cores' on the same rows,
and the logistic link between the two products (sigma by integer arithmetic, csrc/fixed.cuh)."""

import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2605_22188_gb300 import kglm, synth

pytestmark = pytest.mark.gpu

LINE = 2.5e7                       # multiply-adds from which a product runs as digits


def _two_prod(a, b):
    """a b as an unevaluated sum of two doubles (Dekker 1971)."""
    c = 134217729.0
    ah, bh = c * a - (c * a - a), c * b - (c * b - b)
    al, bl = a - ah, b - bh
    p = a * b
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


def _xtr(eng, R, p):
    r = torch.from_numpy(np.ascontiguousarray(R)).cuda()
    g = torch.full((len(R), p), float("nan"), device="cuda", dtype=torch.float64)
    kglm.kglm_xtr(eng.ctx, len(R), r.data_ptr(), g.data_ptr())
    return g.cpu().numpy()


@pytest.mark.parametrize("n,p,m", [(2000, 200, 64), (2001, 199, 129), (5000, 1000, 8), (640, 1500, 300)])
def test_digits_are_no_further_off_than_the_cuda_cores(n, p, m):
    """Two rows as part of a call above the line and in a call of their own below it, in the
    root mean square against exact sums."""
    assert m * n * p >= LINE and 2 * n * p < LINE
    rng = np.random.default_rng(n + p + m)
    X, y, _ = synth.instance(n, p, 3, synth.LSQ, rho=0.7, seed=2)
    X = X * np.exp(rng.uniform(-4, 4, (1, p)))
    R = rng.standard_normal((m, n)) * np.exp(rng.uniform(-6, 6, (m, 1)))
    few = [0, m - 1]
    with kglm.Engine(X, y, 3, 1e-2, 2.0, synth.LSQ, prec="fp64", max_batch=m) as eng:
        before = eng.device_bytes()
        core = _xtr(eng, R[few], p)
        assert eng.device_bytes() == before                      # the CUDA cores
        digits = _xtr(eng, R, p)[few]
        assert eng.device_bytes() > before                       # digits
        assert np.array_equal(_xtr(eng, R[few], p), core)        # and the cores again
    want = np.array([[math.fsum(np.concatenate(_two_prod(R[b], X[:, j]))) for j in range(p)] for b in few])
    unit = np.abs(want).mean(1)[:, None]
    rms = [float(np.sqrt(np.mean(((g - want) / unit) ** 2))) for g in (digits, core)]
    assert rms[0] <= rms[1], rms


def test_logistic_link():
    """X the identity: S = V, G = R = -y sigma(-y V), so one step from V gives
    beta = (V - eta R) / (1 + 2 eta lambda2) with every coordinate free.  Units of 2^-53: the
    reference's exp, addition and division 5 of sigma, times eta = 4, the device's sigma 4.3, its
    S 2^-59; two roundings of the difference and two of the quotient, |V| + 4 each: 25 + 4 (|V| + 4)."""
    n = p = k = 64
    m, eta, lam2 = 8192, 4.0, 2.0 ** -20
    assert m * n * p >= LINE
    rng = np.random.default_rng(0)
    y = rng.choice([-1.0, 1.0], n)
    V = rng.uniform(-30, 30, (m, p))
    V[:64] = np.linspace(-30, 30, 64)[:, None]
    V[64:128] = rng.choice([-1, 1], (64, p)) * 2.0 ** rng.uniform(-60, 0, (64, p))
    csr = (np.zeros(m + 1, np.int32), np.zeros(0, np.int32)) * 2
    with kglm.Engine(np.eye(n), y, k, lam2, 64.0, synth.LOGISTIC, prec="fp64", max_batch=m, lipschitz=1 / eta) as eng:
        before = eng.device_bytes()
        eng.push(*csr, warm_B=V)
        held = eng.device_bytes()
        eng.evaluate(1)
        assert held > before and eng.device_bytes() > held       # digits
        B = eng.read_batch(zeta=False)[0]
    want = (V + eta * y / (1.0 + np.exp(y * V))) / (1.0 + 2.0 * eta * lam2)
    err = np.abs(B - want) * 2.0 ** 53 / (4.0 * np.abs(V) + 41.0)
    assert np.all(err <= 1.0), float(err.max())
