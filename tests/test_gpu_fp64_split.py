"""The FP64 products that run as BF16 digit products (about 10^7 FMAs and more),
against sums of exact products rounded once (math.fsum over Dekker products).

Bound: the digits of both operands stop at 2^-65 of their row scales (at most 4 max
each) and the levels past the eighth are left out, together below 8 n 2^-64 of the
product of the scales, 16 max|r| max|x_j|; the last operation rounds once (2^-53 of
the result).  The CUDA-core product of the same rows (a call below the line) must
not be nearer to the exact values than the digit product in the root mean square."""

import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2605_22188_gb300 import kglm, synth

pytestmark = pytest.mark.gpu


def _two_prod(a, b):
    """a b as an unevaluated sum of two doubles (Dekker 1971)."""
    c = 134217729.0
    ah = c * a - (c * a - a)
    bh = c * b - (c * b - b)
    al, bl = a - ah, b - bh
    p = a * b
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


def _exact(R, X, rows, cols):
    out = np.empty((len(rows), len(cols)))
    for i, b in enumerate(rows):
        for t, j in enumerate(cols):
            p, e = _two_prod(R[b], X[:, j])
            out[i, t] = math.fsum(np.concatenate([p, e]))
    return out


def _xtr(eng, R, p):
    m = R.shape[0]
    r = torch.from_numpy(np.ascontiguousarray(R)).cuda()
    g = torch.full((m, p), float("nan"), device="cuda", dtype=torch.float64)
    kglm.kglm_xtr(eng.ctx, m, r.data_ptr(), g.data_ptr())
    return g.cpu().numpy()


def _rows_cols(m, p):
    return sorted({0, m - 1, m // 2, min(m - 1, 128)}), sorted({0, p - 1, p // 2, min(p - 1, 255), min(p - 1, 17)})


@pytest.mark.parametrize("n,p,m", [
    (2000, 200, 64), (2001, 199, 129), (1023, 111, 256), (1025, 257, 300), (5000, 1000, 8), (20011, 129, 128),
    (640, 2000, 1000),
])
def test_digit_product_error(n, p, m):
    rng = np.random.default_rng(n + p + m)
    X, y, _ = synth.instance(n, p, 3, synth.LSQ, rho=0.7, seed=2)
    X = X * np.exp(rng.uniform(-4, 4, (1, p)))                   # features on their own scales
    R = rng.standard_normal((m, n)) * np.exp(rng.uniform(-6, 6, (m, 1)))
    R[m // 2] = 0.0                                              # a zero row stays exact
    with kglm.Engine(X, y, 3, 1e-2, 2.0, synth.LSQ, prec="fp64", max_batch=m) as eng:
        before = eng.device_bytes()
        G = _xtr(eng, R, p)
        assert eng.device_bytes() > before                       # the digits were set up
        few = [b for b in _rows_cols(m, p)[0] if len(R) * n * p >= 1e7][:2]
        Gc = _xtr(eng, R[few], p) if len(few) * n * p < 1e7 else None
    rows, cols = _rows_cols(m, p)
    want = _exact(R, X, rows, cols)
    scale = 16.0 * np.abs(R[rows]).max(1)[:, None] * np.abs(X[:, cols]).max(0)[None, :]
    tol = 8.0 * n * 2.0 ** -64 * scale + 2.0 ** -53 * np.abs(want)
    err = np.abs(G[np.ix_(rows, cols)] - want)
    assert np.all(err <= tol), float((err / np.maximum(tol, 1e-300)).max())
    assert np.all(G[m // 2] == 0.0)
    if Gc is not None:
        # over every column of those rows, each row in units of its own size
        w = _exact(R, X, few, range(p))
        unit = np.abs(w).mean(1)[:, None] + 1e-300
        rms = lambda e: float(np.sqrt(np.mean((e / unit) ** 2)))
        split, core = rms(G[few] - w), rms(Gc - w)
        print("n %d p %d: rms error, digits %.3g, FP64 pipe %.3g" % (n, p, split, core))
        assert split <= core


@pytest.mark.parametrize("prec,n", [("fp64", 33000), ("bf16", 22400)])
def test_levels_past_31_bits(prec, n):
    """Rows of one value whose leading bytes are all 127: the sums of a level's digit
    products pass 2^31 from n = 16640 on (six-digit levels from 22188), so they are held
    in parts.  FP64: X^T R against the exact sum (the bound above).  BF16: kglm_xtz
    within its own entrywise bound, at a size where it runs as digits (at 33000 its
    slices are too many and it is an FP64 sum with an entrywise bound of 0)."""
    p, m = 130, 128
    v = sum(127.0 * 2.0 ** (-8 * a) for a in range(1, 7))
    rng = np.random.default_rng(0)
    X = np.full((n, p), v) * rng.choice([1.0, 2.0, 0.5], (1, p))
    R = np.full((m, n), v) * rng.choice([1.0, -1.0, 4.0], (m, 1))
    y = rng.standard_normal(n)
    with kglm.Engine(X, y, 3, 1e-2, 2.0, synth.LSQ, prec=prec, max_batch=m, lipschitz=1e5) as eng:
        if prec == "fp64":
            before = eng.device_bytes()
            G = _xtr(eng, R, p)
            assert eng.device_bytes() > before
            err = np.zeros_like(G)
        else:
            G, err = eng.xtz(R)
            assert np.all(err > 0.0)                                 # digits, not the FP64 sum
    want = _exact(R, X, [0, 1, 77], [0, 1, 2, 129])
    tol = 8.0 * n * 2.0 ** -64 * 16.0 * np.abs(R[[0, 1, 77]]).max(1)[:, None] * np.abs(X[:, [0, 1, 2, 129]]).max(0)
    tol = tol + 2.0 ** -53 * np.abs(want) + err[np.ix_([0, 1, 77], [0, 1, 2, 129])]
    assert np.all(np.abs(G[np.ix_([0, 1, 77], [0, 1, 2, 129])] - want) <= tol)


@pytest.mark.parametrize("where", ["X", "R", "nan"])
def test_rows_spread_over_many_binades_keep_fp64(where):
    """An outlier of 10^9 in a column of X, or in a row of R next to it, would cost the
    fixed-point rows their low bits: those calls take the FP64 pipe, and keep the
    componentwise bound n 2^-53 sum |r||x| of an FP64 sum (2 n 2^-53 against numpy's)."""
    n, p, m = 3000, 150, 64
    rng = np.random.default_rng(5)
    X = rng.standard_normal((n, p))
    R = rng.standard_normal((m, n))
    if where == "X":
        X[7, 3] = 1e9
        R[:, 7] = 0.0
    elif where == "R":
        R[5, 11] = 1e9
        X[11, :] = 0.0
    else:
        R[5, 11] = np.nan
    y = rng.standard_normal(n)
    with kglm.Engine(X, y, 3, 1e-2, 2.0, synth.LSQ, prec="fp64", max_batch=m) as eng:
        G = _xtr(eng, R, p)
    if where == "nan":
        assert np.all(np.isnan(G[5])) and np.all(np.isfinite(np.delete(G, 5, 0)))
        return
    tol = 2.0 * n * 2.0 ** -53 * (1 + 2.0 ** -20) * (np.abs(R) @ np.abs(X))
    assert np.all(np.abs(G - R @ X) <= tol)


def test_budget_keeps_the_old_footprint():
    """A context that may hold no more than its estimate evaluates on the FP64 pipe and
    gives the same bounds (both FP64 sums of the same terms; 1e-12 over ten iterations)."""
    n, p, m, k = 2000, 300, 64, 5
    X, y, _ = synth.instance(n, p, k, synth.LSQ, seed=3)
    csr = synth.random_nodes(m, p, k, np.random.default_rng(0))
    out = []
    for tight in (False, True):
        need = kglm.kglm_estimate_bytes(kglm.make_desc(n, p, k, 1e-2, 2.0, synth.LSQ, "fp64", m))
        with kglm.Engine(X, y, k, 1e-2, 2.0, synth.LSQ, prec="fp64", max_batch=m,
                         hbm_budget=need if tight else 0) as eng:
            eng.push(*csr)
            out.append(eng.evaluate(10, 5))
            assert (eng.device_bytes() == need) == tight
    a, b = out
    for key in ("lb", "primal", "ub"):
        assert np.all(np.abs(a[key] - b[key]) <= 1e-12 * np.maximum(1.0, np.abs(a[key]))), key
    assert np.array_equal(a["support"], b["support"])
