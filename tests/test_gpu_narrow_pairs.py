"""Outputs of at most 16 columns with more than 128 nodes: one 16-column tile, which stays with
single CTAs however the pairs are set; 17 columns take a 32-column tile, in pairs.  The same bits
either way, and the certificate's product within its own bound."""

import numpy as np
import pytest

pytest.importorskip("torch")

from paper_2605_22188_gb300 import kglm, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [3, 16, 17])
@pytest.mark.parametrize("n,m", [(12, 300), (500, 129), (900, 400)])
def test_narrow_products(p, n, m):
    k = 3
    rng = np.random.default_rng(n + p)
    X, y = rng.standard_normal((n, p)), rng.standard_normal(n)
    csr = synth.random_nodes(m, p, k, rng)
    Z = rng.standard_normal((m, n))
    out = []
    with kglm.Engine(X, y, k, 1e-2, 2.0, synth.LSQ, prec="bf16", max_batch=m) as eng:
        for pair in (0, -1, 1):
            eng.configure(pair=pair)
            eng.push(*csr)
            res = eng.evaluate(9, 3)
            res["B"], res["zeta"] = eng.read_batch()
            res["Q"], res["E"] = eng.xtz(Z)
            out.append(res)
    for res in out[1:]:
        for key in res:
            assert np.array_equal(res[key], out[0][key]), key
    # the bound, and numpy's own n 2^-53 sum |z||x|
    slack = n * 2.0 ** -52 * (np.abs(Z) @ np.abs(X))
    assert np.all(np.abs(out[0]["Q"] - Z @ X) <= out[0]["E"] + slack)


def test_narrow_fp64_products():
    """m n p above the line from which FP64 products run as digits, 16 columns."""
    n, p, m, k = 4000, 16, 400, 3
    rng = np.random.default_rng(1)
    X, y = rng.standard_normal((n, p)), rng.standard_normal(n)
    csr = synth.random_nodes(m, p, k, rng)
    out = []
    need = kglm.kglm_estimate_bytes(kglm.make_desc(n, p, k, 1e-2, 2.0, synth.LSQ, "fp64", m))
    for budget in (0, need):
        with kglm.Engine(X, y, k, 1e-2, 2.0, synth.LSQ, prec="fp64", max_batch=m, hbm_budget=budget) as eng:
            eng.push(*csr)
            out.append(eng.evaluate(10, 5))
            assert (eng.device_bytes() > need) == (budget == 0)
    a, b = out
    for key in ("lb", "primal", "ub"):          # FP64 sums of the same terms over ten iterations
        assert np.all(np.abs(a[key] - b[key]) <= 1e-12 * np.maximum(1.0, np.abs(a[key]))), key
