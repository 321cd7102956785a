"""kglm_read_batch after kglm_xtz: the rows of Z that the call put in the batch's dual points,
and the batch's own dual points behind them, as FP64 values in every mode (no tolerance)."""

import numpy as np
import pytest

pytest.importorskip("torch")

from paper_2605_22188_gb300 import kglm, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16", "tf32x3"])
@pytest.mark.parametrize("n,p,m", [(301, 40, 1), (301, 40, 7), (1024, 90, 130)])
def test_dual_points_after_xtz(prec, n, p, m):
    X, y, _ = synth.instance(n, p, 3, synth.LOGISTIC, seed=4)
    csr = synth.random_nodes(m, p, 3, np.random.default_rng(m))
    rng = np.random.default_rng(n + m)
    with kglm.Engine(X, y, 3, 1e-2, 2.0, synth.LOGISTIC, prec=prec, max_batch=m) as eng:
        for rows in sorted({1, m // 2, m - 1, m} - {0}):
            eng.push(*csr)
            eng.evaluate(6, 3)
            zeta = eng.read_batch()[1]
            for _ in range(2):                                   # a second call finds FP64 rows
                Z = rng.standard_normal((rows, n))
                eng.xtz(Z)
                got = eng.read_batch()[1]
                assert np.array_equal(got[:rows], Z)
                assert np.array_equal(got[rows:], zeta[rows:])
            eng.push(*csr)
            eng.evaluate(6, 3)
            assert np.array_equal(eng.read_batch()[1], zeta)
