"""Batches whose finished nodes leave the iterations and the checks, against the same batch
with every row kept (tiles set by hand to the default widths, which the rule leaves as
they are): the same bits.

A node's own arithmetic does not depend on the rows around it: its sums over K run in the
same order in the same split-K slices.  So nothing may differ (no tolerance)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2605_22188_gb300 import kglm, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["bf16", "tf32", "tf32x3"])
@pytest.mark.parametrize("loss", [synth.LSQ, synth.LOGISTIC])
@pytest.mark.parametrize("n,p,m", [(400, 90, 24), (1373, 611, 64), (2000, 200, 333), (5003, 1001, 700), (300, 2100, 2100)])
@pytest.mark.parametrize("quantile", [0.02, 0.6])
def test_rows_that_leave(prec, loss, n, p, m, quantile):
    X, y, _ = synth.instance(n, p, 5, loss, seed=1)
    csr = synth.random_nodes(m, p, 5, np.random.default_rng(m))
    with kglm.Engine(X, y, 5, 1e-2, 2.0, loss, prec=prec, max_batch=m) as eng:
        eng.push(*csr)
        ub = float(np.quantile(eng.evaluate(8)["lb"], quantile))
    out, left = [], 0
    for by_hand in (False, True):
        with kglm.Engine(X, y, 5, 1e-2, 2.0, loss, prec=prec, max_batch=m) as eng:
            if by_hand:
                up16 = lambda v: (v + 15) // 16 * 16
                eng.configure(link_tile_cols=128 if n > 256 else up16(n), grad_tile_cols=min(256, up16(p)), pair=-1)
            eng.set_incumbent(ub)
            eng.push(*csr)
            res = {}
            for run, (iters, every) in enumerate([(21, 4), (7, 3), (5, 0)]):   # goes on from the last one
                res.update({f"{key}{run}": v for key, v in eng.evaluate(iters, every).items()})
            left = int((res["iters_done0"] < 21).sum())
            res["B"], res["zeta"] = eng.read_batch()
            out.append(res)
    assert 0 < left, "no node finished early: nothing tested"
    for key in out[0]:
        assert np.array_equal(out[0][key], out[1][key], equal_nan=True), key
