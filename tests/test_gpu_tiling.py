"""Tiles and CTA pairs by rule against the default widths set by hand: the same bits.

A product's sums run over K in the same order at any column tile and in pairs, and the
rule keeps the number of split-K slices, so nothing may differ (no tolerance)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2605_22188_gb300 import kglm, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["bf16", "tf32", "tf32x3"])
@pytest.mark.parametrize("n,p,m", [(2500, 520, 1), (1373, 611, 129), (2000, 200, 1024), (3000, 700, 1000), (5003, 1001, 2100)])
def test_rule_gives_the_default_tiles_bits(prec, n, p, m):
    X, y, _ = synth.instance(n, p, 5, synth.LOGISTIC, seed=1)
    csr = synth.random_nodes(m, p, 5, np.random.default_rng(m))
    R = torch.from_numpy(np.random.default_rng(1).standard_normal((m, n)).astype(np.float32)).cuda()
    out = []
    for by_hand in (False, True):
        with kglm.Engine(X, y, 5, 1e-2, 2.0, synth.LOGISTIC, prec=prec, max_batch=m) as eng:
            if by_hand:
                up16 = lambda v: (v + 15) // 16 * 16
                eng.configure(link_tile_cols=128 if n > 256 else up16(n), grad_tile_cols=min(256, up16(p)), pair=-1)
            eng.push(*csr)
            res = eng.evaluate(6, 3)
            res["B"], _ = eng.read_batch(zeta=False)
            G = torch.empty(m, p, device="cuda")
            kglm.kglm_xtr(eng.ctx, m, R.data_ptr(), G.data_ptr())
            res["G"] = G.cpu().numpy()
            out.append(res)
    for key in out[0]:
        assert np.array_equal(out[0][key], out[1][key]), key
