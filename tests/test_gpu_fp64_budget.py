"""The optional digits of the FP64 products against the buffers that a later call must have
(warm_B's staging, kglm_xtz's bounds): with a budget that holds the footprint and the digits
but not such a buffer beside them the call goes through, the digits are given back, and what
follows has the bits of a context that never held them."""

import numpy as np
import pytest

pytest.importorskip("torch")

from paper_2605_22188_gb300 import kglm, synth

pytestmark = pytest.mark.gpu

N, P_, M, K = 2000, 300, 64, 5


def _engine(X, y, budget):
    return kglm.Engine(X, y, K, 1e-2, 2.0, synth.LSQ, prec="fp64", max_batch=M, hbm_budget=budget)


@pytest.mark.parametrize("call", ["warm_B", "xtz"])
@pytest.mark.parametrize("slack", [64, 8 * M * P_ - 1024])
def test_first_use_buffers_come_before_the_digits(call, slack):
    X, y, _ = synth.instance(N, P_, K, synth.LSQ, seed=3)
    csr = synth.random_nodes(M, P_, K, np.random.default_rng(0))
    rng = np.random.default_rng(1)
    B, Z = rng.uniform(-1, 1, (M, P_)), rng.standard_normal((M, N))
    need = kglm.kglm_estimate_bytes(kglm.make_desc(N, P_, K, 1e-2, 2.0, synth.LSQ, "fp64", M))
    with _engine(X, y, 0) as eng:
        eng.push(*csr)
        eng.evaluate(2)
        digits = eng.device_bytes() - need
    assert digits > 0

    def later(eng):
        out = {}
        if call == "xtz":
            out["Q"], out["E"] = eng.xtz(Z)
        eng.push(*csr, warm_B=B if call == "warm_B" else None)
        out.update(eng.evaluate(12, 4))
        out["B"], out["zeta"] = eng.read_batch()
        return out

    with _engine(X, y, need + digits + slack) as eng:
        eng.push(*csr)
        eng.evaluate(12, 4)
        assert eng.device_bytes() == need + digits               # they were taken
        got = later(eng)
        assert eng.device_bytes() == need + 8 * M * P_           # and given back
    with _engine(X, y, need + 8 * M * P_) as eng:
        want = later(eng)
    for key in want:
        assert np.array_equal(want[key], got[key]), key


def test_without_a_budget_both_fit():
    X, y, _ = synth.instance(N, P_, K, synth.LSQ, seed=3)
    csr = synth.random_nodes(M, P_, K, np.random.default_rng(0))
    with _engine(X, y, 0) as eng:
        eng.push(*csr)
        eng.evaluate(2)
        held = eng.device_bytes()
        eng.push(*csr, warm_B=np.zeros((M, P_)))
        eng.evaluate(2)
        assert eng.device_bytes() == held + 8 * M * P_
