"""Index checks of large batches run on the device: the same errors as the host's (which the
three nodes around the fault, as a small batch, are checked by), and a refused batch
leaves the pushed one in place."""

import numpy as np
import pytest

pytest.importorskip("torch")

from paper_2605_22188_gb300 import kglm, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fault", ["range_in", "negative", "repeat_out", "overlap", "repeat_in", "offsets", "k"])
def test_refused_batches(fault):
    n, p, k, m = 300, 700, 6, 200
    X, y, _ = synth.instance(n, p, k, synth.LSQ, seed=0)
    good = synth.random_nodes(m, p, k, np.random.default_rng(0), max_out=600)
    assert good[1].size + good[3].size >= 32768
    ip, ii, op, oi = (a.copy() for a in good)
    b = next(b for b in range(50, m) if ip[b + 1] - ip[b] >= 2 and op[b + 1] - op[b] >= 2)
    if fault == "range_in":
        ii[ip[b]] = p
    elif fault == "negative":
        oi[op[b] + 1] = -1
    elif fault == "repeat_out":
        oi[op[b] + 1] = oi[op[b]]
    elif fault == "overlap":
        oi[op[b]] = ii[ip[b] + 1]
    elif fault == "repeat_in":
        ii[ip[b] + 1] = ii[ip[b]]
    elif fault == "offsets":
        op[b + 1], op[b] = op[b], op[b + 1]
    else:
        ip[1:b + 1] = 0
    i0, o0 = int(ip[b - 1]), int(op[b - 1])
    near = (ip[b - 1:b + 3] - i0, ii[i0:i0 + 4 * p], op[b - 1:b + 3] - o0, oi[o0:o0 + 4 * p])
    with kglm.Engine(X, y, k, 1e-2, 2.0, synth.LSQ, prec="bf16", max_batch=m) as eng:
        with pytest.raises(kglm.KglmError) as host:
            eng.push(*near)
        eng.push(*good)
        want = eng.evaluate(5)
        eng.push(*good)
        with pytest.raises(kglm.KglmError) as e:
            eng.push(ip, ii, op, oi)
        assert e.value.status == kglm.KGLM_EINVAL and str(e.value) == str(host.value)
        eng.m = m
        got = eng.evaluate(5)
    for key in want:
        assert np.array_equal(want[key], got[key]), key
