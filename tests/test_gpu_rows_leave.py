"""Batches at the edges of the 128-row tiles whose finished nodes leave: the rows leave exactly
where the rule says (the operand gathers are counted among the layout launches), also twice in
one evaluation, and no bit differs from the same batch with every row kept (tiles set by hand
keep them).  The same in the searches of two requests of the serving loop."""

import numpy as np
import pytest

pytest.importorskip("torch")

from paper_2605_22188_gb300 import kglm, synth

pytestmark = pytest.mark.gpu

ITERS, EVERY = 41, 4


def _by_hand(eng, n, p):
    up16 = lambda v: (v + 15) // 16 * 16
    eng.configure(link_tile_cols=128 if n > 256 else up16(n), grad_tile_cols=min(256, up16(p)), pair=-1)


def _compactions(done, m):
    """How often rows leave, from the iterations after which each node was finished."""
    rows_now = times = 0
    for it in range(EVERY, ITERS, EVERY):
        left = int((done > it).sum())
        if left == 0:
            break
        rows = 16 if left <= 16 else -(-left // 32) * 32 if left <= 128 else -(-left // 128) * 128
        fewer = 4 * rows <= 3 * rows_now if rows_now else 4 * -(-rows // 128) <= 3 * -(-m // 128)
        if fewer:
            rows_now = rows
            times += 1
    return times


@pytest.mark.parametrize("prec", ["bf16", "tf32x3"])
@pytest.mark.parametrize("loss", [synth.LSQ, synth.LOGISTIC])
@pytest.mark.parametrize("n,p,m", [(400, 90, 128), (400, 90, 129), (1373, 611, 257), (2000, 200, 385), (900, 700, 513)])
def test_rows_leave_by_the_rule(prec, loss, n, p, m):
    X, y, _ = synth.instance(n, p, 5, loss, seed=1)
    csr = synth.random_nodes(m, p, 5, np.random.default_rng(m))
    with kglm.Engine(X, y, 5, 1e-2, 2.0, loss, prec=prec, max_batch=m) as eng:
        _by_hand(eng, n, p)
        eng.push(*csr)
        lb = eng.evaluate(8)["lb"]
        # the incumbent under which rows leave most often
        best = (-1, 0.0)
        for q in np.linspace(0.02, 0.98, 25):
            ub = float(np.quantile(lb, q))
            eng.set_incumbent(ub)
            eng.push(*csr)
            best = max(best, (_compactions(eng.evaluate(ITERS, EVERY)["iters_done"], m), ub))
    times, ub = best
    assert times >= (0 if m <= 128 else 1), times
    out, launches = [], []
    for hand in (False, True):
        with kglm.Engine(X, y, 5, 1e-2, 2.0, loss, prec=prec, max_batch=m) as eng:
            if hand:
                _by_hand(eng, n, p)
            eng.set_incumbent(ub)
            eng.push(*csr)
            res = eng.evaluate(ITERS, EVERY)
            launches.append(eng.stats()["layout"]["launches"])
            eng.evaluate(5, 2)
            res["B"], res["zeta"] = eng.read_batch()
            out.append(res)
    # one gather each time rows leave, one when the whole batch is back
    assert launches[0] - launches[1] == times + (times > 0)
    for key in out[0]:
        assert np.array_equal(out[0][key], out[1][key], equal_nan=True), key


def test_rows_leave_twice():
    """A batch whose nodes finish in three groups."""
    n, p, m, loss = 700, 60, 520, synth.LSQ
    X, y, _ = synth.instance(n, p, 5, loss, rho=0.9, snr=2.0, seed=7)
    csr = synth.random_nodes(m, p, 5, np.random.default_rng(3))
    out = []
    with kglm.Engine(X, y, 5, 1e-3, 2.0, loss, prec="bf16", max_batch=m) as eng:
        _by_hand(eng, n, p)
        eng.push(*csr)
        lb = eng.evaluate(8)["lb"]
        for ub in np.quantile(lb, np.linspace(0.01, 0.99, 60)):
            eng.set_incumbent(float(ub))
            eng.push(*csr)
            out.append((_compactions(eng.evaluate(ITERS, EVERY)["iters_done"], m), float(ub)))
    times, ub = max(out)
    assert times >= 2, "no incumbent makes rows leave twice"
    got = []
    for hand in (False, True):
        with kglm.Engine(X, y, 5, 1e-3, 2.0, loss, prec="bf16", max_batch=m) as eng:
            if hand:
                _by_hand(eng, n, p)
            eng.set_incumbent(ub)
            eng.push(*csr)
            res = eng.evaluate(ITERS, EVERY)
            res["n"] = eng.stats()["layout"]["launches"]
            got.append(res)
    assert got[0].pop("n") - got[1].pop("n") == times + 1
    for key in got[0]:
        assert np.array_equal(got[0][key], got[1][key], equal_nan=True), key


def test_requests_whose_rows_leave_are_the_same_alone_and_together():
    """Two BF16 searches whose batches pass 128 nodes and lose rows (shown on the context's own
    launches), through the serving loop alone and together: bit for bit."""
    specs = [(1500, 300, 10, 0.9, 3.0, 512), (2000, 400, 12, 0.9, 3.0, 512)]
    inst = []
    for i, (n, p, k, rho, snr, batch) in enumerate(specs):
        X, y, _ = synth.instance(n, p, k, synth.LSQ, rho=rho, snr=snr, seed=1 + i)
        inst.append((X, y, k, batch))
        layout = []
        for hand in (False, True):
            with kglm.Engine(X, y, k, 1e-3, 2.0, synth.LSQ, prec="bf16", max_batch=batch, open_cap=1 << 16) as eng:
                if hand:
                    _by_hand(eng, n, p)
                res = eng.solve_device(batch, 200, 10)
                layout.append((eng.stats()["layout"]["launches"], res["opt"], res["nodes"], res["batches"]))
        assert layout[0][0] > layout[1][0], "rows never left"
        assert layout[0][1:] == layout[1][1:]

    def serve(which):
        with kglm.Server(max_active=4, iters=200, check_every=10) as srv:
            ids = [srv.submit(X, y, k, 1e-3, 2.0, synth.LSQ, prec="bf16", max_batch=batch) for X, y, k, batch in which]
            srv.drain(timeout=300)
            infos = [srv.info(r) for r in ids]
            shared = srv.stats()["shared_launches"]
        assert all(r["state"] == kglm.REQ_DONE and r["gap"] <= 1e-6 for r in infos)
        return [(r["opt"], r["support"], r["nodes"], r["batches"]) for r in infos], shared

    alone = [serve([one])[0][0] for one in inst]
    together, shared = serve(inst)
    assert shared > 0 and together == alone
