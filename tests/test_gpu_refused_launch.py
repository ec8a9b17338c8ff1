"""A launch that the driver refuses (here: that the library is told to refuse on the host) is reported by the call it
belongs to, with its cause, and costs that call only: every handle goes on afterwards, and its results are the oracle's."""
import numpy as np
import pytest

from oracle import dsfacto_oracle as O
from paper_2004_13940_b200 import dsfacto as D
from paper_2004_13940_b200 import workloads as W

pytestmark = pytest.mark.gpu


def _refused(g, rc):
    return rc == D.ERR_CUDA and b"too many resources" in D.lib().dsfacto_last_error(g._h)


def _same(g, o):
    w0, w, V = g.get_params()
    assert w0 == pytest.approx(o.w0, abs=1e-5)
    assert np.abs(w - o.w).max() <= 1e-4 * (1 + np.abs(o.w).max()) and np.all(np.abs(V - o.V) <= 1e-4 * (1 + np.abs(o.V)))


# by column runs in one band and in several (tail composites), cut into segments, as a graph, and by tiles
@pytest.mark.parametrize("env,every,before", [({}, 0, 1), ({"DSFACTO_BANDS": "3"}, 0, 1), ({}, 2, 1), ({}, 0, 20),
                                              ({"DSFACTO_ROW_MERGE": "2"}, 0, 1), ({"DSFACTO_ROW_MERGE": "1"}, 2, 1)])
def test_a_refused_launch_of_an_epoch(monkeypatch, env, every, before):
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    wl = W.make("C1")
    o = O.Oracle(wl.n, wl.d, wl.K, wl.p, wl.loss, wl.lambda_w, wl.lambda_v, wl.eta, wl.init_seed)
    o.load_csr(wl.indptr, wl.indices, wl.values, wl.y)
    step = (lambda: o.epoch_segmented(every)) if every else o.epoch
    with D.DSFacto(wl.n, wl.d, wl.K, wl.p, wl.loss, wl.lambda_w, wl.lambda_v, wl.eta, wl.init_seed) as g:
        g.set_refresh_every(every)
        g.load_csr(wl.indptr, wl.indices, wl.values, wl.y)
        start = g.launch_count()
        for _ in range(before):
            assert g.epoch() == pytest.approx(step(), rel=1e-4)
        launches = 1 if before > 16 else (g.launch_count() - start) // before
        assert before > 16 or launches >= 3
        for k in range(1, launches + 1):
            params = g.get_params()
            g.debug_set(D.DEBUG_REFUSE_LAUNCH, k)
            assert _refused(g, D.dsfacto_epoch(g._h)), k
            if k > 1:       # parameters part of the way
                assert D.dsfacto_epoch(g._h) == D.ERR_CUDA and b"set the parameters again" in D.lib().dsfacto_last_error(g._h)
                g.set_params(*params)
            assert g.epoch() == pytest.approx(step(), rel=1e-4), k
            _same(g, o)


@pytest.mark.parametrize("m", [10, 300, 3000])      # through the mailbox in two and in many blocks; copied and checked on the device
def test_a_refused_launch_of_other_calls(m):
    wl = W.make("C3", n=3000)
    ip = wl.indptr[: m + 1].copy()
    ix, v, y, out = wl.indices[: ip[-1]].copy(), wl.values[: ip[-1]].copy(), wl.y[:m].copy(), np.empty(m, np.float32)
    bad = ix.copy()
    bad[0] = wl.d
    with D.DSFacto(wl.n, wl.d, 30, wl.p, wl.loss, wl.lambda_w, wl.lambda_v, wl.eta, 3) as g:      # (30: rows are padded)
        o = O.Oracle(wl.n, wl.d, 30, wl.p, wl.loss, wl.lambda_w, wl.lambda_v, wl.eta, 3)
        o.load_csr(wl.indptr, wl.indices, wl.values, wl.y)
        f = o.predict(ip, ix, v)
        w, V = np.empty(wl.d, np.float32), np.empty((wl.d, 30), np.float32)
        calls = {"load": lambda: D.dsfacto_load_csr(g._h, wl.indptr, wl.indices, wl.values, wl.y),
                 "predict": lambda: D.dsfacto_predict(g._h, m, ip, ix, v, out),
                 "predict unsound": lambda: D.dsfacto_predict(g._h, m, ip, bad, v, out),
                 "evaluate": lambda: D.dsfacto_evaluate(g._h, m, ip, ix, v, y)[0],
                 "get": lambda: D.dsfacto_get_params(g._h, None, w, V),
                 "set": lambda: D.dsfacto_set_params(g._h, None, w, V)}
        for name, call in calls.items():
            want = D.ERR_INVALID_CSR if name.endswith("unsound") else D.OK
            for k in range(1, 40):
                before = g.launch_count()
                g.debug_set(D.DEBUG_REFUSE_LAUNCH, k)
                rc = call()
                g.debug_set(D.DEBUG_REFUSE_LAUNCH, 0)
                if rc == want:        # fewer than k launches
                    assert k > 1 or name.endswith("unsound")
                    break
                assert _refused(g, rc) or name.endswith("unsound"), (name, k)
                assert g.launch_count() - before < k      # (launches that follow the refused one are left out)
                assert call() == want, (name, k)
                np.testing.assert_allclose(g.predict(ip, ix, v), f, rtol=0, atol=2e-5 * (1 + np.abs(f).max()))
            assert call() == want
        assert g.epoch() == pytest.approx(o.epoch(), rel=1e-4)
        _same(g, o)


def test_a_handle_does_not_train_on_half_of_the_parameters_it_was_given():
    wl = W.make("C1")
    K = 7                          # padded on the device: the launch that is refused
    o = O.Oracle(wl.n, wl.d, K, wl.p, wl.loss, wl.lambda_w, wl.lambda_v, wl.eta, 3)
    o.load_csr(wl.indptr, wl.indices, wl.values, wl.y)
    rng = np.random.default_rng(1)
    w, V = rng.standard_normal(wl.d).astype(np.float32), rng.standard_normal((wl.d, K)).astype(np.float32)
    with D.DSFacto(wl.n, wl.d, K, wl.p, wl.loss, wl.lambda_w, wl.lambda_v, wl.eta, 3) as g:
        g.load_csr(wl.indptr, wl.indices, wl.values, wl.y)
        g.debug_set(D.DEBUG_REFUSE_LAUNCH, 1)
        assert _refused(g, D.dsfacto_set_params(g._h, None, w, V))
        assert D.dsfacto_epoch(g._h) == D.ERR_CUDA and b"set the parameters again" in D.lib().dsfacto_last_error(g._h)
        g.set_params(None, w, V)
        o.w[:], o.V[:] = w, V
        o.refresh()
        assert g.epoch() == pytest.approx(o.epoch(), rel=1e-4)
        _same(g, o)


@pytest.mark.parametrize("env", [{"DSFACTO_BANDS": "3"}, {}, {"DSFACTO_ROW_MERGE": "2"}])
def test_parameters_left_part_of_the_way_are_scored_as_they_are(monkeypatch, env):
    # what an epoch that broke off leaves behind is no result, but scores and a new load go by it as by any parameters
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    wl = W.make("C1")
    ip = wl.indptr[:1001]
    ix, v = wl.indices[: ip[-1]].copy(), wl.values[: ip[-1]].copy()
    o = O.Oracle(wl.n, wl.d, wl.K, wl.p, wl.loss, wl.lambda_w, wl.lambda_v, 50.0, wl.init_seed)
    o.load_csr(wl.indptr, wl.indices, wl.values, wl.y)
    for k in range(2, 9):
        with D.DSFacto(wl.n, wl.d, wl.K, wl.p, wl.loss, wl.lambda_w, wl.lambda_v, 50.0, wl.init_seed) as g:
            g.load_csr(wl.indptr, wl.indices, wl.values, wl.y)
            w0 = g.get_params()[0]
            g.debug_set(D.DEBUG_REFUSE_LAUNCH, k)
            if D.dsfacto_epoch(g._h) == D.OK:
                break
            w0_after, w, V = g.get_params()
            assert w0_after == w0
            o.w0, o.w[:], o.V[:] = float(w0), w, V
            o.refresh()
            f = o.predict(ip, ix, v)
            np.testing.assert_allclose(g.predict(ip, ix, v), f, rtol=0, atol=2e-5 * (1 + np.abs(f).max()))
            g.load_csr(wl.indptr, wl.indices, wl.values, wl.y)
            assert g.objective() == pytest.approx(o.objective, rel=1e-5), k
            A, G = g.get_aux()
            np.testing.assert_allclose(G, o.G, rtol=0, atol=2e-5 * (1 + np.abs(o.G).max()))
