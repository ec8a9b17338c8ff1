"""Several threads, each with a handle of its own, share the memory pool, the transfers and the result buffers of the
process: what each gets is, bit for bit, what it gets alone."""
import threading

import numpy as np
import pytest

from paper_2004_13940_b200 import dsfacto as D
from paper_2004_13940_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("own_streams", [False, True])
def test_threads_with_handles_of_their_own(own_streams):
    import torch

    big, small = W.make("C3", n=40_000), W.make("C3", n=4_000)       # arrays of 8 MB (several threads carry them) and of 0.8 MB
    rng = np.random.default_rng(5)
    w, V = (0.1 * rng.standard_normal(big.d)).astype(np.float32), (0.1 * rng.standard_normal((big.d, 32))).astype(np.float32)

    def stream(g):
        if not own_streams:
            return None
        s = torch.cuda.Stream()
        g.set_stream(s.cuda_stream)
        return s

    def train(wl):
        out = []
        for _ in range(3):
            with D.DSFacto(wl.n, wl.d, wl.K, wl.p, wl.loss, wl.lambda_w, wl.lambda_v, wl.eta, wl.init_seed) as g:
                kept = stream(g)
                g.load_csr(wl.indptr, wl.indices, wl.values, wl.y)
                out += [np.float64(g.epoch()) for _ in range(20)]
                out += [np.array(a) for a in g.get_params()[1:]]
                g.set_stream(0)
                del kept
        return out

    def score(m):
        ip = big.indptr[: m + 1]
        ix, v, y = big.indices[: ip[-1]], big.values[: ip[-1]], big.y[:m]
        out = []
        with D.DSFacto(1, big.d, 32, 1, D.LOGISTIC, 0.0, 0.0, 0.1, 1) as g:
            kept = stream(g)
            g.set_params(0.25, w, V)
            for _ in range(40):
                out += [g.predict(ip, ix, v), np.array(g.evaluate(ip, ix, v, y))]
            g.set_stream(0)
            del kept
        return out

    jobs = [lambda: train(big), lambda: train(small), lambda: score(40_000), lambda: score(2_000), lambda: score(20)]
    alone = [job() for job in jobs]
    got, errors = [None] * len(jobs), []
    start = threading.Barrier(len(jobs) + 1)

    def body(k):
        try:
            start.wait()
            got[k] = jobs[k]()
        except Exception as e:      # (told by the thread that can)
            errors.append((k, e))

    team = [threading.Thread(target=body, args=(k,)) for k in range(len(jobs))]
    for t in team:
        t.start()
    start.wait()
    while any(t.is_alive() for t in team):
        D.dsfacto_trim()            # memory that is kept for the next call may go at any time
        team[0].join(0.02)
        for t in team:
            if not t.is_alive():
                t.join()
    assert not errors, errors
    for a, b in zip(alone, got):
        assert len(a) == len(b) and all(np.array_equal(x, y) for x, y in zip(a, b))
