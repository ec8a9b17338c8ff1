"""Edges of the ways a call takes between host and device: scoring batches that go through the mailbox or are copied; launches of an epoch one by one and as a graph; results in ordinary and in page-locked
arrays; the entry point that allocates nothing at every factor width it takes."""
import numpy as np
import pytest

from oracle import dsfacto_oracle as O
from paper_2004_13940_b200 import dsfacto as D
from paper_2004_13940_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [5, 16, 32, 64, 128, 200])
@pytest.mark.parametrize("m", [1, 40, 63, 64, 65, 290, 300, 310, 4000])
def test_scoring_batches_of_every_size(m, K):
    # about 50 entries per row: the mailbox (127 KB) is full near 310 rows, larger batches are copied; a CTA has 8 rows
    wl = W.make("C3", n=4000)
    ip = wl.indptr[: m + 1].copy()
    ix, v, y = wl.indices[: ip[-1]].copy(), wl.values[: ip[-1]].copy(), wl.y[:m].copy()
    rng = np.random.default_rng(K)
    w, V = (0.1 * rng.standard_normal(wl.d)).astype(np.float32), (0.1 * rng.standard_normal((wl.d, K))).astype(np.float32)
    with D.DSFacto(1, wl.d, K, 1, D.LOGISTIC, 0.0, 0.0, 0.1, 1) as g:
        g.set_params(0.25, w, V)
        rows = np.repeat(np.arange(m), np.diff(ip))
        x, Vx = v.astype(np.float64), v[:, None].astype(np.float64) * V[ix]
        A = np.add.reduceat(Vx, ip[:-1], axis=0)      # (no row is empty)
        f = 0.25 + np.bincount(rows, x * w[ix], m) + 0.5 * ((A * A).sum(1) - np.bincount(rows, (Vx * Vx).sum(1), m))
        for _ in range(3):
            np.testing.assert_allclose(g.predict(ip, ix, v), f, rtol=0, atol=2e-5 * (1 + np.abs(f).max()))
        loss, acc = g.evaluate(ip, ix, v, y)
        assert loss == pytest.approx(np.logaddexp(0.0, -y * f).mean(), rel=1e-5)
        assert abs(acc - np.mean(y * f > 0)) * m <= np.count_nonzero(np.abs(f) <= 2e-5 * (1 + np.abs(f).max())) + 1e-9
        # an unsound batch is refused on every way, and the next sound one is served
        bad_ix, bad_v, bad_y = ix.copy(), v.copy(), y.copy()
        bad_ix[-1], bad_v[-1], bad_y[-1] = wl.d, np.inf, np.nan
        out = np.empty(m, np.float32)
        assert D.dsfacto_predict(g._h, m, ip, bad_ix, v, out) == D.ERR_INVALID_CSR
        assert D.dsfacto_predict(g._h, m, ip, ix, bad_v, out) == D.ERR_INVALID_CSR
        assert D.dsfacto_evaluate(g._h, m, ip, ix, v, bad_y)[0] == D.ERR_INVALID_CSR
        assert D.dsfacto_predict(g._h, m, ip, ix, v, out) == D.OK
        np.testing.assert_allclose(out, f, rtol=0, atol=2e-5 * (1 + np.abs(f).max()))


@pytest.mark.parametrize("every", [0, 2])
def test_epochs_before_and_after_they_become_a_graph(every):
    wl = W.make("C1")
    o = O.Oracle(wl.n, wl.d, wl.K, wl.p, wl.loss, wl.lambda_w, wl.lambda_v, wl.eta, wl.init_seed)
    o.load_csr(wl.indptr, wl.indices, wl.values, wl.y)
    with D.DSFacto(wl.n, wl.d, wl.K, wl.p, wl.loss, wl.lambda_w, wl.lambda_v, wl.eta, wl.init_seed) as g:
        g.set_refresh_every(every)
        g.load_csr(wl.indptr, wl.indices, wl.values, wl.y)
        before = g.launch_count()
        g.epoch(), (o.epoch_segmented(every) if every else o.epoch())
        per_epoch = g.launch_count() - before
        for e in range(60):
            if e == 25:      # other kernel arguments: the graph has to go
                o.set_eta(0.5), g.set_eta(0.5)
            if e == 45:      # other parameters: the graph stays
                w, V = (0.9 * o.w).astype(np.float32), (0.9 * o.V).astype(np.float32)
                g.set_params(0.1, w, V)
                o.w0, o.w[:], o.V[:] = float(np.float32(0.1)), w, V
                o.refresh()
            before = g.launch_count()
            want, got = (o.epoch_segmented(every) if every else o.epoch()), g.epoch()
            assert got == pytest.approx(want, rel=1e-4), e
            assert g.launch_count() - before == per_epoch
        w0, w, V = g.get_params()
        assert np.abs(w - o.w).max() <= 1e-4 * (1 + np.abs(o.w).max()) and np.all(np.abs(V - o.V) <= 1e-4 * (1 + np.abs(o.V)))


@pytest.mark.parametrize("d,K", [(700, 45), (40_000, 20), (300_001, 7)])
def test_parameters_come_back_whole(d, K):
    # through the mailbox, through the driver, through several threads; several arrays alive at a time, and after a trim
    rng = np.random.default_rng(d)
    with D.DSFacto(1, d, K, 1, D.SQUARED, 0.0, 0.0, 0.1, 1) as g:
        kept = []
        for k in range(5):
            w, V = rng.standard_normal(d).astype(np.float32), rng.standard_normal((d, K)).astype(np.float32)
            g.set_params(float(k), w, V)
            kept.append((g.get_params(), (float(k), w, V)))
            if k == 2:
                D.dsfacto_trim()
        for (w0, w, V), (rw0, rw, rV) in kept:
            assert w0 == rw0 and np.array_equal(w, rw) and np.array_equal(V, rV)


@pytest.mark.parametrize("K", [4, 8, 16, 32, 64, 128, 256])
@pytest.mark.parametrize("m", [1, 1003])
def test_allocation_free_scoring_at_every_width(K, m):
    import torch

    wl = W.make("C3", n=1003)
    ip = wl.indptr[: m + 1].copy()
    ip[m // 2 + 1:] -= ip[m // 2 + 1] - ip[m // 2] if m > 1 else 0      # one row in the middle is empty
    ix, v, y = wl.indices[: ip[-1]].copy(), wl.values[: ip[-1]].copy(), wl.y[:m].copy()
    for i in range(m // 2, m):                                           # (rows behind it take what lies there)
        ix[ip[i]:ip[i + 1]] = np.sort(np.random.default_rng(i).choice(wl.d, ip[i + 1] - ip[i], replace=False))
    rng = np.random.default_rng(K)
    w, V = (0.1 * rng.standard_normal(wl.d)).astype(np.float32), (0.1 * rng.standard_normal((wl.d, K))).astype(np.float32)
    with D.DSFacto(1, wl.d, K, 1, D.LOGISTIC, 0.0, 0.0, 0.1, 1) as g:
        g.set_params(0.25, w, V)
        want = g.predict(ip, ix, v)
        loss, _ = g.evaluate(ip, ix, v, y)
    t = [torch.from_numpy(a).cuda() for a in (ip, ix, v, y, w, V)]
    scores, sums = torch.empty(m, device="cuda"), torch.empty(2, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert D.dsfacto_score_loss_noalloc(m, wl.d, K, D.LOGISTIC, *[a.data_ptr() for a in t[:4]], 0.25, t[4].data_ptr(),
                                        t[5].data_ptr(), scores.data_ptr(), sums.data_ptr()) == D.OK
    np.testing.assert_allclose(scores.cpu().numpy(), want, rtol=0, atol=2e-5 * (1 + np.abs(want).max()))
    assert float(sums[0]) == pytest.approx(loss * m, rel=1e-5)


def _short_rows(m, per_row, d, seed):
    rng = np.random.default_rng(seed)
    ix = (np.sort(rng.integers(0, d // per_row, (m, per_row)), axis=1) + np.arange(per_row) * (d // per_row)).astype(np.int32)
    return np.arange(m + 1, dtype=np.int64) * per_row, ix.ravel(), rng.standard_normal(m * per_row).astype(np.float32)


@pytest.mark.parametrize("K,per_row", [(8, 1), (32, 1), (32, 3), (128, 8)])
@pytest.mark.parametrize("m", [33, 96, 129, 160, 256, 300, 1200])
def test_batches_of_short_rows(K, per_row, m):
    # many rows of few entries: blocks of 8 rows, full and with a rest, as many CTAs as there are blocks
    d = 4096
    ip, ix, v = _short_rows(m, per_row, d, m)
    rng = np.random.default_rng(K)
    w, V = rng.standard_normal(d).astype(np.float32), (0.3 * rng.standard_normal((d, K))).astype(np.float32)
    with D.DSFacto(1, d, K, 1, D.SQUARED, 0.0, 0.0, 0.1, 1) as g:
        g.set_params(0.25, w, V)
        f = O.score(ip, ix, v, 0.25, w.astype(np.float64), V.astype(np.float64))
        for _ in range(2):
            np.testing.assert_allclose(g.predict(ip, ix, v), f, rtol=0, atol=2e-5 * (1 + np.abs(f).max()))


def test_many_short_rows_do_not_wait_for_copies_of_the_whole_batch():
    # 5000 rows of one entry are 100 KB in 209 CTAs, each of which fetches its own block: 32 us, 300 rows 14 us.  If each fetched
    # the batch, 20 MB would cross the link: 400 us.
    import time

    d, K = 8192, 32
    with D.DSFacto(1, d, K, 1, D.SQUARED, 0.0, 0.0, 0.1, 1) as g:
        def median_us(m):
            ip, ix, v = _short_rows(m, 1, d, 1)
            out, took = np.empty(m, np.float32), []
            for _ in range(300):
                t = time.perf_counter()
                assert D.dsfacto_predict(g._h, m, ip, ix, v, out) == D.OK
                took.append(time.perf_counter() - t)
            return 1e6 * float(np.median(took[50:]))

        median_us(300)
        assert min(median_us(5000) for _ in range(3)) <= 6 * min(median_us(300) for _ in range(3))


@pytest.mark.parametrize("n", [2_000, 40_000])
def test_page_locked_arrays_belong_to_the_caller_again_on_return(n):
    # copies of page-locked arrays are queued, not made, while a call is under way; each call has read them when it returns
    import torch

    def pinned(a):
        t = torch.empty(a.shape, dtype=torch.from_numpy(a[:1]).dtype, pin_memory=True)
        t.numpy()[...] = a
        return t.numpy()

    wl = W.make("C3", n=n)
    rng = np.random.default_rng(n)
    w, V = (0.1 * rng.standard_normal(wl.d)).astype(np.float32), (0.1 * rng.standard_normal((wl.d, wl.K))).astype(np.float32)
    got = []
    for make, spoil in ((np.array, False), (pinned, True)):
        def call(f, *arrays):
            arrays = [make(a) for a in arrays]
            out = f(*arrays)
            if spoil:
                for a in arrays:
                    a.view(np.uint8)[...] = 0xFF
            return out

        with D.DSFacto(wl.n, wl.d, wl.K, wl.p, wl.loss, wl.lambda_w, wl.lambda_v, wl.eta, wl.init_seed) as g:
            call(g.load_csr, wl.indptr, wl.indices, wl.values, wl.y)
            objective = [g.epoch() for _ in range(2)]
            call(lambda a, b: g.set_params(0.5, a, b), w, V)
            objective.append(g.epoch())
            f = call(g.predict, wl.indptr, wl.indices, wl.values)
            held = call(g.evaluate, wl.indptr, wl.indices, wl.values, wl.y)
            got.append((objective, held, f, *g.get_params()))
    for a, b in zip(*got):
        assert np.array_equal(np.asarray(a), np.asarray(b))


def _batch(lens, d, seed):
    lens, rng = np.asarray(lens), np.random.default_rng(seed)
    ip = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    ix = np.concatenate([np.sort(rng.choice(d, n, replace=False)) for n in lens]).astype(np.int32)
    return ip, ix, rng.standard_normal(len(ix)).astype(np.float32), np.where(rng.random(len(lens)) < 0.5, 1.0, -1.0).astype(np.float32)


_uneven = np.random.default_rng(5)
RAGGED = {
    "one of 400 among 8s": [8] * 500 + [400] + [8] * 500,
    "one long among 8s, to the last bytes": [8] * 800 + [408] + [8] * 878,                # 12 m + 8 + 8 nnz: 128 KB less the reports
    "log-normal, mean 40": _uneven.lognormal(np.log(40) - 0.5, 1.0, 300).astype(int).clip(1, 2000),
    "log-normal, mean 8": _uneven.lognormal(np.log(8) - 0.5, 1.0, 700).astype(int).clip(1, 2000),
    "26 to 76": _uneven.integers(26, 77, 300),
    "a long row and 2000 empty ones": [0] * 1000 + [9000] + [0] * 1000,
}


@pytest.mark.parametrize("K", [8, 32, 128])
@pytest.mark.parametrize("shape", sorted(RAGGED))
def test_ragged_batches_go_through_the_mailbox(K, shape):
    """One launch, whatever the longest row, while the batch's own bytes fit; and the scores that its rows have in a batch
    that is too large for it."""
    d = 20000
    ip, ix, v, y = _batch(RAGGED[shape], d, K)
    m = len(y)
    assert 12 * m + 8 + 8 * len(ix) <= (128 << 10) - 256
    rng = np.random.default_rng(K)
    with D.DSFacto(1, d, K, 1, D.LOGISTIC, 0.0, 0.0, 0.1, 1) as g:
        w, V = (0.1 * rng.standard_normal(d)).astype(np.float32), (0.1 * rng.standard_normal((d, K))).astype(np.float32)
        g.set_params(0.25, w, V)
        copied = g.predict(np.concatenate([ip, ip[-1] + ip[1:], 2 * ip[-1] + np.arange(1, 12001)]),
                           np.concatenate([ix, ix, np.arange(12000, dtype=np.int32) % d]), np.concatenate([v, v, np.ones(12000, np.float32)]))
        before = g.launch_count()
        f = g.predict(ip, ix, v)
        assert g.launch_count() - before == 1
        assert np.array_equal(f, copied[:m]) and np.array_equal(f, copied[m:2 * m])
        loss, acc = g.evaluate(ip, ix, v, y)
        assert g.launch_count() - before == 2
        assert loss == pytest.approx(np.logaddexp(0.0, -y * f.astype(np.float64)).mean(), rel=1e-5)
        assert acc == pytest.approx(np.mean(y * f > 0), abs=1e-12)


REQUESTS = {
    "steps": [7, 8, 9, 31, 32, 33, 63, 64, 65, 0, 127, 128, 129, 1, 0, 15, 16, 17],   # around the entries of a warp's step
    "several rows per warp": list(np.random.default_rng(0).integers(0, 4, 2500)),
    "more than 24 KB in a block": [0, 3100, 1, 64, 0],
    "more than 48 KB in a block": [5, 6500, 3100, 0, 64],
    "one row of 96 KB": [12000],
    "too large for the mailbox": [3, 16300, 0],
    "empty rows": [0] * 9,
}


@pytest.mark.parametrize("K", [4, 8, 16, 32, 64, 128, 200])
@pytest.mark.parametrize("shape", sorted(REQUESTS))
def test_requests_in_blocks_of_rows(K, shape):
    lens = np.array(REQUESTS[shape])
    rng = np.random.default_rng(K)
    d, m = 20000, len(lens)
    ip = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    ix = np.concatenate([np.sort(rng.choice(d, n, replace=False)) for n in lens]).astype(np.int32)
    v = rng.standard_normal(len(ix)).astype(np.float32) / np.sqrt(np.repeat(lens, lens).clip(1)).astype(np.float32)
    y = np.where(rng.random(m) < 0.5, 1.0, -1.0).astype(np.float32)
    w, V = (0.1 * rng.standard_normal(d)).astype(np.float32), (0.1 * rng.standard_normal((d, K))).astype(np.float32)
    rows = np.repeat(np.arange(m), lens)
    x, A, q = v.astype(np.float64), np.zeros((m, K)), np.zeros(m)
    np.add.at(A, rows, x[:, None] * V[ix])
    np.add.at(q, rows, x * x * (V[ix].astype(np.float64) ** 2).sum(1))
    f = 0.25 + np.bincount(rows, x * w[ix], m) + 0.5 * ((A * A).sum(1) - q)
    # fp32 sums of up to 16300 products whose squares add up to one: error below 16300 * 2^-24 in the worst order
    tol = 2e-5 * (1 + np.abs(f).max())
    for loss, code in ((D.LOGISTIC, "logistic"), (D.SQUARED, "squared")):
        with D.DSFacto(1, d, K, 1, loss, 0.0, 0.0, 0.1, 1) as g:
            g.set_params(0.25, w, V)
            for _ in range(2):
                np.testing.assert_allclose(g.predict(ip, ix, v), f, rtol=0, atol=tol)
            mean, metric = g.evaluate(ip, ix, v, y)
            if loss == D.LOGISTIC:
                assert mean == pytest.approx(np.logaddexp(0.0, -y * f).mean(), rel=1e-5, abs=tol)
                assert abs(metric - np.mean(y * f > 0)) * m <= np.count_nonzero(np.abs(f) <= tol) + 1e-9
            else:
                assert mean == pytest.approx(0.5 * np.mean((f - y) ** 2), rel=1e-4)
                assert metric == pytest.approx(np.sqrt(np.mean((f - y) ** 2)), rel=1e-4)
            if len(ix) > 1 and lens.max() > 1:   # columns that do not rise inside a row, beside falls from row to row
                t = int(ip[np.argmax(lens)]) + 1
                bad = ix.copy()
                bad[t] = bad[t - 1]
                assert D.dsfacto_predict(g._h, m, ip, bad, v, np.empty(m, np.float32)) == D.ERR_INVALID_CSR
                falling = ip.copy()
                falling[np.argmax(lens) + 1] = ip[np.argmax(lens)] - 1 if ip[np.argmax(lens)] > 0 else len(ix) + 1
                if m > 1 and falling[-1] == ip[-1]:
                    assert D.dsfacto_predict(g._h, m, falling, ix, v, np.empty(m, np.float32)) == D.ERR_INVALID_CSR


@pytest.mark.parametrize("K", [3, 8, 16, 20, 64, 128, 190, 256])
@pytest.mark.parametrize("d", [150, 3000])        # 128 factors and more: both widths of the recompute kernel's lane groups
def test_a_row_on_its_own_has_the_score_it_has_among_others(K, d):
    rng = np.random.default_rng(K)
    lens = np.concatenate([rng.integers(0, 140, 250), [0, 1, 7, 8, 9, 63, 64, 65, 140]])
    m = len(lens)
    ip = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    ix = np.concatenate([np.sort(rng.choice(d, n, replace=False)) for n in lens]).astype(np.int32)
    v = rng.standard_normal(len(ix)).astype(np.float32)
    with D.DSFacto(1, d, K, 1, D.LOGISTIC, 0.0, 0.0, 0.1, 1) as g:
        g.set_params(0.25, (0.1 * rng.standard_normal(d)).astype(np.float32), (0.1 * rng.standard_normal((d, K))).astype(np.float32))
        f = g.predict(ip, ix, v)                  # 140 KB: copied to the device and scored by the recompute kernel
        for a, b in [(0, 20), (100, 101), (m - 9, m), (200, 230)]:
            part = g.predict(ip[a:b + 1] - ip[a], ix[ip[a]:ip[b]], v[ip[a]:ip[b]])
            assert np.array_equal(part, f[a:b])


@pytest.mark.parametrize("K", [4, 8, 16, 32, 64, 128, 256])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_infinite_factors_stay_in_the_rows_that_have_them(K, value):
    """Rows of very different lengths side by side, some of which have a column of infinite factors: the others' scores are
    finite and as they are without it."""
    rng = np.random.default_rng(K)
    d, m = 900, 3000
    lens = rng.choice([0, 1, 2, 3, 5, 8, 9, 17, 40], m)
    rows = [np.sort(rng.choice(d - 1, n, replace=False) + 1) for n in lens]
    hit = rng.random(m) < 0.2
    rows = [np.concatenate([[0], r]) if h else r for r, h in zip(rows, hit)]      # column 0 comes first
    lens = np.array([len(r) for r in rows])
    ip, ix = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64), np.concatenate(rows).astype(np.int32)
    v = rng.standard_normal(len(ix)).astype(np.float32)
    w, V = (0.1 * rng.standard_normal(d)).astype(np.float32), (0.1 * rng.standard_normal((d, K))).astype(np.float32)
    with D.DSFacto(1, d, K, 1, D.LOGISTIC, 0.0, 0.0, 0.1, 1) as g:
        assert len(ix) * 8 > 128 << 10                                            # by the recompute kernel
        g.set_params(0.25, w, V)
        want = g.predict(ip, ix, v)
        V[0] = value
        g.set_params(0.25, w, V)
        got = g.predict(ip, ix, v)
        assert np.isfinite(got[~hit]).all() and np.array_equal(got[~hit], want[~hit])
        few = slice(0, 40)
        part = g.predict(ip[:41], ix[:ip[40]], v[:ip[40]])
        assert np.array_equal(part[~hit[few]], want[few][~hit[few]])


# columns on both sides of the line between 8 and 16 lanes for wide rows (320 KB), and of the one between repeating the last
# entry of a row and not (192 KB, 256-byte rows only)
@pytest.mark.parametrize("K,d", [(4, 900), (8, 900), (16, 900), (32, 900), (64, 768), (64, 769), (128, 640), (128, 641), (256, 320), (256, 321)])
@pytest.mark.parametrize("value", [0.25, np.inf, np.nan])
def test_allocation_free_scoring_of_uneven_rows(K, d, value):
    """Rows of very different lengths side by side, against 64 bits; a column of infinite factors spoils the rows that have it
    and no other."""
    import torch

    rng = np.random.default_rng(K + d)
    m = 3000
    lens = rng.choice([0, 1, 2, 3, 5, 8, 9, 17, 40, 90], m)
    rows = [np.sort(rng.choice(d - 1, n, replace=False) + 1) for n in lens]
    hit = rng.random(m) < 0.2
    rows = [np.concatenate([[0], r]) if h else r for r, h in zip(rows, hit)]      # column 0 comes first
    lens = np.array([len(r) for r in rows])
    ip, ix = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64), np.concatenate(rows).astype(np.int32)
    v = rng.standard_normal(len(ix)).astype(np.float32) / np.sqrt(np.repeat(lens, lens)).astype(np.float32)
    y = np.where(rng.random(m) < 0.5, 1.0, -1.0).astype(np.float32)
    w, V = (0.1 * rng.standard_normal(d)).astype(np.float32), (0.1 * rng.standard_normal((d, K))).astype(np.float32)
    V[0] = value
    t = [torch.from_numpy(a).cuda() for a in (ip, ix, v, y, w, V)]
    scores, sums = torch.empty(m, device="cuda"), torch.empty(2, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert D.dsfacto_score_loss_noalloc(m, d, K, D.LOGISTIC, *[a.data_ptr() for a in t[:4]], 0.25, t[4].data_ptr(),
                                        t[5].data_ptr(), scores.data_ptr(), sums.data_ptr()) == D.OK
    got = scores.cpu().numpy()
    f = O.score(ip, ix, v, 0.25, w.astype(np.float64), np.where(np.isfinite(V), V, 0).astype(np.float64))
    sound = ~hit if value != 0.25 else np.ones(m, bool)
    # fp32 sums of up to 91 products whose squares add up to about one: error below 91 * 2^-24 in the worst order
    np.testing.assert_allclose(got[sound], f[sound], rtol=0, atol=2e-5 * (1 + np.abs(f).max()))
    if value == 0.25:
        assert float(sums[0]) == pytest.approx(np.logaddexp(0.0, -y * f).sum(), rel=1e-5)
    else:
        assert not np.isfinite(got[hit]).any()
