"""The update loop by column runs where its plan has edges: one and several bands of rows (DSFACTO_BANDS), cut inside
row blocks; units of 32 entries to a few hundred (DSFACTO_CHUNK), so that runs end at, before and behind the ends of
passes, units and CTAs; every lane layout of the factor rows; segments of the second schedule."""
import numpy as np
import pytest

from oracle import dsfacto_oracle as O
from paper_2004_13940_b200 import dsfacto as D
from paper_2004_13940_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bands", [1, 2, 7])
@pytest.mark.parametrize("chunk", [16, 64, 512])
@pytest.mark.parametrize("K,p,every", [(3, 5, 0), (8, 1, 0), (16, 3, 0), (16, 6, 4), (30, 4, 0), (64, 3, 0), (128, 2, 0), (200, 3, 2)])
def test_bands_units_and_widths(monkeypatch, bands, chunk, K, p, every):
    monkeypatch.setenv("DSFACTO_BANDS", str(bands))
    monkeypatch.setenv("DSFACTO_CHUNK", str(chunk))
    rng = np.random.default_rng(7 * K + p)
    n, d = 1201, 60
    # column j is present with probability falling from 1 to almost nothing: runs of one entry to runs over many CTAs
    mask = rng.random((n, d)) < np.linspace(1.0, 0.0, d) ** 4
    mask[::13] = False
    indptr = np.concatenate([[0], np.cumsum(mask.sum(1))]).astype(np.int64)
    indices = np.nonzero(mask)[1].astype(np.int32)
    values = rng.standard_normal(len(indices)).astype(np.float32)
    y = np.where(rng.random(n) < 0.5, 1.0, -1.0).astype(np.float32)
    o = O.Oracle(n, d, K, p, O.LOGISTIC, 1e-2, 1e-2, 0.7, 3)
    o.load_csr(indptr, indices, values, y)
    with D.DSFacto(n, d, K, p, D.LOGISTIC, 1e-2, 1e-2, 0.7, 3) as g:
        if every:
            g.set_refresh_every(every)
        g.load_csr(indptr, indices, values, y)
        tp, rows, cols, vals = g.get_tiles()
        assert np.array_equal(tp, o.tile_ptr) and np.array_equal(rows, o.rows) and np.array_equal(cols, o.cols)
        assert np.array_equal(vals, o.vals)
        for _ in range(2):
            bw, bV = o.w.copy(), o.V.copy()
            want, got = (o.epoch_segmented(every) if every else o.epoch()), g.epoch()
            assert got == pytest.approx(want, rel=1e-5)
            w0, w, V = g.get_params()
            assert w0 == pytest.approx(o.w0, abs=1e-6)
            for new, ref, old in ((w, o.w, bw), (V, o.V, bV)):
                assert np.abs(new.astype(np.float64) - ref).max() <= 1e-4 * np.abs(ref - old).max() + 1e-7
        A, G = g.get_aux()
        np.testing.assert_allclose(A, o.A, rtol=0, atol=2e-5 * (1 + np.abs(o.A).max()))
        np.testing.assert_allclose(G, o.G, rtol=0, atol=2e-5)


@pytest.mark.parametrize("K", [4, 8, 16, 30, 64, 128])
def test_long_runs_among_many_short_ones(monkeypatch, K):
    """More runs than a warp each is given to, and among them runs of 1 to 33 pieces (a CTA of the sweep has 128 entries
    here), so that a warp joins pieces for some of its runs: fewer pieces than lane groups, as many, more."""
    monkeypatch.setenv("DSFACTO_CHUNK", "32")
    rng = np.random.default_rng(K)
    n, short = 4200, 10000
    rows, cols = [], []
    for j, length in enumerate([127, 128, 129, 256, 257, 385, 512, 640, 1023, 1025, 2049, 4100, 4200]):
        rows.append(rng.choice(n, length, replace=False))
        cols.append(np.full(length, 700 * j + 3))
    d = short + 700 * 13
    taken = set(700 * j + 3 for j in range(13))
    others = np.array([j for j in rng.permutation(d) if j not in taken][:short])
    rows.append(rng.integers(0, n, short))
    cols.append(others)
    rows, cols = np.concatenate(rows), np.concatenate(cols)
    order = np.lexsort((cols, rows))
    indices = cols[order].astype(np.int32)
    indptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=n))]).astype(np.int64)
    values = rng.standard_normal(len(indices)).astype(np.float32)
    y = np.where(rng.random(n) < 0.5, 1.0, -1.0).astype(np.float32)
    o = O.Oracle(n, d, K, 3, O.LOGISTIC, 1e-2, 1e-2, 0.7, 3)
    o.load_csr(indptr, indices, values, y)
    with D.DSFacto(n, d, K, 3, D.LOGISTIC, 1e-2, 1e-2, 0.7, 3) as g:
        g.load_csr(indptr, indices, values, y)
        for _ in range(2):
            bw, bV = o.w.copy(), o.V.copy()
            assert g.epoch() == pytest.approx(o.epoch(), rel=1e-5)
            w0, w, V = g.get_params()
            assert w0 == pytest.approx(o.w0, abs=1e-6)
            for new, ref, old in ((w, o.w, bw), (V, o.V, bV)):
                assert np.abs(new.astype(np.float64) - ref).max() <= 1e-4 * np.abs(ref - old).max() + 1e-7


def _wide_rows(n, d, per_row, seed):
    rng = np.random.default_rng(seed)
    idx = rng.integers(0, d // per_row, (n, per_row), dtype=np.int32) + (np.arange(per_row, dtype=np.int32) * (d // per_row))
    indptr = np.arange(n + 1, dtype=np.int64) * per_row
    return indptr, idx.ravel(), rng.standard_normal(n * per_row, dtype=np.float32), rng.standard_normal(n, dtype=np.float32)


def _launches_per_epoch(g):
    g.epoch()
    before = g.launch_count()
    g.epoch()
    return g.launch_count() - before


_TILES = 6      # w0, sweep, two kernels back to plain parameters, views, recompute; by runs two per band and more


# a data set that just goes by tiles, and one step over each line of the rule
@pytest.mark.parametrize("K,n,d,per_row,p,tiles", [(256, 800_000, 60_000, 30, 48, True), (130, 1_200_000, 80_000, 27, 13, True),
                                                   (256, 800_000, 60_000, 30, 81, False), (256, 800_000, 60_000, 29, 12, False),
                                                   (256, 700_000, 60_000, 35, 12, False), (256, 800_000, 40_000, 30, 48, False),
                                                   (256, 800_000, 60_000, 30, 11, False), (64, 3_400_000, 1_000_000, 28, 48, False)])
def test_many_short_runs_of_wide_rows_go_by_tiles(K, n, d, per_row, p, tiles):
    indptr, idx, val, y = _wide_rows(n, d, per_row, K)
    with D.DSFacto(n, d, K, p, D.SQUARED, 1e-3, 1e-3, 20.0, 11) as g:
        g.load_csr(indptr, idx, val, y)
        first = _launches_per_epoch(g)
        assert first == _TILES if tiles else first >= 2 * 10
        if not tiles:
            return
        w0, w, V = g.get_params()
        objective = g.objective()
    o = O.Oracle(n, d, K, p, O.SQUARED, 1e-3, 1e-3, 20.0, 11)
    o.load_csr(indptr, idx, val, y)
    before = o.V.copy()
    o.epoch()
    assert objective == pytest.approx(o.epoch(), rel=1e-4)
    assert w0 == pytest.approx(o.w0, abs=1e-6)
    assert np.abs(w - o.w).max() <= 1e-4 * (1 + np.abs(o.w).max())
    assert np.abs(o.V - before).max() > 1e-5
    assert np.abs(V - o.V).max() <= 2e-3 * np.abs(o.V - before).max() + 4e-7     # (two epochs: twice the rounding of one)


@pytest.mark.parametrize("bands", ["2", "12", "40"])
def test_the_number_of_bands_does_not_choose_the_update_loop(monkeypatch, bands):
    n, d, K, p = 800_000, 60_000, 256, 48
    indptr, idx, val, y = _wide_rows(n, d, 30, 4)
    with D.DSFacto(n, d, K, p, D.SQUARED, 1e-3, 1e-3, 20.0, 11) as g:
        g.load_csr(indptr, idx, val, y)
        assert _launches_per_epoch(g) == _TILES
        monkeypatch.setenv("DSFACTO_BANDS", bands)
        g.load_csr(indptr, idx, val, y)
        assert _launches_per_epoch(g) == _TILES
