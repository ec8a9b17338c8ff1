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
