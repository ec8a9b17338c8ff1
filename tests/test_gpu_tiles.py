"""The sweep over tiles where data sets of this size no longer take it by themselves: asked for with DSFACTO_ROW_MERGE (row
blocks per slot), row block by row block on tile lists that the device has built.  Chunks and the ring of entry blocks
that they are read through, runs over many chunks, plans cut into segments, and the bounds-checked build; the oracle and
the tolerances are those of the default update loop's tests."""
import numpy as np
import pytest

from oracle import dsfacto_oracle as O
from paper_2004_13940_b200 import dsfacto as D
from paper_2004_13940_b200 import workloads as W
from tests.test_gpu_parity import _hot_column_problem, check_params

pytestmark = pytest.mark.gpu


def _by_tiles(g, epoch):
    before = g.launch_count()
    out = epoch()
    assert (g.launch_count() - before) % 6 == 0     # w0, sweep, two kernels back to plain parameters, views, recompute
    return out


def _epochs(wl, count, every=0, load=None):
    o = O.Oracle(wl.n, wl.d, wl.K, wl.p, wl.loss, wl.lambda_w, wl.lambda_v, wl.eta, wl.init_seed)
    o.load_csr(wl.indptr, wl.indices, wl.values, wl.y)
    with D.DSFacto(wl.n, wl.d, wl.K, wl.p, wl.loss, wl.lambda_w, wl.lambda_v, wl.eta, wl.init_seed) as g:
        g.set_refresh_every(every)
        g.load_csr(wl.indptr, wl.indices, wl.values, wl.y)
        for _ in range(count):
            before = (o.w0, o.w.copy(), o.V.copy())
            want = o.epoch_segmented(every) if every else o.epoch()
            assert _by_tiles(g, g.epoch) == pytest.approx(want, rel=1e-4)
            check_params(o, g, before)


# chunks of part of a pass, of one block, of a few and of more blocks than the ring has slots, a last block of a few entries
@pytest.mark.parametrize("chunk,block", [(16, 0), (100, 32), (512, 0), (1000, 64), (2048, 256), (4096, 0)])
@pytest.mark.parametrize("name", ["C3", "C4s", "C5s"])
def test_any_chunk_length_and_ring(monkeypatch, name, chunk, block):
    monkeypatch.setenv("DSFACTO_ROW_MERGE", "2")
    monkeypatch.setenv("DSFACTO_CHUNK", str(chunk))
    if block:
        monkeypatch.setenv("DSFACTO_BLOCK", str(block))
    _epochs(W.make(name), 2)


@pytest.mark.parametrize("merge", ["1", "4"])
@pytest.mark.parametrize("K,p,loss", [(16, 3, 1), (8, 8, 0), (128, 5, 0), (40, 4, 1), (200, 4, 0)])
def test_runs_over_many_chunks(monkeypatch, K, p, loss, merge):
    monkeypatch.setenv("DSFACTO_ROW_MERGE", merge)
    n, d = 9000, 12
    indptr, indices, values, y = _hot_column_problem(n, d, 3)
    if loss:
        y = np.where(y > 0, 1.0, -1.0).astype(np.float32)
    o = O.Oracle(n, d, K, p, loss, 1e-3, 1e-3, 0.5, 77)
    o.load_csr(indptr, indices, values, y)
    with D.DSFacto(n, d, K, p, loss, 1e-3, 1e-3, 0.5, 77) as g:
        g.load_csr(indptr, indices, values, y)
        for _ in range(3):
            before = (o.w0, o.w.copy(), o.V.copy())
            assert _by_tiles(g, g.epoch) == pytest.approx(o.epoch(), rel=1e-4)
            check_params(o, g, before)


@pytest.mark.parametrize("name,every", [("C1", 1), ("C1", 3), ("C2", 5), ("C3", 16), ("C4s", 8), ("C5s", 3)])
def test_plans_cut_into_segments(monkeypatch, name, every):
    monkeypatch.setenv("DSFACTO_ROW_MERGE", "1")
    _epochs(W.make(name), 2, every)


@pytest.mark.parametrize("merge", ["1", "16"])
@pytest.mark.parametrize("name", ["C1", "C2", "C3", "C5s"])
def test_bounds_checked_build(monkeypatch, name, merge):
    # every row, column, chunk and run index that the sweep forms is checked; a bad one would fail the epoch
    monkeypatch.setenv("DSFACTO_ROW_MERGE", merge)
    with D.use_debug_library():
        _epochs(W.make(name), 2)
