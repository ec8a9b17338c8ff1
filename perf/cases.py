"""The work that users of this package have it do, as cases to be timed.

Every case goes through the public entry points of paper_2004_13940_b200.dsfacto, in the way a program that
uses the package calls them:

  train     a handle with its data set loaded: `epochs` epochs, the objective read after each, then the
            parameters copied out (a checkpoint)
  job       a new data set in host arrays: create, load, `epochs` epochs, parameters out, destroy
  predict   held-out rows in host arrays scored with a model that is in place (a request, or a bulk job)
  evaluate  held-out labelled rows in host arrays: mean loss and accuracy or RMSE
  score     rows, labels and parameters in device memory of the caller: the entry point that allocates nothing

The data sets are made on the GPU from the seed, with the structures of the package's own workloads: `uniform`
(tabular: columns equally likely), `zipf` (text: column frequencies fall as a power of the rank, values
log-normal and rows of unit length, or normal) and `fields` (click logs: one id per field, power-law ids inside
a field, all values 1).  Labels come from a planted linear model with noise."""
import math

import numpy as np
import torch

from paper_2004_13940_b200 import dsfacto as D

DEV = "cuda:0"
LAMBDA = 1e-3            # both regularisers, as in the package's workloads
CHUNK = 1 << 24          # entries generated at a time


def _case(name, kind, structure, n, d, lmin, lmax, K, loss, **more):
    c = dict(name=name, kind=kind, structure=structure, n=n, d=d, lmin=lmin, lmax=lmax, K=K, loss=loss, p=1, epochs=0,
             refresh_every=0, rows=0)
    c.update(more)
    return c


def listed():
    return [
        # a small regression table (housing, diabetes), an epoch of which is all launches and latency
        _case("train_table", "train", "uniform", 2_000, 100, 10, 10, 8, "squared", p=4, epochs=10),
        # tens of thousands of rows over a handful of columns (ijcnn1): few long columns
        _case("train_dense", "train", "uniform", 50_000, 22, 13, 13, 16, "logistic", p=16, epochs=20),
        # bag-of-words classification (realsim): ragged rows, many short columns
        _case("train_text", "train", "zipf", 72_000, 21_000, 26, 76, 32, "logistic", p=64, epochs=5),
        # the same kind of data with the auxiliaries recomputed four times per epoch (shorter staleness)
        _case("train_text_fresh", "train", "zipf", 71_993, 21_000, 26, 76, 32, "logistic", p=64, epochs=5, refresh_every=16),
        # click logs, the flagship: hashed categorical fields, more rows than caches hold auxiliaries for
        _case("train_clicks", "train", "fields", 10_000_000, 1_048_554, 39, 39, 16, "logistic", p=256, epochs=5),
        # wide factor rows on long text-like rows
        _case("train_wide", "train", "zipf", 400_000, 131_072, 100, 100, 128, "squared", p=48, epochs=4),
        # a data set that is new to the process, trained from scratch: ragged text with a K that is no power of two
        _case("job_text", "job", "zipf", 72_001, 21_000, 26, 76, 20, "logistic", p=32, epochs=5),
        # ... and a day of click logs
        _case("job_clicks", "job", "fields", 1_000_003, 1_048_554, 39, 39, 16, "logistic", p=64, epochs=3),
        # one scoring request against a click model
        _case("predict_request", "predict", "fields", 0, 1_048_554, 39, 39, 16, "logistic", rows=32),
        # scoring a whole file of documents
        _case("predict_bulk", "predict", "zipf", 0, 21_000, 26, 76, 32, "logistic", rows=300_000),
        # the held-out curve that is drawn beside the objective
        _case("evaluate_heldout", "evaluate", "fields", 0, 1_048_554, 39, 39, 16, "logistic", rows=100_000),
        # rows that another part of the program already keeps on the device
        _case("score_device", "score", "zipf", 0, 262_144, 20, 60, 64, "logistic", rows=500_000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["train"] * 8 + ["job"] * 4 + ["predict"] * 4 + ["evaluate"] * 2 + ["score"] * 2)
    structure = rng.choice(["uniform", "zipf", "fields"])
    loss = rng.choice(["squared", "logistic"])
    K = _log_int(rng, 4, 128)
    if kind == "score":
        K = 2 ** rng.randint(2, 7)   # the widths that entry point takes
    if structure == "uniform":       # tables: up to a few hundred columns
        d = _log_int(rng, 20, 500)
        lmin = lmax = rng.randint(5, min(d, 60))
    elif structure == "zipf":
        d = _log_int(rng, 2_000, min(500_000, (1 << 24) // K))
        lmin = _log_int(rng, 10, 60)
        lmax = lmin + rng.randint(0, 60)
    else:
        lmin = lmax = rng.randint(8, 40)
        d = lmax * _log_int(rng, 50, min(30_000, (1 << 24) // (K * lmax)))
    most = max(2_000, min(1 << 24, 600_000_000 // K) // lmax)   # rows that keep a drawn case below the largest listed one
    if kind in ("predict", "evaluate", "score"):
        fewest = 1 if kind == "predict" else 1_000
        return _case("", kind, structure, 0, d, lmin, lmax, K, loss, rows=_log_int(rng, fewest, min(most, 500_000)))
    n = _log_int(rng, 1_000, min(most, 1_000_000))
    p = _log_int(rng, 4, 128)
    fresh = max(1, p // 4) if kind == "train" and rng.random() < 0.2 else 0
    return _case("", kind, structure, n, d, lmin, lmax, K, loss, p=p, epochs=rng.randint(1, 8), refresh_every=fresh)


# ---- data ----
def _exponent(case):
    """Of the power law that the column frequencies (of a field, or of the whole) follow."""
    return 1.2 if case["structure"] == "fields" else 1.1 if case["K"] < 64 else 1.05


def _column_sampler(case, gen):
    """-> f(rows): column ids [rows, lmax], drawn with the case's column frequencies (repeats possible but for fields)."""
    d, L = case["d"], case["lmax"]
    if case["structure"] == "uniform":
        # distinct columns of a row: the first L of a random order
        return lambda rows: torch.rand((rows, d), generator=gen, device=DEV).topk(L, dim=1).indices
    size = d // L if case["structure"] == "fields" else d
    cdf = torch.arange(1, size + 1, dtype=torch.float64, device=DEV).pow(-_exponent(case)).cumsum(0)
    cdf = cdf / cdf[-1]
    ranks = lambda rows: torch.searchsorted(cdf, torch.rand((rows, L), generator=gen, device=DEV, dtype=torch.float64)).clamp_(max=size - 1)
    if case["structure"] == "zipf":
        ids = torch.randperm(size, generator=gen, device=DEV)
        return lambda rows: ids[ranks(rows)]
    ids = torch.stack([torch.randperm(size, generator=gen, device=DEV) + f * size for f in range(L)]).reshape(-1)
    base = torch.arange(L, device=DEV) * size
    return lambda rows: ids[ranks(rows) + base]


def _rows(case, n, gen):
    """n rows as CSR tensors on the device: indptr int64, indices int32 (rising inside a row), values and labels fp32."""
    d, L = case["d"], case["lmax"]
    columns = _column_sampler(case, gen)
    planted = torch.randn(d, generator=gen, device=DEV)
    wide = d if case["structure"] == "uniform" else L
    step = max(1, CHUNK // max(wide, 1))
    lens, idx, val, score = [], [], [], []
    for at in range(0, n, step):
        m = min(step, n - at)
        ids = columns(m)
        if case["structure"] != "fields":
            if case["lmin"] < L:
                length = torch.randint(case["lmin"], L + 1, (m, 1), generator=gen, device=DEV)
                ids = torch.where(torch.arange(L, device=DEV) < length, ids, d)
            ids = ids.sort(dim=1).values
            keep = ids < d
            keep[:, 1:] &= ids[:, 1:] != ids[:, :-1]
        else:
            keep = None
        if case["structure"] == "fields":
            x = torch.ones((m, L), device=DEV)
        elif case["structure"] == "zipf" and case["K"] < 64:
            x = torch.randn((m, L), generator=gen, device=DEV).exp_() * keep
            x /= x.square().sum(1, keepdim=True).sqrt()
        else:
            x = torch.randn((m, L), generator=gen, device=DEV) * keep
        score.append((x * planted[ids.clamp(max=d - 1)]).sum(1))
        lens.append(torch.full((m,), L, device=DEV) if keep is None else keep.sum(1))
        idx.append((ids.reshape(-1) if keep is None else ids[keep]).to(torch.int32))
        val.append(x.reshape(-1) if keep is None else x[keep])
        del ids, keep, x
    indptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    indptr[1:] = torch.cat(lens).cumsum(0)
    score = torch.cat(score)
    if n > 1:
        score = score / score.std().clamp(min=1e-6)
    if case["loss"] == "squared":
        y = score + 0.1 * torch.randn(n, generator=gen, device=DEV)
    else:   # about a quarter positives on click logs, half elsewhere
        shift = -1.5 if case["structure"] == "fields" else 0.0
        y = torch.where(torch.rand(n, generator=gen, device=DEV) < torch.sigmoid(2.0 * score + shift), 1.0, -1.0)
    return indptr, torch.cat(idx), torch.cat(val), y.float()


def _loss(case):
    return D.SQUARED if case["loss"] == "squared" else D.LOGISTIC


def _eta(case):
    return 0.02 if case["loss"] == "squared" else 1.0


def _handle(case, n, p):
    return D.DSFacto(n, case["d"], case["K"], p, _loss(case), LAMBDA, LAMBDA, _eta(case), 2004)


def _model(case, gen):
    """Parameters of the size training leaves behind."""
    w = 0.2 * torch.randn(case["d"], generator=gen, device=DEV)
    V = 0.05 * torch.randn((case["d"], case["K"]), generator=gen, device=DEV)
    return 0.1, w, V


def prepare(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    kind = case["kind"]
    data = _rows(case, case["n"] or case["rows"], gen)
    if kind == "score":   # all of it stays on the device
        w0, w, V = _model(case, gen)
        m = case["rows"]
        return dict(case=case, data=data, w0=w0, w=w, V=V, scores=torch.empty(m, device=DEV),
                    sums=torch.empty(2, dtype=torch.float64, device=DEV))
    data = tuple(t.cpu().numpy() for t in data)
    if kind == "job":
        return dict(case=case, data=data)
    if kind == "train":
        fm = _handle(case, case["n"], case["p"])
        if case["refresh_every"]:
            fm.set_refresh_every(case["refresh_every"])
        fm.load_csr(*data)
        return dict(case=case, fm=fm)
    w0, w, V = _model(case, gen)
    fm = _handle(case, 1, 1)
    fm.set_params(w0, w.cpu().numpy(), V.cpu().numpy())
    return dict(case=case, fm=fm, data=data)


# ---- one pass ----
def _train(fm, epochs):
    objective = [fm.epoch() for _ in range(epochs)]
    w0, w, V = fm.get_params()
    return dict(objective=objective, w0=w0, w=w, V=V)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "train":
        return _train(state["fm"], case["epochs"])
    if kind == "job":
        with _handle(case, case["n"], case["p"]) as fm:
            fm.load_csr(*state["data"])
            return _train(fm, case["epochs"])
    if kind == "predict":
        return state["fm"].predict(*state["data"][:3])
    if kind == "evaluate":
        return state["fm"].evaluate(*state["data"])
    indptr, idx, val, y = state["data"]
    rc = D.dsfacto_score_loss_noalloc(case["rows"], case["d"], case["K"], _loss(case), indptr.data_ptr(), idx.data_ptr(),
                                      val.data_ptr(), y.data_ptr(), state["w0"], state["w"].data_ptr(), state["V"].data_ptr(),
                                      state["scores"].data_ptr(), state["sums"].data_ptr(),
                                      torch.cuda.current_stream().cuda_stream)
    if rc != D.OK:
        raise RuntimeError("dsfacto_score_loss_noalloc: status %d" % rc)
    return state["scores"], state["sums"]


# ---- what a pass cannot do without ----
def work(case):
    n, K, d = case["n"] or case["rows"], case["K"], case["d"]
    length = (case["lmin"] + case["lmax"]) / 2.0
    if case["structure"] == "zipf":   # columns a row drew twice count once
        share = np.arange(1, d + 1, dtype=np.float64) ** -_exponent(case)
        length = float(-np.expm1(length * np.log1p(-share / share.sum())).sum())
    nnz = n * length
    rows = 8.0 * nnz + 8.0 * (n + 1)                           # CSR: index and value of every entry, row pointers
    touched = min(float(d), nnz)                               # columns of which parameters can be needed at all
    params = 4.0 * touched * (K + 1)
    score_flops = nnz * (2.0 * K + 6.0) + n * (2.0 * K + 20.0)
    if case["kind"] in ("predict", "evaluate", "score"):
        out = {"predict": 4.0 * n, "evaluate": 4.0 * n + 16.0, "score": 8.0 * n + 16.0}[case["kind"]]
        return {"bytes": rows + params + out, "flops": score_flops}
    # an epoch: the updates read every entry, the frozen auxiliaries and multipliers, and rewrite the parameters; the
    # recompute pass that follows needs all of the new parameters, so it reads every entry and writes the auxiliaries
    passes = 1 if not case["refresh_every"] else -(-case["p"] // case["refresh_every"])
    update = 8.0 * nnz + passes * (4.0 * n * (K + 1) + 2.0 * params)
    recompute = rows + params + 4.0 * n * (K + 2)
    epoch = update + passes * recompute
    flops = nnz * (2.0 * K + 12.0) + passes * score_flops
    total, ops = case["epochs"] * epoch, case["epochs"] * flops
    total += 4.0 * d * (K + 1)                                 # the parameters copied out
    if case["kind"] == "job":                                  # the data set in, the first auxiliaries
        total += 2.0 * rows + recompute
        ops += score_flops
    return {"bytes": total, "flops": ops}


def tolerance(case):
    # fp32 sums over up to a few hundred (scores) or a few hundred thousand (columns) products in another order;
    # a class decided the other way round moves an accuracy by one row
    if case["kind"] == "evaluate":
        return {"rel": max(2e-5, 2.0 / case["rows"]) if case["loss"] == "logistic" else 2e-5}
    return {"rel": 2e-5}
