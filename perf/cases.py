"""The calls that a user of this library makes, at the sizes at which they make them.

A case is one training run, one more epoch of a run that goes on, one conflict build, or one run
of the two comparison methods (BSP batches, admissible delay), always through the binding's public
calls.  The sizes are those of the repository's own workloads (tiny, zipf-1m, ctr, low-conflict,
deep-chain, dense-lr), scaled where the strictly serial engines would take seconds.

  kind    train    conflicts, schedule (AUTO), all epochs from w = 0, status: a run from scratch
          epoch    one more epoch on handles that the program keeps
          build    conflicts and all of their arrays
          bsp      BSP batches from w = 0, on kept conflicts
          delayed  admissible delay from w = 0, on a kept READY schedule
  rows, cols       examples and features; each row holds k_lo..k_hi distinct ids (uniform length)
  ids              uniform; zipf (exponent s, over a random permutation of the ids); dense (every feature)
  in_order         ids ascend within a row (else as they come out of a hash: any order)
"""
import math

import numpy as np
import torch

import paper_1508_00703_gb300 as pdb

LOSS = {"logistic": pdb.PDB_LOSS_LOGISTIC, "squared": pdb.PDB_LOSS_SQUARED, "hinge": pdb.PDB_LOSS_HINGE}


def _case(name=None, **kw):
    c = dict(kind="train", ids="uniform", s=0.0, rows=1, cols=1, k_lo=1, k_hi=1, in_order=True, vals="normal",
             labels="sign", loss="logistic", eta=0.01, epochs=1, batch=0, delay=0)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the next epoch over a set of a thousand short examples: a call whose latency is what counts
        _case("epoch-small", kind="epoch", rows=1000, cols=600, k_lo=4, k_hi=16),
        # a small set trained from scratch (the tiny workload)
        _case("train-tiny", rows=20_000, cols=10_000, k_lo=10, k_hi=10),
        # a middling set with ragged rows: conflicts are common, no chain dominates
        _case("train-mid", rows=60_000, cols=300_000, k_lo=10, k_hi=60, vals="uniform", labels="linear",
              loss="squared", eta=0.005),
        # word-like ids with a hot head, short rows (the zipf-1m workload, a fifth of its rows)
        _case("train-zipf", ids="zipf", s=1.0, rows=200_000, cols=1_000_000, k_lo=20, k_hi=20),
        # click logs: binary features (no value array), one chain as long as the data (ctr, fewer rows)
        _case("train-clicks", ids="zipf", s=1.1, rows=100_000, cols=10_000_000, k_lo=50, k_hi=50, vals="ones",
              labels="bernoulli", eta=0.05),
        # long documents, a linear SVM (deep-chain, fewer rows, one epoch)
        _case("train-hinge", ids="zipf", s=1.3, rows=50_000, cols=50_000, k_lo=200, k_hi=200, loss="hinge"),
        # dense linear regression, exact SGD (dense-lr)
        _case("train-dense", ids="dense", rows=5000, cols=960, k_lo=960, k_hi=960, labels="linear", loss="squared",
              eta=1e-4, epochs=20),
        # the largest: 400 million nonzeros over 100 million features, few conflicts (low-conflict)
        _case("train-large", rows=4_000_000, cols=100_000_000, k_lo=100, k_hi=100, vals="uniform", labels="linear",
              loss="squared", eta=0.001, epochs=2),
        # hashed click logs, ids in hash order: the conflict structure itself, read back
        _case("build-hashed", kind="build", ids="zipf", s=1.1, rows=400_000, cols=10_000_000, k_lo=50, k_hi=50,
              in_order=False, vals="ones", labels="bernoulli"),
        # BSP mini-batches on the word-like ids
        _case("bsp-zipf", kind="bsp", ids="zipf", s=1.0, rows=200_000, cols=1_000_000, k_lo=20, k_hi=20, batch=4096,
              eta=2.0 / 4096),
        # full-batch gradient descent on the dense data (the paper's batch GD)
        _case("gd-dense", kind="bsp", ids="dense", rows=5000, cols=960, k_lo=960, k_hi=960, labels="linear",
              loss="squared", batch=5000, eta=5e-5, epochs=20),
        # admissible delay on the word-like ids
        _case("delayed-zipf", kind="delayed", ids="zipf", s=1.0, rows=200_000, cols=1_000_000, k_lo=20, k_hi=20,
              delay=1024, eta=0.1 / 1024),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _ragged(rng, lo, hi):
    """Row lengths: one length for all rows, or a range of them."""
    a = rng.randint(lo, hi)
    return (a, a) if rng.random() < 0.5 else (rng.randint(lo, a), a)


def _loss(rng):
    loss = rng.choice(["logistic", "squared", "hinge"])
    return dict(loss=loss, labels="linear" if loss == "squared" else "sign", eta=0.005)


def draw(rng):
    what = rng.choice(["small", "tiny", "mid", "zipf", "clicks", "hinge", "dense", "large", "build", "bsp", "gd",
                       "delayed"])
    if what in ("small", "tiny"):
        k_lo, k_hi = _ragged(rng, 2, 32)
        rows = _log(rng, 300, 3000) if what == "small" else _log(rng, 3000, 20_000)
        return _case(kind="epoch" if what == "small" else "train", rows=rows, cols=_log(rng, max(200, rows // 2), 20_000),
                     k_lo=k_lo, k_hi=k_hi, in_order=rng.random() < 0.7, **_loss(rng))
    if what == "mid":
        k_lo, k_hi = _ragged(rng, 8, 64)
        return _case(rows=_log(rng, 10_000, 60_000), cols=_log(rng, 100_000, 1_000_000), k_lo=k_lo, k_hi=k_hi,
                     vals=rng.choice(["uniform", "ones"]), in_order=rng.random() < 0.7, **_loss(rng))
    if what == "zipf":
        k_lo, k_hi = _ragged(rng, 8, 32)
        return _case(ids="zipf", s=rng.choice([1.0, 1.1]), rows=_log(rng, 10_000, 200_000), cols=_log(rng, 50_000, 1_000_000),
                     k_lo=k_lo, k_hi=k_hi, vals=rng.choice(["normal", "ones"]), **_loss(rng))
    if what == "clicks":
        k_lo, k_hi = _ragged(rng, 33, 64)
        return _case(ids="zipf", s=rng.choice([1.0, 1.1]), rows=_log(rng, 10_000, 100_000),
                     cols=_log(rng, 100_000, 10_000_000), k_lo=k_lo, k_hi=k_hi, vals="ones", labels="bernoulli",
                     eta=0.05)
    if what == "hinge":
        k_lo, k_hi = _ragged(rng, 65, 320)
        return _case(ids="zipf", s=rng.choice([1.0, 1.3]), rows=_log(rng, 3000, 30_000), cols=_log(rng, 10_000, 40_000),
                     k_lo=k_lo, k_hi=k_hi, in_order=rng.random() < 0.7, loss="hinge")
    if what in ("dense", "gd"):
        rows, cols = _log(rng, 500, 5000), rng.randint(50, 960)
        c = dict(ids="dense", rows=rows, cols=cols, k_lo=cols, k_hi=cols, epochs=rng.randint(1, 20))
        if what == "dense":
            return _case(labels="linear", loss="squared", eta=1e-4, **c)
        loss = rng.choice(["squared", "logistic"])
        batch = rng.choice([100, rows])
        return _case(kind="bsp", loss=loss, labels="linear" if loss == "squared" else "sign", batch=batch,
                     eta=0.25 / (math.sqrt(batch) + math.sqrt(cols)) ** 2, **c)
    if what == "large":
        rows = _log(rng, 200_000, 4_000_000)
        k_lo, k_hi = _ragged(rng, 20, 100)
        return _case(rows=rows, cols=_log(rng, 20_000_000, 100_000_000), k_lo=k_lo, k_hi=k_hi, vals="uniform",
                     labels="linear", loss="squared", eta=0.001, epochs=rng.randint(1, 2))
    if what == "build":
        k_lo, k_hi = _ragged(rng, 5, 50)
        return _case(kind="build", ids=rng.choice(["zipf", "uniform"]), s=1.1, rows=_log(rng, 5000, 400_000),
                     cols=_log(rng, 10_000, 10_000_000), k_lo=k_lo, k_hi=k_hi, in_order=rng.random() < 0.5,
                     vals="ones", labels="bernoulli")
    k_lo, k_hi = _ragged(rng, 8, 50)
    c = dict(ids="zipf", s=rng.choice([1.0, 1.1]), rows=_log(rng, 20_000, 200_000), cols=_log(rng, 50_000, 1_000_000),
             k_lo=k_lo, k_hi=k_hi)
    if what == "bsp":
        batch = _log(rng, 256, 8192)
        return _case(kind="bsp", batch=batch, eta=2.0 / batch, vals=rng.choice(["normal", "ones"]), **c)
    delay = _log(rng, 512, 4096)
    return _case(kind="delayed", delay=delay, eta=0.1 / delay, **c)


# ------------------------------------------------------------------ inputs
def _zipf_ids(n, lens, K, cum, perm, g):
    """(n, K) ids, row t's first lens[t] of them distinct and ascending, the rest >= cols: ranks by inverse CDF,
    repeats drawn again until there are none."""
    F = perm.numel()
    dev = cum.device
    slot = torch.arange(K, device=dev)

    def ranks(m):
        u = torch.rand(m, device=dev, dtype=torch.float64, generator=g) * cum[-1]
        return torch.searchsorted(cum, u).clamp_(max=F - 1)

    r = ranks(n * K).view(n, K)
    r = torch.where(slot < lens[:, None], r, F + slot)
    live = torch.arange(n, device=dev)
    while live.numel():
        a = r[live].sort(dim=1).values
        dup = torch.zeros_like(a, dtype=torch.bool)
        dup[:, 1:] = a[:, 1:] == a[:, :-1]
        a[dup] = ranks(int(dup.sum()))
        r[live] = a
        live = live[dup.any(dim=1)]
    ids = torch.where(r < F, perm[r.clamp(max=F - 1)].long(), r)
    return ids.sort(dim=1).values


def _uniform_ids(n, lens, K, F, g, dev):
    """The same for uniform ids: ordered draws from exponential spacings, made distinct by adding each one's index."""
    slot = torch.arange(K, device=dev)
    c = torch.empty(n, K + 1, device=dev, dtype=torch.float64).exponential_(generator=g).cumsum(dim=1)
    top = c.gather(1, lens[:, None])
    u = (c[:, :K] / top).clamp_(max=1.0 - 1e-12)
    span = (F - lens + 1)[:, None]
    ids = (u * span).long().clamp_(max=F) + slot
    return torch.where(slot < lens[:, None], ids, F + slot)


def _data(case, seed):
    dev = "cuda"
    g = torch.Generator(device=dev).manual_seed(int(seed))
    N, F, K = case["rows"], case["cols"], case["k_hi"]
    lens = torch.randint(case["k_lo"], K + 1, (N,), device=dev, generator=g)
    row_ptr = torch.zeros(N + 1, dtype=torch.int64, device=dev)
    torch.cumsum(lens, 0, out=row_ptr[1:])
    nnz = int(row_ptr[-1])
    wstar = torch.randn(F, device=dev, generator=g) * (0.1 if case["labels"] == "bernoulli" else 1.0)
    if case["ids"] == "zipf":
        cum = torch.arange(1, F + 1, device=dev, dtype=torch.float64).pow_(-case["s"]).cumsum(0)
        perm = torch.randperm(F, device=dev, generator=g).int()
    col = torch.empty(nnz, dtype=torch.int32, device=dev)
    val = None if case["vals"] == "ones" else torch.empty(nnz, device=dev)
    y = torch.empty(N, device=dev)
    step = max(1, 24_000_000 // K)
    for t0 in range(0, N, step):
        n = min(step, N - t0)
        ln = lens[t0:t0 + n]
        if case["ids"] == "dense":
            ids = torch.arange(F, device=dev).expand(n, K)
        elif case["ids"] == "zipf":
            ids = _zipf_ids(n, ln, K, cum, perm, g)
        else:
            ids = _uniform_ids(n, ln, K, F, g, dev)
        real = torch.arange(K, device=dev) < ln[:, None]
        if not case["in_order"]:
            key = torch.rand(n, K, device=dev, generator=g) + 2.0 * ~real
            ids = ids.gather(1, key.argsort(dim=1))
        x = None
        if val is not None:
            x = torch.empty(n, K, device=dev)
            x = x.normal_(generator=g) if case["vals"] == "normal" else x.uniform_(-1.0, 1.0, generator=g)
        at = wstar[ids.clamp(max=F - 1)]
        m = torch.where(real, at if x is None else at * x, 0.0).sum(dim=1)
        if case["labels"] == "sign":
            y[t0:t0 + n] = torch.where(m < 0, -1.0, 1.0)
        elif case["labels"] == "bernoulli":
            y[t0:t0 + n] = torch.where(torch.rand(n, device=dev, generator=g) < torch.sigmoid(m), 1.0, -1.0)
        else:
            y[t0:t0 + n] = m + 0.1 * torch.randn(n, device=dev, generator=g)
        p0 = int(row_ptr[t0])
        p1 = int(row_ptr[t0 + n])
        col[p0:p1] = ids[real].int()
        if val is not None:
            val[p0:p1] = x[real]
    return pdb.Csr(row_ptr, col, val, F), y


def prepare(case, seed):
    X, y = _data(case, seed)
    st = {"case": case, "X": X, "y": y}
    if case["kind"] in ("epoch", "bsp", "delayed"):
        st["c"] = pdb.pdb_build_conflicts(X)
        if case["kind"] != "bsp":
            st["s"] = pdb.pdb_schedule_build(
                st["c"], pdb.PDB_SCHED_AUTO if case["kind"] == "epoch" else pdb.PDB_SCHED_READY)
        pdb.check_status(st["c"])
    if case["kind"] == "epoch":
        st["w"] = torch.zeros(case["cols"], device="cuda")
    return st


# ------------------------------------------------------------------ one pass
def run(state):
    case, X, y = state["case"], state["X"], state["y"]
    loss, eta, epochs = LOSS[case["loss"]], case["eta"], case["epochs"]
    kind = case["kind"]
    if kind == "epoch":
        pdb.pdb_sgd_epoch(X, y, state["c"], state["s"], state["w"], loss, eta, epochs)
        return state["w"]
    if kind == "build":
        c = pdb.pdb_build_conflicts(X)
        a = pdb.pdb_conflicts_arrays(c)
        nnz = X.col.numel()
        out = {k: pdb.device_array(a[k], nnz, torch.int32) for k in ("csc_pos", "prev", "next", "rank")}
        out["feat_ptr"] = pdb.device_array(a["feat_ptr"], case["cols"] + 1, torch.int64)
        pdb.check_status(c)
        return out
    w = torch.zeros(case["cols"], device="cuda")
    if kind == "train":
        c = pdb.pdb_build_conflicts(X)
        s = pdb.pdb_schedule_build(c, pdb.PDB_SCHED_AUTO)
        pdb.pdb_sgd_epoch(X, y, c, s, w, loss, eta, epochs)
        pdb.check_status(c)
    elif kind == "bsp":
        pdb.pdb_bsp_epoch(X, y, state["c"], w, loss, eta, case["batch"], epochs)
    else:
        pdb.pdb_ssp_epoch(X, y, state["c"], state["s"], w, loss, eta, epochs, case["delay"])
    return w


def work(case):
    """Per pass over the data: row bounds and labels, ids and values once, and the weights once in and once out (of
    a feature set larger than the nonzeros, at most one weight in and out per nonzero).  A build reads the rows and
    writes its five arrays; the other kinds do two operations per nonzero for the margin and two for the step."""
    N, F = case["rows"], case["cols"]
    nnz = N * (case["k_lo"] + case["k_hi"]) / 2
    if case["kind"] == "build":
        return {"bytes": 8 * (N + 1) + 4 * nnz + 16 * nnz + 8 * (F + 1), "flops": 0}
    per_nnz = 4 + (0 if case["vals"] == "ones" else 4)
    once = N * 12 + nnz * per_nnz + 8 * min(F, nnz)
    return {"bytes": case["epochs"] * once, "flops": 4 * nnz * case["epochs"]}


def tolerance(case):
    """Every call but the delayed one gives one result: the rounding and the order of each sum are part of the
    interface (a fixed 32-partial margin, one rounding per operation, updates in data order), so another correct
    implementation gives the same bits.  A delayed run depends on timing: over seven drawn cases the same run twice
    differed by up to 4.2e-4 (relative, 2-norm) and 0.013 (largest); about four times that is allowed."""
    return {"rel": 2e-3, "max": 0.06} if case["kind"] == "delayed" else "exact"


# ------------------------------------------------------------------ in 64 bits
def _grad(loss, m, y):
    if loss == "logistic":
        return -y / (1.0 + np.exp(np.minimum(y * m, 700.0)))
    if loss == "squared":
        return m - y
    return np.where(y * m < 1.0, -y, 0.0)


def exact(case, seed):
    """The same run in 64 bits: sequential SGD example by example, BSP batch by batch.  None for a delayed run (any
    of many results is right), a build (whole numbers), and a run of more than about 20 seconds here."""
    kind, N, F = case["kind"], case["rows"], case["cols"]
    if kind in ("build", "delayed"):
        return None
    if kind != "bsp" and N * case["epochs"] > 400_000:
        return None
    X, y = _data(case, seed)
    if kind == "bsp":
        return _exact_bsp(case, X, y)
    rp = X.row_ptr.tolist()
    col, yy = X.col.cpu().numpy(), y.double().cpu().numpy()
    val = None if X.val is None else X.val.double().cpu().numpy()
    w = np.zeros(F)
    eta, loss = float(np.float32(case["eta"])), case["loss"]
    one = np.ones(case["k_hi"])
    for _ in range(case["epochs"]):
        for t in range(N):
            b, e = rp[t], rp[t + 1]
            j = col[b:e]
            x = one[:e - b] if val is None else val[b:e]
            wj = w[j]
            w[j] = wj - (eta * _grad(loss, float(wj @ x), yy[t])) * x
    return torch.from_numpy(w)


def _exact_bsp(case, X, y):
    dev = y.device
    N, B = case["rows"], min(case["batch"], case["rows"])
    rp = X.row_ptr
    row = torch.repeat_interleave(torch.arange(N, device=dev), rp[1:] - rp[:-1])
    col = X.col.long()
    val = torch.ones(col.numel(), device=dev, dtype=torch.float64) if X.val is None else X.val.double()
    yy = y.double()
    w = torch.zeros(case["cols"], device=dev, dtype=torch.float64)
    eta = float(np.float32(case["eta"]))
    bounds = [(r, min(N, r + B)) for r in range(0, N, B)]
    at = rp[torch.tensor([b[0] for b in bounds] + [N], device=dev)].tolist()
    for _ in range(case["epochs"]):
        for (r0, r1), p0, p1 in zip(bounds, at[:-1], at[1:]):
            j, x, t = col[p0:p1], val[p0:p1], row[p0:p1] - r0
            m = torch.zeros(r1 - r0, device=dev, dtype=torch.float64).index_add_(0, t, w[j] * x)
            ys = yy[r0:r1]
            if case["loss"] == "logistic":
                g = -ys / (1.0 + torch.exp((ys * m).clamp(max=700.0)))
            elif case["loss"] == "squared":
                g = m - ys
            else:
                g = torch.where(ys * m < 1.0, -ys, torch.zeros_like(ys))
            w = w.index_add(0, j, -eta * g[t] * x)
    return w
