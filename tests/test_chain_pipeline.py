"""A model of the CHAIN engine's pipeline schedule, on the CPU.

One thread block runs the examples in data order, G per pipeline step, and
its warps work on different steps in the same iteration t of the step loop,
separated only by the __syncthreads that ends each iteration:

  P   (G warps, example g of a step each)  keeps its loads in registers from
                   one iteration to the next: row bounds of step t + RS, with
                   those of the iteration before the ids, link words, values
                   and label of step t + AS, with those the global weights
                   nobody pushes of step t + BS; writes step t + BS's values,
                   label and store addresses (ring of XS example slots) and
                   write-through ids (ring of WS), and the weights gathered
                   one iteration ago, for step t + BS - 1, to the weight slots
                   (ring of WS);
  C   (one warp)  runs the examples of step t in order, each reading its
                   weights, label, values and store addresses from its slots
                   and storing each new weight to its address: the slot of the
                   feature's next occurrence when that lies within D = G * DS
                   examples (a push), its own out slot (ring of OS) otherwise.
                   Values are read one example ahead, so the last example of a
                   step reads those of the next step's first.  When a margin
                   lies outside the fast derivative's range the whole step runs
                   again;
  W   (G / WPER warps)  writes step t - 1's out slots through to global w.

The model replays that schedule with the link words the engine builds from
the conflict chains and checks, on problems full of near repeats: every
example uses, for every feature, exactly the weight its previous occurrence
wrote (in the epoch, or the last one of the epoch before), also in steps that
run twice; every slot the compute warp reads holds the example it reads it for;
global w ends each epoch holding each feature's last writer; no two warps touch
one shared or global cell in the same iteration unless both only read it.  A
gathered weight's load may complete one iteration after its issue: its global
cell counts as read in both.

The rings and distances are read from the engine's source, so a change there is
checked here.  The same checks fail when a constant breaks one of the engine's
compile-time conditions (each ring one power of two shorter, a shorter and a
longer forwarding window, weights stored in the step that reads them), when a
repeated step is not run again whole, and when values are read a step instead of
an example ahead."""
import os
import re

import numpy as np
import pytest

import oracle
import synthdata

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1508_00703_gb300", "csrc", "chain.cu")


def _engine():
    """The constants of ChainCfg, the same for every row width."""
    body = re.search(r"struct ChainCfg \{(.*?)\};", open(SRC).read(), re.S).group(1)
    c = {}
    for decl in re.findall(r"static constexpr int ([^;]*);", body):
        for item in decl.split(","):
            name, expr = item.split("=")
            if "R" not in re.findall(r"\w+", expr):              # all but the longest row
                c[name.strip()] = eval(expr, {}, c)
    return {k: c[k] for k in ("G", "DS", "BS", "AS", "RS", "PS", "D", "XS", "WS", "OS", "WPER")}


ENGINE = _engine()


def test_constants_were_found():
    assert ENGINE["D"] == ENGINE["G"] * ENGINE["DS"] and ENGINE["AS"] == ENGINE["BS"] + 1 and ENGINE["RS"] == ENGINE["AS"] + 1


def _links(p, D):
    ch = oracle.chains(p)
    prev, nxt = ch["prev"], ch["next"]
    row_of = np.repeat(np.arange(p.n_rows), np.diff(p.row_ptr))
    recv = np.zeros(p.nnz, bool)
    push = {}
    for q in range(p.nnz):
        t = row_of[q]
        if prev[q] >= 0 and t - row_of[prev[q]] <= D:
            recv[q] = True
        if nxt[q] >= 0 and row_of[nxt[q]] - t <= D:
            push[q] = (int(row_of[nxt[q]] - t), int(nxt[q] - p.row_ptr[row_of[nxt[q]]]))
    return recv, push


class _Iteration:
    """Cells each warp reads and writes during one iteration of the step loop."""

    def __init__(self):
        self.reads, self.writes = {}, {}

    def r(self, warp, cell):
        self.reads.setdefault(cell, set()).add(warp)

    def w(self, warp, cell):
        self.writes.setdefault(cell, set()).add(warp)

    def check(self, t):
        for cell, ws in self.writes.items():
            others = (ws | self.reads.get(cell, set()))
            assert len(others) == 1, ("two warps touch one cell in one iteration", t, cell, sorted(others))


def _simulate(p, epochs, G, DS, BS, AS, RS, PS, D, XS, WS, OS, WPER, twice=(), redo="whole", ahead=True):
    """twice: examples whose step runs again; redo: "whole" step, or (planted) that example alone; ahead:
    values read one example ahead (planted: a whole step ahead)."""
    N, rp = p.n_rows, p.row_ptr
    K = max(1, int(np.max(np.diff(rp))) if N else 1)      # slots are written to their full width
    recv, push = _links(p, D)
    steps = (N + G - 1) // G
    mem = {}                              # shared memory: cell -> what it holds
    w = {}                                # global: feature -> (epoch, example) of its writer, None = w0
    last_writer = {}
    for ep in range(epochs):
        expect = dict(last_writer)        # the weight the next occurrence of each feature must read
        bounds, loaded, gathered = {}, {}, {}     # registers of warp P g
        late = []                         # global cells of loads that may complete in the next iteration
        vals = None                       # C's registers: the values of the next example
        for t in range(-PS, steps + 1):
            it = _Iteration()
            effects = []                  # stores: visible to the others after the iteration's barrier
            for warp, cell in late:
                it.r(warp, cell)
            late = []

            def store(warp, cell, v):
                it.w(warp, cell)
                effects.append((cell, v))

            for g in range(G):
                warp = f"P{g}"
                # the weights gathered one iteration ago, to step t + BS - 1's slots
                for r, i, v in gathered.pop(g, []):
                    store(warp, ("wp", r % WS, i), v)
                # step t + BS, from the ids and link words loaded one iteration ago
                r = (t + BS) * G + g
                if 0 <= r < N:
                    assert loaded[g] == r, ("registers of another example", r, loaded[g])
                    b, k = int(rp[r]), int(rp[r + 1] - rp[r])
                    new = []
                    for i in range(K):
                        q, inside = b + i, i < k
                        if inside and not recv[q]:
                            j = int(p.col[q])
                            it.r(warp, ("w", j))
                            late.append((warp, ("w", j)))
                            new.append((r, i, w.get(j)))
                        elif not inside:
                            new.append((r, i, "zero"))
                        if inside and q in push:
                            dr, e = push[q]
                            to = ("wp", (r + dr) % WS, e)
                        else:
                            to = ("out", r % OS, i) if inside else None
                        store(warp, ("pa", r % XS, i), (r, to))
                        store(warp, ("wcol", r % WS, i), (r, int(p.col[q]) if inside and q not in push else -1))
                        store(warp, ("xa", r % XS, i), (r, i) if inside else (r, "-0"))
                    store(warp, ("y", r % XS), r)
                    gathered[g] = new
                r = (t + AS) * G + g
                if 0 <= r < N:
                    assert bounds[g] == r, ("row bounds of another example", r, bounds[g])
                    loaded[g] = r
                r = (t + RS) * G + g
                if 0 <= r < N:
                    bounds[g] = r
            for i in range(G // WPER):
                for r in range((t - 1) * G + i * WPER, (t - 1) * G + (i + 1) * WPER):
                    if not (t >= 1 and r < N):
                        continue
                    for e in range(K):
                        it.r(f"W{i}", ("wcol", r % WS, e))
                        it.r(f"W{i}", ("out", r % OS, e))
                        of, j = mem[("wcol", r % WS, e)]
                        assert of == r, ("write-through ids of another example", r, of)
                        if j >= 0:
                            store(f"W{i}", ("w", j), mem[("out", r % OS, e)])
            if 0 <= t < steps:
                local = {}                # C's own stores, visible to its later reads

                def read(cell):
                    it.r("C", cell)
                    return local.get(cell, mem.get(cell))

                def load_values(r):
                    return [read(("xa", r % XS, i)) for i in range(K)]

                def run(r, bad):
                    """One example; bad: in a first run of its step that gives wrong weights from here on."""
                    nonlocal vals
                    b, k = int(rp[r]), int(rp[r + 1] - rp[r])
                    got = [read(("wp", r % WS, i)) for i in range(K)]
                    x = vals
                    assert read(("y", r % XS)) == r
                    vals = load_values(r + (1 if ahead else G))
                    assert x == [(r, i) if i < k else (r, "-0") for i in range(K)], ("values of another example", r, x)
                    assert all(v == "zero" for v in got[k:]), ("padding reads a weight", r, got)
                    if not bad:
                        for i in range(k):
                            j = int(p.col[b + i])
                            assert got[i] == expect.get(j), ("wrong weight read", ep, r, j, got[i], expect.get(j))
                    for i in range(K):
                        of, to = read(("pa", r % XS, i))
                        assert of == r, ("store address of another example", r, of)
                        if to is not None:
                            it.w("C", to)
                            local[to] = ("bad", ep, r) if bad else (ep, r)
                    if not bad:
                        for i in range(k):
                            expect[int(p.col[b + i])] = (ep, r)

                r0, r1 = t * G, min(N, t * G + G)
                flagged = [r for r in range(r0, r1) if (ep, r) in twice]
                if t == 0:
                    vals = load_values(0)
                if not flagged:
                    for r in range(r0, r1):
                        run(r, False)
                else:
                    before = dict(expect)
                    for r in range(r0, r1):              # from the first flagged example on, wrong
                        run(r, r >= flagged[0])
                    expect = before
                    again = range(r0, r1) if redo == "whole" else flagged
                    vals = load_values(again[0])
                    for r in again:
                        run(r, False)
                effects.extend(local.items())
            it.check(t)
            for cell, v in effects:
                if cell[0] == "w":
                    w[cell[1]] = v
                else:
                    mem[cell] = v
        last_writer = expect
        for j, v in last_writer.items():                  # the drain leaves every feature's last writer in w
            assert w.get(j) == v, ("w after the epoch", ep, j, w.get(j), v)


def _problem(seed, rng):
    return synthdata.generate("tiny", seed=seed, n_rows=int(rng.integers(60, 160)), n_cols=int(rng.integers(3, 30)),
                              k=int(rng.integers(1, 6)), k_lo=0, ids="zipf" if seed % 2 else "uniform", zipf_s=1.2)


def _periods(n=150):
    """A feature for every distance from 28 to 72 between its occurrences (the window and the rings end in there)."""
    ds = range(28, 73)
    rows = [[d - 28 for d in ds if (t + d // 2) % d == 0] for t in range(n)]
    return synthdata.from_arrays(np.r_[0, np.cumsum([len(r) for r in rows])], np.concatenate(rows).astype(np.int32), None,
                                 np.ones(n), n_cols=len(ds))


def test_chain_pipeline_every_distance():
    p = _periods()
    _simulate(p, epochs=2, **ENGINE)
    _simulate(p, epochs=2, twice={(0, r) for r in range(0, p.n_rows, 5)}, **ENGINE)


@pytest.mark.parametrize("seed", range(10))
def test_chain_pipeline_schedule(seed):
    rng = np.random.default_rng(700 + seed)
    p = _problem(seed, rng)
    _simulate(p, epochs=2, **ENGINE)
    # and with steps that run again: a tenth of the examples outside the fast derivative's range
    twice = {(ep, r) for ep in range(2) for r in range(p.n_rows) if rng.random() < 0.1}
    _simulate(p, epochs=2, twice=twice, **ENGINE)


def test_chain_pipeline_one_feature_and_ragged():
    # every example holds feature 0: every weight is pushed; and a ragged
    # problem with empty examples and a short last step
    n = 37
    p = synthdata.from_arrays(np.arange(n + 1), np.zeros(n, np.int32), None, np.ones(n), n_cols=1)
    _simulate(p, epochs=3, **ENGINE)
    q = synthdata.generate("tiny", seed=5, n_rows=101, n_cols=7, k=4, k_lo=0)
    _simulate(q, epochs=2, twice={(1, 0), (1, 100), (0, 50)}, **ENGINE)


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 15, 16, 17, 40, 41, 63, 65])
def test_chain_pipeline_short_data(n):
    for k in (1, 3):
        p = synthdata.generate("tiny", seed=n, n_rows=n, n_cols=5, k=k, k_lo=k)
        _simulate(p, epochs=3, twice={(1, n - 1)}, **ENGINE)


def _fails(change, **plant):
    cfg = dict(ENGINE)
    cfg.update(change)
    failures = 0
    for seed in range(6):
        rng = np.random.default_rng(800 + seed)
        p = _problem(seed, rng) if seed else _periods()
        twice = {(0, r) for r in range(p.n_rows) if rng.random() < 0.1}
        try:
            _simulate(p, epochs=2, twice=twice, **plant, **cfg)
        except AssertionError:
            failures += 1
    return failures


def _at_distance(BS):
    return dict(BS=BS, AS=BS + 1, RS=BS + 2)


@pytest.mark.parametrize("change", [
    dict(XS=ENGINE["XS"] // 2),                       # XS >= (BS + 1) G
    dict(WS=ENGINE["WS"] // 2),                       # WS >= (DS + 1) G and (BS + 2) G
    dict(DS=ENGINE["WS"] // ENGINE["G"], D=ENGINE["WS"]),   # the same: a push to its own example's slot, read again
    dict(OS=ENGINE["OS"] // 2),                       # OS >= 2 G
    dict(D=(ENGINE["BS"] + 2) * ENGINE["G"] - 2),     # (D + 1) / G >= BS + 2
    dict(DS=2, D=2 * ENGINE["G"]),
    _at_distance(1),                                  # BS >= 2
    _at_distance(4),                                  # values live longer than XS; weights gathered too early
])
def test_chain_pipeline_model_rejects_broken_constants(change):
    assert _fails(change) > 0


@pytest.mark.parametrize("plant", [dict(redo="one"), dict(ahead=False)])
def test_chain_pipeline_model_rejects_planted_mistakes(plant):
    assert _fails({}, **plant) > 0


def test_element_layout():
    # rows of up to 64 ids: element i of each 32 at chain_at(i), so that a lane's four neighbouring words hold the
    # partial sums p, p + 8, p + 16, p + 24 of the margin and its own element is one of them
    at = [(i & ~31) | ((i & 7) << 2) | ((i >> 3) & 3) for i in range(64)]
    assert re.search(r"return QUAD<R> \? \(i & ~31\) \| \(\(i & 7\) << 2\) \| \(\(i >> 3\) & 3\) : i;", open(SRC).read())
    assert sorted(at) == list(range(64))
    where = {a: i for i, a in enumerate(at)}
    for lane in range(32):
        four = [where[(lane & 7) * 4 + e] for e in range(4)]
        assert four == [lane % 8 + 8 * e for e in range(4)]
        assert where[(lane & 7) * 4 + (lane >> 3)] == lane
