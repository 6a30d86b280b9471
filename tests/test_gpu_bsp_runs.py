"""BSP's run sums at the edges of their forms: runs of one to seventeen terms
(the longest a thread sums, the shortest a block does), around the stages a
block adds (768 terms) and their multiples, long and short runs of one feature
set in one batch, batches of one row and of all rows, batches without a
nonzero, rows around a warp's load (32, 256 ids).  Bit for bit the oracle's
BSP, and so is the split form on the same data."""
import numpy as np
import pytest

import oracle
import synthdata

torch = pytest.importorskip("torch")
pdb = pytest.importorskip("paper_1508_00703_gb300")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pdb.load()


def _equal(p, batch, epochs=2, opts=None):
    p.epochs = epochs
    X = pdb.Csr.from_problem(p)
    y = torch.from_numpy(p.y).cuda()
    c = pdb.pdb_build_conflicts(X)
    ref = oracle.bsp(p, batch).view(np.uint32)
    w = torch.zeros(p.n_cols, dtype=torch.float32, device="cuda")
    pdb.pdb_bsp_epoch(X, y, c, w, p.loss, p.eta, batch, epochs, opts=opts)
    pdb.check_status(c)
    assert np.array_equal(w.cpu().numpy().view(np.uint32), ref)
    w.zero_()
    pdb.bsp_epoch_data_parallel(X, y, c, w, p.loss, p.eta, batch, epochs)
    pdb.check_status(c)
    assert np.array_equal(w.cpu().numpy().view(np.uint32), ref)


def _head(n, k=6, cols=400, seed=0):
    """Feature 0 in every row (one run of the batch's length), k - 1 others at random."""
    rng = np.random.default_rng(seed + n)
    col = np.stack([np.sort(np.r_[0, 1 + rng.permutation(cols - 1)[:k - 1]]) for _ in range(n)]).astype(np.int32)
    return synthdata.from_arrays(np.arange(n + 1) * k, col.ravel(), rng.standard_normal(n * k).astype(np.float32),
                                 np.where(rng.random(n) < 0.5, -1.0, 1.0), n_cols=cols, eta=0.01)


@pytest.mark.parametrize("n", [1, 2, 3, 6, 7, 15, 16, 17, 18, 32, 33, 191, 192, 193, 767, 768, 769, 1535, 1536, 1537, 2400])
def test_run_lengths(n):
    _equal(_head(n), n)


@pytest.mark.parametrize("batch", [1, 2, 16, 17, 100, 768, 769, 5000])
def test_batches(batch):
    _equal(_head(1700), batch, epochs=1)


@pytest.mark.parametrize("k", [1, 31, 32, 33, 255, 256, 257, 600])
def test_row_lengths(k):
    _equal(synthdata.generate("tiny", n_rows=150, n_cols=700, k=k, seed=k), 64)


def test_batches_without_nonzeros():
    n, empty = 90, np.arange(90) % 30 >= 10        # rows 10..29 of every 30 are empty
    lens = np.where(empty, 0, 3)
    rng = np.random.default_rng(5)
    col = np.concatenate([np.sort(rng.permutation(9)[:3]) for _ in range(int((~empty).sum()))])
    p = synthdata.from_arrays(np.r_[0, np.cumsum(lens)], col, rng.standard_normal(col.size), np.ones(n), n_cols=9)
    for batch in (1, 10, 30, 90):
        _equal(p, batch)


@pytest.mark.parametrize("batch", [8, 40, 130])
def test_neighbouring_weights_over_overlapping_batches(batch):
    # 70 features, so a few 128-byte lines of weights, each updated by many blocks
    # (runs summed by threads at 8 rows a batch, by blocks above) in every one of
    # hundreds of batches whose launches overlap: a line that a block kept in its
    # L1 from the batch before would give a stale weight
    p = synthdata.generate("tiny", n_rows=2600, n_cols=70, k=50, seed=batch)
    _equal(p, batch, epochs=3)


@pytest.mark.parametrize("per_sm", [1, 2, 1000])
def test_blocks_per_sm_keeps_the_result(per_sm):
    # grids smaller than the work: rows, long runs and short runs by strides
    _equal(_head(9000, cols=30000), 9000, opts=dict(blocks_per_sm=per_sm))
    _equal(synthdata.generate("tiny", n_rows=3000, n_cols=3000, k=60, seed=1), 1500, opts=dict(blocks_per_sm=per_sm))


def test_blocks_per_sm_limits_the_grid():
    # margins bound by the latency of random reads: one block of 8 warps per SM
    # takes several times as long as the 5 that fit (measured 0.77 against 0.17 ms)
    n, k, cols = 300_000, 32, 4_000_000
    g = torch.Generator(device="cuda").manual_seed(1)
    at = torch.arange(k, device="cuda") * (cols // k)
    col = (torch.randint(0, cols // k, (n, k), device="cuda", generator=g) + at).int().reshape(-1)
    X = pdb.Csr(torch.arange(n + 1, device="cuda") * k, col, torch.randn(n * k, device="cuda", generator=g), cols)
    y = torch.randn(n, device="cuda", generator=g)
    c = pdb.pdb_build_conflicts(X)
    w = torch.zeros(cols, device="cuda")

    def ms(opts, epochs):
        times = []
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            pdb.pdb_bsp_epoch(X, y, c, w, pdb.PDB_LOSS_SQUARED, 1e-6, n, epochs, opts=opts)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)

    def per_epoch(opts):
        return ms(opts, 11) - ms(opts, 1)
    assert per_epoch(dict(blocks_per_sm=1)) > 2 * per_epoch(None)
    pdb.check_status(c)


@pytest.mark.parametrize("turns", [1, 2, 3])
def test_many_short_runs(turns):
    # as many runs of one term as one turn of the apply grid's threads takes, and one
    # fewer and more; then two and three turns (a thread holds two runs at once)
    step = torch.cuda.get_device_properties(0).multi_processor_count * 8 * 128
    for n in (turns * step - 1, turns * step, turns * step + 1):
        rng = np.random.default_rng(n)
        row_ptr = np.minimum(np.arange((n + 63) // 64 + 1) * 64, n)
        p = synthdata.from_arrays(row_ptr, np.arange(n), rng.standard_normal(n).astype(np.float32),
                                  rng.standard_normal(len(row_ptr) - 1), n_cols=n + 3, loss="squared", eta=0.01)
        _equal(p, p.n_rows, epochs=1)


@pytest.mark.parametrize("batch", [600_000, 130_000])
def test_run_lists_of_large_batches(batch):
    # 12M pairs: the run lists' blocks take several turns, of one batch and of two
    _equal(synthdata.generate("low-conflict", n_rows=600_000, n_cols=3_000_000, k=20, k_lo=20), batch, epochs=1)
