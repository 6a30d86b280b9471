"""The grid-wide READY engine where its loop and versions can go wrong: rows
around 64, 128 and 256 ids (its register widths and the two-pass path), a row
alone, more epochs in flight than the data has examples (versions must not
repeat), every ticket size and grid, and the allocation-free form.  Bit for bit
the oracle's SGD."""
import numpy as np
import pytest

import oracle
import synthdata

torch = pytest.importorskip("torch")
pdb = pytest.importorskip("paper_1508_00703_gb300")

pytestmark = pytest.mark.gpu

COLS = 40_000            # more than one block's shared memory holds records for


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pdb.load()


def _equal(p, opts=None):
    X = pdb.Csr.from_problem(p)
    y = torch.from_numpy(p.y).cuda()
    c = pdb.pdb_build_conflicts(X)
    s = pdb.pdb_schedule_build(c, pdb.PDB_SCHED_READY)
    ref = oracle.sgd(p).view(np.uint32)
    w = torch.zeros(p.n_cols, dtype=torch.float32, device="cuda")
    pdb.pdb_sgd_epoch(X, y, c, s, w, p.loss, p.eta, p.epochs, opts=opts)
    pdb.check_status(c)
    assert np.array_equal(w.cpu().numpy().view(np.uint32), ref)
    w.zero_()
    assert pdb.pdb_sgd_epoch_ready_noalloc(X, y, pdb.pdb_schedule_ready(s)["gate"], w, p.loss, p.eta,
                                           p.epochs) == pdb.PDB_OK
    assert np.array_equal(w.cpu().numpy().view(np.uint32), ref)


@pytest.mark.parametrize("k", [1, 31, 33, 64, 65, 127, 128, 129, 255, 256, 257, 300])
def test_row_lengths(k):
    for lo in (k, 0):
        _equal(synthdata.generate("tiny", n_rows=600, n_cols=COLS, k=k, k_lo=lo, ids="zipf", zipf_s=1.1, epochs=2, seed=k))


@pytest.mark.parametrize("n", [1, 2, 5, 40, 300])
def test_many_epochs_of_few_examples(n):
    _equal(synthdata.generate("tiny", n_rows=n, n_cols=COLS, k=12, epochs=40, seed=n))


@pytest.mark.parametrize("chunk", [0, 1, 2, 5])
@pytest.mark.parametrize("blocks", [0, 1, 3])
def test_tickets_and_grids(chunk, blocks):
    _equal(synthdata.generate("tiny", n_rows=3000, n_cols=COLS, k=20, k_lo=3, epochs=2, seed=4),
           dict(ticket_chunk=chunk, blocks_per_sm=blocks))


@pytest.mark.parametrize("k", [511, 512, 513, 768, 769, 1030])
def test_long_rows(k):
    # rows of several times the ids a warp takes at once (256), with shorter ones among them
    for lo in (k, 0):
        _equal(synthdata.generate("tiny", n_rows=200, n_cols=COLS, k=k, k_lo=lo, ids="zipf", zipf_s=1.0, epochs=2, seed=k))
