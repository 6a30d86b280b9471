"""The block-resident READY engine at the edges of its forms: rows around 8,
16, 32 and 64 ids (groups of 8, 16 and 32 lanes, one and two elements per
lane), fewer examples than groups, one example, empty rows, several epochs
(more of them in flight than examples in one), every feature in every example (each example
waits for the one before), margins and labels that take the general
derivative.  Bit for bit the oracle's SGD."""
import numpy as np
import pytest

import oracle
import synthdata
from oracle import history

torch = pytest.importorskip("torch")
pdb = pytest.importorskip("paper_1508_00703_gb300")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pdb.load()


def _equal(p):
    X = pdb.Csr.from_problem(p)
    y = torch.from_numpy(p.y).cuda()
    c = pdb.pdb_build_conflicts(X)
    s = pdb.pdb_schedule_build(c, pdb.PDB_SCHED_READY)
    w = torch.zeros(p.n_cols, dtype=torch.float32, device="cuda")
    pdb.pdb_sgd_epoch(X, y, c, s, w, p.loss, p.eta, p.epochs)
    pdb.check_status(c)
    assert np.array_equal(w.cpu().numpy().view(np.uint32), oracle.sgd(p).view(np.uint32))


@pytest.mark.parametrize("loss", ["logistic", "squared", "hinge"])
@pytest.mark.parametrize("k", [1, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64])
def test_row_lengths(k, loss):
    for cols in (k + 1, 3000):
        _equal(synthdata.generate("tiny", n_rows=700, n_cols=cols, k=k, k_lo=0 if k % 2 else k, loss=loss, epochs=2,
                                  seed=k))


@pytest.mark.parametrize("n", [1, 2, 16, 31, 32, 33, 63, 64, 65, 95, 97])
def test_few_examples_many_epochs(n):
    for k in (4, 12, 40):
        _equal(synthdata.generate("tiny", n_rows=n, n_cols=90, k=k, epochs=9, seed=n))


@pytest.mark.parametrize("k", [5, 13, 30, 60])
def test_general_derivative(k):
    p = synthdata.generate("tiny", n_rows=900, n_cols=500, k=k, epochs=2, seed=2)
    rng = np.random.default_rng(k)
    wild = np.repeat(rng.random(p.n_rows) < 0.3, k)
    p.val = np.where(wild, p.val * np.float32(3000.0), p.val).astype(np.float32)
    p.y = np.where(rng.random(p.n_rows) < 0.1, p.y * np.float32(0.5), p.y).astype(np.float32)
    _equal(p)


def test_largest_feature_count():
    _equal(synthdata.generate("tiny", n_rows=4000, n_cols=28000, k=12, seed=8))


def _wild(k):
    """Margins and labels of which a part takes the general derivative."""
    p = synthdata.generate("tiny", n_rows=900, n_cols=500, k=k, epochs=2, seed=2)
    rng = np.random.default_rng(k)
    p.val = np.where(np.repeat(rng.random(p.n_rows) < 0.3, k), p.val * np.float32(3000.0), p.val).astype(np.float32)
    return p


@pytest.mark.parametrize("wild", [False, True])
@pytest.mark.parametrize("k", [5, 13, 30, 60])
def test_trace_stamps_the_reads_when_the_weights_arrived(k, wild):
    # two moments per example, as the interface says: between them lie the margin,
    # the combine and the derivative (more than 100 ns), so over many examples the
    # timer has to tick between the two of some, also of those taken by the
    # general derivative.  One time for both would hide a read made too early.
    p = _wild(k) if wild else synthdata.generate("tiny", n_rows=6000, n_cols=3000, k=k, epochs=2, seed=k)
    X = pdb.Csr.from_problem(p)
    y = torch.from_numpy(p.y).cuda()
    c = pdb.pdb_build_conflicts(X)
    s = pdb.pdb_schedule_build(c, pdb.PDB_SCHED_READY)
    w = torch.zeros(p.n_cols, dtype=torch.float32, device="cuda")
    trace = torch.zeros(2 * p.epochs * p.n_rows, dtype=torch.int64, device="cuda")
    pdb.pdb_sgd_epoch(X, y, c, s, w, p.loss, p.eta, p.epochs, opts=dict(trace=trace))
    pdb.check_status(c)
    assert np.array_equal(w.cpu().numpy().view(np.uint32), oracle.sgd(p).view(np.uint32))
    tr = trace.cpu().numpy().reshape(-1, 2)
    assert np.all(tr > 0)
    v = history.trace_order_violations(p.row_ptr, p.col, p.epochs, tr)
    assert v["self"] == 0 and v["rc"] == 0, v
    assert np.mean(tr[:, 0] < tr[:, 1]) > 0.02
