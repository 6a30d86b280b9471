"""CHAIN at every register width and at the edges of its pipeline: rows one
id short of, at and past each multiple of 32, data shorter than a step of 8
examples, ragged and empty rows, and margins or labels that take the general
derivative instead of the short one (a step that holds one is run again).
The result is the oracle's bit for bit."""
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


def _chain_equals_oracle(p):
    X = pdb.Csr.from_problem(p)
    y = torch.from_numpy(p.y).cuda()
    c = pdb.pdb_build_conflicts(X)
    s = pdb.pdb_schedule_build(c, pdb.PDB_SCHED_CHAIN)
    w = torch.zeros(p.n_cols, dtype=torch.float32, device="cuda")
    pdb.pdb_sgd_epoch(X, y, c, s, w, p.loss, p.eta, p.epochs)
    pdb.check_status(c)
    assert np.array_equal(w.cpu().numpy().view(np.uint32), oracle.sgd(p).view(np.uint32))


@pytest.mark.parametrize("loss", ["logistic", "squared", "hinge"])
@pytest.mark.parametrize("k", [1, 31, 32, 33, 64, 65, 96, 97, 128, 129, 160, 161, 192, 193, 224, 225, 255, 256])
def test_row_widths(k, loss):
    p = synthdata.generate("tiny", n_rows=203, n_cols=max(k + 5, 300), k=k, k_lo=0 if k % 2 else k, ids="zipf",
                           zipf_s=1.2, loss=loss, epochs=2, seed=k)
    _chain_equals_oracle(p)


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 15, 16, 17, 39, 40, 41, 48, 49])
def test_short_data(n):
    for k, cols in ((3, 4), (40, 60)):
        _chain_equals_oracle(synthdata.generate("tiny", n_rows=n, n_cols=cols, k=k, epochs=3, seed=n))


@pytest.mark.parametrize("k", [4, 40, 200])
def test_general_derivative_inside_a_step(k):
    # rows whose margin leaves the short form's range, at every place of a step,
    # and labels other than +1 and -1
    p = synthdata.generate("tiny", n_rows=400, n_cols=300, k=k, ids="zipf", zipf_s=1.1, epochs=2, seed=3)
    rng = np.random.default_rng(k)
    wild = np.repeat(rng.random(p.n_rows) < 0.2, k)
    p.val = np.where(wild, p.val * np.float32(3000.0), p.val).astype(np.float32)
    p.y = np.where(rng.random(p.n_rows) < 0.1, p.y * np.float32(0.5), p.y).astype(np.float32)
    _chain_equals_oracle(p)
