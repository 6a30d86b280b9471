"""The dense CHAIN engine (every example holds every feature) at the edges of
its tiles: one feature, one short of, at and past 32, 128 and multiples, the
largest it takes (1024) and one past it (the resident-weight engine); data
shorter than its pipeline, several epochs, every loss, no value array, margins
outside the short derivative, rows whose start is not 16-byte aligned.  The
result is the oracle's bit for bit.  Data that only looks dense (unordered
ids) must take another engine and give the same."""
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


def _equal(p):
    X = pdb.Csr.from_problem(p)
    y = torch.from_numpy(p.y).cuda()
    c = pdb.pdb_build_conflicts(X)
    s = pdb.pdb_schedule_build(c, pdb.PDB_SCHED_CHAIN)
    w = torch.zeros(p.n_cols, dtype=torch.float32, device="cuda")
    pdb.pdb_sgd_epoch(X, y, c, s, w, p.loss, p.eta, p.epochs)
    pdb.check_status(c)
    got, ref = w.cpu().numpy(), oracle.sgd(p)
    nan = np.isnan(ref)                     # a NaN's payload is not specified; everything else is
    assert np.array_equal(np.isnan(got), nan)
    assert np.array_equal(got.view(np.uint32)[~nan], ref.view(np.uint32)[~nan])


def _dense(n, f, loss="squared", epochs=1, vals=True, eta=1e-3, seed=0, scale=1.0):
    rng = np.random.default_rng(1000 * f + n + seed)
    val = (scale * rng.standard_normal(n * f)).astype(np.float32) if vals else None
    y = rng.standard_normal(n) if loss == "squared" else np.where(rng.random(n) < 0.5, -1.0, 1.0)
    return synthdata.from_arrays(np.arange(n + 1) * f, np.tile(np.arange(f), n), val, y, n_cols=f, loss=loss, eta=eta,
                                 epochs=epochs)


@pytest.mark.parametrize("loss", ["squared", "logistic", "hinge"])
@pytest.mark.parametrize("f", [1, 31, 32, 33, 127, 128, 129, 255, 257, 384, 511, 513, 640, 767, 895, 960, 961, 1023, 1024,
                               1025])
def test_widths(f, loss):
    _equal(_dense(75, f, loss, epochs=2))


@pytest.mark.parametrize("n,epochs", [(1, 1), (1, 5), (2, 4), (7, 1), (8, 1), (9, 3), (16, 2), (31, 1), (33, 2)])
def test_short_data(n, epochs):
    for f in (5, 130):
        _equal(_dense(n, f, "squared", epochs))


def test_no_values_and_general_derivative():
    _equal(_dense(40, 70, "logistic", 2, vals=False))
    _equal(_dense(200, 40, "logistic", 2, scale=200.0))


def test_divergence_to_infinity_and_nan():
    # the weights overflow after a few examples: runs that end before, at and after
    for n in range(4, 24):
        _equal(_dense(n, 37, "squared", 1, eta=50.0, scale=30.0, seed=7 - n))


def test_unordered_ids_take_another_engine():
    p = _dense(60, 50, "squared", 2)
    q = np.concatenate([np.random.default_rng(t).permutation(50) for t in range(60)])
    _equal(synthdata.from_arrays(p.row_ptr, q, p.val, p.y, n_cols=50, loss="squared", eta=1e-3, epochs=2))
