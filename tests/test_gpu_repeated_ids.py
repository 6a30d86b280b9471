"""The repeated-id check (PDB_EDUP) on rows whose ids do not ascend: a repeat
anywhere in a row, next to each other or at the row's two ends, in the longest
row or a shorter one, is reported; the same ids in neighbouring rows are not."""
import numpy as np
import pytest

import synthdata

torch = pytest.importorskip("torch")
pdb = pytest.importorskip("paper_1508_00703_gb300")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pdb.load()


def _status(lens, col, n_cols):
    row_ptr = np.r_[0, np.cumsum(lens)]
    p = synthdata.from_arrays(row_ptr, col, None, np.ones(len(lens)), n_cols=n_cols)
    X = pdb.Csr.from_problem(p)
    return pdb.pdb_status(pdb.pdb_build_conflicts(X))


@pytest.mark.parametrize("longest", [2, 3, 33, 200])
@pytest.mark.parametrize("row", ["longest", "shorter"])
def test_repeat_in_a_row(longest, row):
    rng = np.random.default_rng(longest)
    lens = np.where(np.arange(60) == 29, longest, np.maximum(2, longest - 1))
    rows = [rng.permutation(400)[:k] for k in lens]
    assert _status(lens, np.concatenate(rows), 400) == pdb.PDB_OK
    t = 29 if row == "longest" else 30
    for a, b in {(0, lens[t] - 1), (0, 1), (lens[t] - 2, lens[t] - 1)}:
        bad = [r.copy() for r in rows]
        bad[t][b] = bad[t][a]
        assert _status(lens, np.concatenate(bad), 400) == pdb.PDB_EDUP


@pytest.mark.parametrize("lens", ["ragged", "empty ends", "one long"])
def test_rows_found_from_any_position(lens):
    # rows far from where rows of one length would put them: the repeat sits in each row in turn
    rng = np.random.default_rng(9)
    n = 120
    k = {"ragged": rng.integers(0, 40, n), "empty ends": np.where((np.arange(n) > 40) & (np.arange(n) < 60), 30, 0),
         "one long": np.where(np.arange(n) == 100, 300, 2)}[lens]
    rows = [rng.permutation(500)[:m] for m in k]
    assert _status(k, np.concatenate(rows), 500) == pdb.PDB_OK
    for t in np.flatnonzero(k >= 2):
        bad = [r.copy() for r in rows]
        a, b = np.sort(rng.choice(k[t], 2, replace=False))
        bad[t][b] = bad[t][a]
        assert _status(k, np.concatenate(bad), 500) == pdb.PDB_EDUP, t


def test_same_ids_in_neighbouring_rows():
    lens = np.array([3, 1, 2, 0, 3, 1])
    assert _status(lens, np.array([5, 2, 7, 7, 5, 2, 7, 5, 2, 2]), 8) == pdb.PDB_OK
