"""The conflict build where its passes change form: sizes around a sort tile
(4096 pairs), around the steps of the scan's chunk length, on both sides of the
switch from the scan inside its last kernel to the one with a kernel of its own
(128 chunks of 256 tiles), and around the sizes at which the gate words are brought to position
order by direct stores, by one radix pass over 2^15-slot blocks and by two over
2^14 (2^22, 2^24, 2^25 positions).  Checked against the definitions on the
device: csc_pos a stable sort of the ids, feat_ptr its bounds, prev, next and
rank its neighbours."""
import pytest

torch = pytest.importorskip("torch")
pdb = pytest.importorskip("paper_1508_00703_gb300")

pytestmark = pytest.mark.gpu

T = 4096


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pdb.load()


@pytest.mark.parametrize("n", [1, T - 1, T, T + 1, 16 * T, 16 * T + 1, 17 * T, 512 * T, 512 * T + 1, (1 << 22) - 1, 1 << 22,
                               (1 << 22) + 1, 2048 * T, 2048 * T + 3, 1 << 24, (1 << 24) + 1, 1 << 25, (1 << 25) + 5,
                               16384 * T + 1, 32768 * T, 32768 * T + 1])
@pytest.mark.parametrize("cols", [300, 5_000_000])
def test_build(n, cols):
    g = torch.Generator(device="cuda").manual_seed(n + cols)
    col = torch.randint(0, cols, (n,), device="cuda", generator=g, dtype=torch.int32)
    col[n // 3: n // 2] = cols // 2                         # one long run
    row_ptr = torch.arange(n + 1, device="cuda")            # one id per row
    X = pdb.Csr(row_ptr, col, None, cols)
    c = pdb.pdb_build_conflicts(X)
    a = pdb.pdb_conflicts_arrays(c)
    pdb.check_status(c)
    got = {k: pdb.device_array(a[k], n, torch.int32).long() for k in ("csc_pos", "prev", "next", "rank")}
    fp = pdb.device_array(a["feat_ptr"], cols + 1, torch.int64)
    pos = got["csc_pos"]
    key = col[pos].long()
    seen = torch.zeros(n, dtype=torch.bool, device="cuda")
    seen[pos] = True
    assert bool(seen.all())
    if n > 1:
        assert bool(((key[1:] > key[:-1]) | ((key[1:] == key[:-1]) & (pos[1:] > pos[:-1]))).all())
    assert torch.equal(fp, torch.searchsorted(key, torch.arange(cols + 1, device="cuda")))
    slot = torch.arange(n, device="cuda")
    assert torch.equal(got["rank"][pos], slot - fp[key])
    first, last = slot == fp[key], slot == fp[key + 1] - 1
    assert torch.equal(got["prev"][pos], torch.where(first, -1, pos.roll(1)))
    assert torch.equal(got["next"][pos], torch.where(last, -1, pos.roll(-1)))
