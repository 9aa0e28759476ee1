"""The schedule's CSC view against a stable sort of the entries by column: sizes
around the sort's runs, tiles and digits, rows and columns of every length, and
rows too long for 32-bit items."""
import numpy as np
import pytest

from paper_1706_02205_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1706_02205_gb300 import kchol as kc  # noqa: E402

DEV = torch.device("cuda:0")


def lower(lengths, seed):
    """CSR of a lower-triangular pattern: row j holds min(lengths[j], j) earlier
    columns, spread with a random start, then its diagonal."""
    N = len(lengths)
    n = np.minimum(lengths, np.arange(N))
    rp = np.concatenate([[0], np.cumsum(n + 1)])
    row = np.repeat(np.arange(N), n + 1)
    p = np.arange(rp[-1]) - rp[row]
    step = np.maximum(1, row // np.maximum(1, n[row]))
    start = inputs.rng(seed).integers(0, 1 << 30, N)[row] % np.maximum(1, row - step * np.maximum(0, n[row] - 1))
    col = np.where(p == n[row], row, start + p * step)
    return rp.astype(np.int64), col.astype(np.int32)


def _mixed(N, seed):
    r = inputs.rng(seed)
    n = r.integers(0, 60, N)
    n[r.random(N) < 0.3] = 0  # diagonals alone: many row starts within a round
    n[r.random(N) < 0.01] = 1500
    return n


CASES = [(f"mixed{N}", lambda N=N: _mixed(N, N)) for N in (1, 2, 31, 255, 256, 257, 511, 513, 4097, 65536, 65537)]
CASES += [("diagonal", lambda: np.zeros(5000, int)), ("dense300", lambda: np.full(300, 300)),
          ("two_digits_more", lambda: np.where(np.arange(140000) % 9, 3, 40)),
          # 17-bit rows leave 15 bits for a place: 32768 fits, 32769 does not
          ("fits32", lambda: np.where(np.arange(70000) == 69999, 32767, 2)),
          ("wide", lambda: np.where(np.arange(70000) == 69990, 32768, 2))]


@pytest.mark.parametrize("name,make", CASES, ids=[c[0] for c in CASES])
def test_csc_view(name, make):
    rp, col = lower(make(), 5)
    N = len(rp) - 1
    assert col.min() >= 0 and np.all(col <= np.repeat(np.arange(N), np.diff(rp)))
    pat = kc.schedule(torch.from_numpy(rp).to(DEV), torch.from_numpy(col).to(DEV))
    slot = np.argsort(col, kind="stable")
    row = np.repeat(np.arange(N), np.diff(rp))
    assert np.array_equal(pat.slot.cpu().numpy(), slot)
    assert np.array_equal(pat.rowidx.cpu().numpy(), row[slot])
    assert np.array_equal(pat.colptr.cpu().numpy(), np.concatenate([[0], np.cumsum(np.bincount(col, minlength=N))]))
