"""Rows whose keys do not go into their two-choice table at the first attempt, and
rows that go into none at all: sets of keys chosen with the kernel's own hashes so
that some of them share fewer slots than they are, under the first multiplier pair
or under every one.  One warp a table and teams of 2, 4 and 8, held to a dense Cholesky
and to the same bits from every form."""
import numpy as np
import pytest
from scipy.sparse import coo_matrix
from scipy.sparse.csgraph import connected_components

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1706_02205_gb300 import kchol as kc  # noqa: E402

DEV = torch.device("cuda:0")
N, LAST = 1 << 20, 24  # the last LAST rows hold the keys and one another; the others their diagonal
TRIES = 4


def T(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def slots(keys, attempt, hbits):
    """The two slots of every key, as csrc/factor.cu's HashPair has them."""
    m1 = (2654435761 + 2 * 0x3C6EF372 * attempt) & 0xFFFFFFFF
    m2 = (2246822519 + 2 * 0x1B873593 * attempt) & 0xFFFFFFFF
    k = keys.astype(np.uint64)
    return [(((k * np.uint64(m)) & np.uint64(0xFFFFFFFF)) >> np.uint64(32 - hbits)).astype(np.int64) for m in (m1, m2)]


def crowded(keys, attempt, hbits):
    """The keys as edges between their two slots: for every component its slots and its keys, and each key's component."""
    a, b = slots(keys, attempt, hbits)
    n, lab = connected_components(coo_matrix((np.ones(len(keys)), (a, b)), shape=(1 << hbits,) * 2), directed=False)
    return np.bincount(lab, minlength=n), np.bincount(lab[a], minlength=n), lab[a]


def no_place(attempt, hbits):
    """Keys of a component with more keys than slots: no arrangement holds them."""
    rng = np.random.default_rng(10 * hbits + attempt)
    best = None
    for _ in range(400):
        keys = rng.choice(N - LAST, (1 << hbits) * 40 // 64, replace=False)
        have, want, of = crowded(keys, attempt, hbits)
        for c in np.flatnonzero(want > have):
            if best is None or want[c] < len(best):
                best = keys[of == c]
    return best


def keys_of(hbits, nr, attempts):
    """nr columns that cannot be placed under the first `attempts` multiplier pairs."""
    keys = np.unique(np.concatenate([no_place(t, hbits) for t in range(attempts)]))
    rng = np.random.default_rng(hbits)
    rest = rng.permutation(np.setdiff1d(rng.integers(0, N - LAST, 4 * nr), keys))
    return np.sort(np.concatenate([keys, rest[:nr - len(keys)]]))


@pytest.mark.parametrize("attempts", [1, TRIES])
@pytest.mark.parametrize("hbits", [7, 9, 10, 11, 12])
@pytest.mark.parametrize("prec", [kc.FP32_FORM, kc.FP64])
def test_keys_without_a_place(hbits, attempts, prec):
    longest = (1 << hbits) * 29 // 64  # of a table of 2^hbits slots; the last row has LAST - 1 entries more
    keys = keys_of(hbits, longest - (LAST - 1), attempts)
    for t in range(attempts):
        have, want, _ = crowded(keys, t, hbits)
        assert len(keys) == longest - (LAST - 1) and (want > have).any()
    m, n0 = len(keys), N - LAST
    rng = np.random.default_rng(100 + hbits)
    B = rng.uniform(-0.01, 0.01, (LAST, m))
    S = np.tril(rng.uniform(-0.01, 0.01, (LAST, LAST)), -1) + np.eye(LAST)
    rows = [np.concatenate([keys, n0 + np.arange(q + 1)]) for q in range(LAST)]
    rowptr = np.concatenate([np.arange(n0), n0 + np.cumsum([0] + [len(r) for r in rows])]).astype(np.int64)
    col = np.concatenate([np.arange(n0)] + rows).astype(np.int32)
    aval = np.concatenate([np.ones(n0)] + [np.concatenate([B[q], S[q, :q + 1]]) for q in range(LAST)])
    pat = kc.schedule(T(rowptr), T(col))
    ref = None
    for opts in ({}, dict(warps_per_cta=1), dict(warps_per_cta=2), dict(lanes_per_row=16), dict(rows_per_task=4)):
        val, diag, zp = kc.factor_given(pat, T(aval), prec, kc.make_opts(**opts))
        assert zp == 0
        if ref is None:
            ref = (val, diag)
            tail = val[n0:].cpu().numpy().astype(np.float64)
            want = np.linalg.cholesky(S + np.tril(S, -1).T - B @ B.T)  # the columns before the last have pivots 1
            got = np.zeros((LAST, LAST))
            at = 0
            # rounding: entries below 0.01 stored in the form's precision, sums compensated or in FP64
            tol = 1e-14 if prec == kc.FP64 else 1e-7
            for q in range(LAST):
                assert np.max(np.abs(tail[at:at + m] - B[q])) <= tol
                got[q, :q + 1] = tail[at + m:at + m + q + 1]
                at += m + q + 1
            # the last rows among themselves: at most LAST steps, each of m + LAST products of such entries
            assert np.max(np.abs(got - want)) <= LAST * (1e-14 if prec == kc.FP64 else 1e-7)
        elif opts != dict(lanes_per_row=16):  # another number of lanes sums in another order
            assert torch.equal(val, ref[0]) and torch.equal(diag, ref[1]), opts
