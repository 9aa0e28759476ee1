"""The factor's ring form at the edges of its row tables and of its copies:
rows of every length up to one below, at and one past what a table of 2^h
slots takes (teams of 1, 2, 4 and 8 warps, and rows without a table), held to
the oracle's factor at the fixed bars, and the same bits from the register form
(taken for arrays that do not start on a 16-byte boundary) and for every number
of rows per task."""
import numpy as np
import pytest

import oracle
from paper_1706_02205_gb300 import inputs
from tests import factor_parity as fp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1706_02205_gb300 import kchol as kc  # noqa: E402

DEV = torch.device("cuda:0")


def T(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def table_rows(h):
    return (1 << h) * 29 // 64


# every row holds all earlier columns, so row j has j entries: N - 1 is the longest
DENSE = [2, 5, 34] + [table_rows(h) + e for h in (9, 10, 11) for e in (0, 1, 2)] + [table_rows(12) + 2]


def dense(N):
    """Points in maximin order, all pairs in the pattern."""
    o = oracle.pipeline(inputs.uniform(N, 2, seed=1000 + N), 1e9, oracle.Kernel(0.5, 0.2))
    assert int(np.diff(o["rowptr"]).max()) == N
    return o


@pytest.mark.parametrize("N", DENSE)
@pytest.mark.parametrize("prec", [kc.FP32_FORM, kc.FP64])
def test_row_lengths_at_the_table_edges(N, prec):
    o = dense(N)
    pat = kc.schedule(T(o["rowptr"]), T(o["col"]))
    xo, kern = T(o["x_ord"]), kc.Kernel(0.5, 0.2)
    val, diag, zp = kc.factor(pat, xo, kern, prec)
    assert zp == 0
    err = np.max(np.abs(val.cpu().numpy().astype(np.float64) - o["val"]))
    assert err < fp.BAR[prec], err
    # the register form: values from an odd place of a larger buffer
    dt = torch.float64 if prec == kc.FP64 else torch.float32
    odd = torch.empty(pat.nnz + 1, dtype=dt, device=DEV)[1:]
    v2, d2, _ = kc.factor(pat, xo, kern, prec, val=odd)
    assert torch.equal(v2, val) and torch.equal(d2, diag)


@pytest.mark.parametrize("rho", [2.0, 4.0])
@pytest.mark.parametrize("d", [2, 3])
@pytest.mark.parametrize("prec", [kc.FP32_FORM, kc.FP64])
def test_rows_per_task_and_cta_sizes_same_bits(rho, d, prec):
    x = T(inputs.uniform(4001, d, seed=77 + d))
    perm, l, xo = kc.order_points(x)
    pat = kc.build_pattern(xo, l, rho)
    kern = kc.Kernel(0.5, 0.3)
    ref = kc.factor(pat, xo, kern, prec)
    for opts in (dict(rows_per_task=1), dict(rows_per_task=37), dict(rows_per_task=4096), dict(warps_per_cta=1),
                 dict(warps_per_cta=3), dict(warps_per_cta=4, rows_per_task=5), dict(ctas_per_sm=1),
                 dict(ctas_per_sm=-1), dict(adaptive_chunks=1)):
        got = kc.factor(pat, xo, kern, prec, kc.make_opts(**opts))
        assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1]) and got[2] == ref[2], opts
