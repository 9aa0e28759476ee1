"""A wait of the factor that runs out gives KC_ETIMEOUT whichever round of a long
row it lies in.  The one row below the diagonal waits in rounds of 8 entries a
lane: 512 entries with teams of two warps, 2048 with teams of eight, 256 with a
warp alone, so the held column is in an early round, in a middle one and in the
last."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1706_02205_gb300 import kchol as kc  # noqa: E402

DEV = torch.device("cuda:0")


def T(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def last_row_full(N):
    """Every row holds its diagonal only, the last one every column."""
    rowptr = np.arange(N + 1, dtype=np.int64)
    rowptr[N] = 2 * N - 1
    col = np.concatenate([np.arange(N - 1), np.arange(N)]).astype(np.int32)
    return kc.schedule(T(rowptr), T(col))


@pytest.mark.parametrize("N", [700, 1500, 3000])
@pytest.mark.parametrize("warps", [0, 1, 2, 8])
@pytest.mark.parametrize("prec", [kc.FP32_FORM, kc.FP64])
@pytest.mark.parametrize("lanes", [0, 16])  # the ring form, the register form
def test_held_column_of_a_long_row_times_out(N, warps, prec, lanes):
    pat = last_row_full(N)
    # far apart: the entries are tiny and the last pivot stays positive
    xo = T(np.arange(N, dtype=np.float64)[:, None] * np.ones((1, 2)))
    kern = kc.Kernel(0.5, 0.2)
    for held in (5, N // 2, N - 2):
        with pytest.raises(kc.KcError) as ei:
            kc.factor(pat, xo, kern, prec, kc.make_opts(spin_limit_cycles=1_000_000, test_hold_column=held,
                                                        warps_per_cta=warps, lanes_per_row=lanes))
        assert ei.value.status == kc.KC_ETIMEOUT, held
    val, diag, zp = kc.factor(pat, xo, kern, prec, kc.make_opts(warps_per_cta=warps, lanes_per_row=lanes))
    assert zp == 0 and bool((diag[:-1] == 1.0).all())
    want = torch.exp(-(xo[-1] - xo[:-1]).norm(dim=1) / kern.ell)
    assert float((val[N - 1:-1].double() - want).abs().max()) <= (1e-15 if prec == kc.FP64 else 1e-6)
