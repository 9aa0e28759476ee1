"""The block factor at prefixes around the sizes where its table of the prefix
grows, becomes denser for want of shared memory, or stops being sparse: on a full
pattern the factor is the Cholesky factor, so its residual is that of a complete
factorisation.

Bars: FP64, the backward error bound of Cholesky, (N + 1) u |L||L|^T <= (N + 1) u
Theta_ii, times 8 for the groups' order and stored reciprocals; FP32 form, the
compensated sums leave the rounding of the stored entries, a few 2^-24 Theta_ii."""
import numpy as np
import pytest

from paper_1706_02205_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1706_02205_gb300 import kchol as kc  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("prec", [kc.FP64, kc.FP32_FORM])
@pytest.mark.parametrize("N", [12, 13, 97, 385, 1537, 2400, 2700])
def test_full_pattern_residual(N, prec):
    x = torch.from_numpy(inputs.uniform(N, 3, seed=401)).to(DEV)
    n = torch.arange(N, device=DEV)
    rowptr = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), torch.cumsum(n + 1, 0)])
    row, col = torch.tril_indices(N, N, device=DEV)
    pat = kc.schedule(rowptr, col.to(torch.int32), x)
    kern = kc.Kernel(0.5, 0.3, 1.0, 1.0)
    val, diag, zero = kc.factor_blocked(pat, x, kern, prec)
    assert zero == 0
    L = torch.zeros(N, N, dtype=torch.float64, device=DEV)
    L[row, col] = val.double()
    A = torch.exp(-(x[:, None] - x[None]).pow(2).sum(-1).sqrt() / 0.3)
    A[n, n] = 2.0
    bar = 8 * (N + 1) * 2.0**-53 * 2.0 if prec == kc.FP64 else 2.0**-24 * 2.0 * 8
    assert float((L @ L.T - A).abs().max()) <= bar
    assert np.allclose(diag.cpu().numpy(), L.diagonal().cpu().numpy(), rtol=2.0**-23, atol=0)


@pytest.mark.parametrize("seed", [411, 412, 413])
def test_compensated_sums_do_not_depend_on_their_split(seed):
    """FP32 form, 8 and 32 lanes a row: the sums of at most 64 products agree to
    about 64 u^2, so the stored entries round alike but for one in 2^16; sums
    without the compensation would differ in a large part of them."""
    N = 64
    x = torch.from_numpy(inputs.uniform(N, 3, seed=seed)).to(DEV)
    n = torch.arange(N, device=DEV)
    rowptr = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), torch.cumsum(n + 1, 0)])
    _, col = torch.tril_indices(N, N, device=DEV)
    pat = kc.schedule(rowptr, col.to(torch.int32), x)
    kern = kc.Kernel(0.5, 0.5, 1.0, 0.01)
    a, _, _ = kc.factor_blocked(pat, x, kern, kc.FP32_FORM)
    b, _, _ = kc.factor_blocked(pat, x, kern, kc.FP32_FORM, opts=kc.kc_opts(lanes_per_row=32))
    assert float((a != b).double().mean()) <= 0.01
