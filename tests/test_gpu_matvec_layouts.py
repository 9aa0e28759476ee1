"""L z, L^T v and L L^T v at every split of the vectors over the lanes: rows
and columns of 0 to 33 entries, around a warp's block of 32, and columns past
the chunk of 1024, against NumPy with the GPU's own factor."""
import numpy as np
import pytest

import oracle
from paper_1706_02205_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1706_02205_gb300 import kchol as kc  # noqa: E402

DEV = torch.device("cuda:0")


def T(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


@pytest.mark.parametrize("N", [1, 2, 32, 33, 34, 65, 1025, 1026, 1100])  # dense pattern: row j holds j earlier columns
@pytest.mark.parametrize("nrhs", [1, 2, 3, 4, 7, 8, 9, 16])
@pytest.mark.parametrize("prec", [kc.FP64, kc.FP32_FORM])
def test_products(N, nrhs, prec):
    o = oracle.pipeline(inputs.uniform(N, 2, seed=700 + N), 1e9, oracle.Kernel(0.5, 0.2))
    pat = kc.schedule(T(o["rowptr"]), T(o["col"]))
    val, diag, _ = kc.factor(pat, T(o["x_ord"]), kc.Kernel(0.5, 0.2), prec)
    L = np.zeros((N, N))
    rows = np.repeat(np.arange(N), np.diff(o["rowptr"]))
    L[rows, o["col"]] = val.double().cpu().numpy()
    L[np.arange(N), np.arange(N)] = diag.cpu().numpy()
    perm = T(o["perm"])
    z = inputs.rhs(N, nrhs, seed=11)
    zp = z[:, o["perm"]]
    for fn, want in ((kc.l_matvec, zp @ L.T), (kc.lt_matvec, zp @ L), (kc.llt_matvec, zp @ L @ L.T)):
        got = fn(pat, prec, val, diag, perm, T(z)).cpu().numpy()[:, o["perm"]]
        # sums of at most 1100 products in FP64, in another order
        assert np.abs(got - want).max() <= 1e-12 * max(1.0, np.abs(want).max())
