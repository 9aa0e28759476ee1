"""The solves' values carry their own readiness (a buffer of all ones until a
value is set): every stride of the vectors, columns whose rows end at, before
and behind a chunk, and NaN right-hand sides, the all-ones NaN among them."""
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
KERN = kc.Kernel(0.5, 0.2)


def T(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def factored(N, rho, prec):
    o = oracle.pipeline(inputs.uniform(N, 2, seed=500 + N), rho, oracle.Kernel(0.5, 0.2))
    pat = kc.schedule(T(o["rowptr"]), T(o["col"]))
    val, diag, zp = kc.factor(pat, T(o["x_ord"]), KERN, prec)
    assert zp == 0
    return o, pat, val, diag, T(o["perm"])


# a dense pattern: column 0 has N - 1 rows below its diagonal (chunks of 128, groups of 32 chunks)
@pytest.mark.parametrize("N,rho", [(1, 1e9), (2, 1e9), (128, 1e9), (129, 1e9), (130, 1e9), (257, 1e9), (4200, 2.0)])
@pytest.mark.parametrize("nrhs", [1, 2, 3, 8, 16])
@pytest.mark.parametrize("prec", [kc.FP64, kc.FP32_FORM])
def test_strides_and_chunks(N, rho, nrhs, prec):
    o, pat, val, diag, perm = factored(N, rho, prec)
    b = inputs.rhs(N, nrhs, seed=9)
    x = kc.solve(pat, prec, val, diag, KERN, perm, T(b))
    # the same solve in FP64 on the host with the GPU's factor
    v = val.double().cpu().numpy()
    dg = diag.cpu().numpy()
    z = np.stack([oracle.solve_upper(o["rowptr"], o["col"], v, dg,
                                     oracle.solve_lower(o["rowptr"], o["col"], v, dg, b[r][o["perm"]]))
                  for r in range(nrhs)])
    got = x.cpu().numpy()[:, o["perm"]]
    # sums of at most N terms in FP64, or to 2^-45 in pairs, with the condition of the small factor on top
    assert np.linalg.norm(got - z) <= 1e-10 * np.linalg.norm(z)
    assert torch.equal(kc.solve(pat, prec, val, diag, KERN, perm, T(b)), x)


@pytest.mark.parametrize("bits", [0x7FF8000000000000, 0xFFFFFFFFFFFFFFFF, 0xFFFFFFFF00000000])
@pytest.mark.parametrize("prec", [kc.FP64, kc.FP32_FORM])
@pytest.mark.parametrize("nrhs", [1, 4, 16])
def test_nan_right_hand_sides_end(bits, prec, nrhs):
    N = 3000
    o, pat, val, diag, perm = factored(N, 3.0, prec)
    b = inputs.rhs(N, nrhs, seed=10)
    clean = kc.solve(pat, prec, val, diag, KERN, perm, T(b))
    bad = b.copy()
    bad[nrhs - 1, int(o["perm"][N // 2])] = np.array([bits], np.uint64).view(np.float64)[0]
    x = kc.solve(pat, prec, val, diag, KERN, perm, T(bad))
    assert torch.isnan(x[nrhs - 1]).any()
    # the point itself, and the first of the order, which every row holds
    assert torch.isnan(x[nrhs - 1, int(o["perm"][N // 2])]) and torch.isnan(x[nrhs - 1, int(o["perm"][0])])
    assert torch.equal(x[:nrhs - 1], clean[:nrhs - 1])
