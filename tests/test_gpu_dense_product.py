"""The refined solve's dense product by split entries: sizes around its tiles
(64 rows, 128 columns), every number of right-hand sides, dimension and
closed-form kernel, coordinates and vectors of very different scales, points
that coincide, checked by the true residual in FP64 on the host."""
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


def theta(x, k):
    r = np.sqrt(((x[:, None, :] - x[None, :, :]) ** 2).sum(-1))
    t = np.sqrt(2 * k.nu) * r / k.ell
    f = {0.5: 1.0, 1.5: 1.0 + t, 2.5: 1.0 + t + t * t / 3}[k.nu]
    return k.sigma2 * f * np.exp(-t) + k.nugget * np.eye(len(x))


def refined(x, kern, b, rho=4.0, prec=kc.FP64):
    r = kc.pipeline(T(x), rho, kern, prec)
    return kc.refine(r["pat"], r["x_ord"], kern, prec, r["val"], r["diag"], r["perm"], T(b), rtol=1e-11, maxit=400)


def check(x, kern, b, **kw):
    xs, it, rel, st = refined(x, kern, b, **kw)
    assert st == kc.KC_OK
    res = b - xs.cpu().numpy() @ theta(x, kern)
    for r in range(b.shape[0]):
        # CG stops at 1e-11; the host's own product in FP64 is about 1e-15 |Theta| |x| off
        floor = 1e-14 * np.linalg.norm(theta(x, kern), 2) * np.linalg.norm(xs[r].cpu().numpy())
        assert np.linalg.norm(res[r]) <= 3e-11 * np.linalg.norm(b[r]) + floor
        assert rel[r] <= 1e-10


@pytest.mark.parametrize("N", [1, 2, 16, 17, 63, 64, 65, 127, 128, 129, 1000])
@pytest.mark.parametrize("nrhs", [1, 8, 9, 16])
def test_sizes(N, nrhs):
    check(inputs.uniform(N, 2, seed=40 + N), kc.Kernel(0.5, 0.2), inputs.rhs(N, nrhs, seed=N))


@pytest.mark.parametrize("d", [1, 2, 3, 5])
@pytest.mark.parametrize("nu", [0.5, 1.5, 2.5])
def test_kernels_and_dimensions(nu, d):
    check(inputs.uniform(900, d, seed=60 + d), kc.Kernel(nu, 0.2, 2.5, 0.01), inputs.rhs(900, 3, seed=d))


@pytest.mark.parametrize("scale", [1e-150, 1e-20, 1e20, 1e150])
@pytest.mark.parametrize("nu", [0.5, 1.5, 2.5])
def test_scales(scale, nu):
    x = inputs.uniform(300, 2, seed=71)
    b = inputs.rhs(300, 2, seed=72)
    plain = refined(x, kc.Kernel(nu, 0.25, 1.0, 0.125), b)[0]
    got = refined(x * scale, kc.Kernel(nu, 0.25 * scale, 1.0, 0.125), b * 1e-30)[0] * 1e30
    assert torch.linalg.vector_norm(got - plain) <= 1e-9 * torch.linalg.vector_norm(plain)


@pytest.mark.parametrize("nu", [0.5, 1.5, 2.5])
def test_coinciding_and_distant_points(nu):
    x = np.repeat(inputs.uniform(100, 2, seed=81), 2, axis=0)
    x[150:] += 1e4  # far beyond the kernel's reach
    b = inputs.rhs(200, 2, seed=82) * np.exp(inputs.rng(83).uniform(-12, 0, (1, 200)))
    check(x, kc.Kernel(nu, 0.2, 1.0, 0.5), b)
