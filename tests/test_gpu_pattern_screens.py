"""The pattern search against the definition, entry for entry, where distances lie
at or within float's resolution of the radii, far from the origin, and at extents
where only the exact test runs; every number of axes the kernels tell apart."""
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
SHAPES = {"1d": (600,), "2d": (31, 27), "3d": (9, 11, 8), "4d": (5, 6, 4, 5)}


@pytest.mark.parametrize("rule", [0, 1], ids=["max", "min"])
@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("scale,shift,jitter",
                         [(1.0, 0.0, 0.0), (1.0, 2.0**20, 0.0), (1.0, 0.0, 1e-8), (2.0**-60, 0.0, 0.0),
                          (2.0**-20, 0.0, 1e-7), (2.0**57, 0.0, 0.0), (2.0**80, 0.0, 0.0)])
def test_pattern_is_the_defined_one(shape, rule, scale, shift, jitter):
    g = np.stack(np.meshgrid(*[np.arange(float(n)) for n in SHAPES[shape]], indexing="ij"), -1)
    g = g.reshape(-1, g.shape[-1])
    r = inputs.rng(301)
    x = (g + jitter * r.uniform(-1.0, 1.0, g.shape))[r.permutation(len(g))] * scale + shift
    rho = 2.0
    perm, l, xo = kc.order_points(torch.from_numpy(np.ascontiguousarray(x)).to(DEV))
    pat = kc.build_pattern(xo, l, rho, rule=rule)
    rowptr, col = oracle.pattern(xo.cpu().numpy(), l.cpu().numpy(), rho, rule)
    assert np.array_equal(pat.rowptr.cpu().numpy(), rowptr)
    assert np.array_equal(pat.col.cpu().numpy(), col)
