"""The supernodal construction's distance tests with an FP32 screen before the
exact test: bit-exact against the oracle where many distances lie at, or within
float's resolution of, the radii, far from the origin, and at extents where
only the exact test runs."""
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


def _lattice(shape, seed, jitter=0.0):
    g = np.stack(np.meshgrid(*[np.arange(float(n)) for n in shape], indexing="ij"), -1).reshape(-1, len(shape))
    r = inputs.rng(seed)
    return (g + jitter * r.uniform(-1.0, 1.0, g.shape))[r.permutation(len(g))]


@pytest.mark.parametrize("shape", [(29, 37), (11, 9, 10)], ids=["2d", "3d"])
@pytest.mark.parametrize("scale,shift,jitter",
                         [(1.0, 0.0, 0.0), (1.0, 2.0**20, 0.0), (1.0, 0.0, 1e-9), (2.0**-52, 0.0, 0.0),
                          (2.0**-20, 0.0, 1e-8), (2.0**60, 0.0, 0.0)])
def test_screened_distances_are_exact(shape, scale, shift, jitter):
    x = _lattice(shape, 201, jitter) * scale + shift
    rho = 2.0
    ref = oracle.supernodal(x, rho)
    X = torch.from_numpy(np.ascontiguousarray(x)).to(DEV)
    perm0, l, xo = kc.order_points(X)
    sn = kc.supernodal(xo, l, rho, kc.build_pattern(xo, l, rho))
    assert np.array_equal(perm0.cpu().numpy()[sn["newm"].cpu().numpy()], ref["order"])
    for k in ("level", "node", "color"):
        assert np.array_equal(sn[k].cpu().numpy(), ref[k])
    assert np.array_equal(sn["pat"].rowptr.cpu().numpy(), ref["rowptr"])
    assert np.array_equal(sn["pat"].col.cpu().numpy(), ref["col"])
