"""The ordering's bands against the oracle's brute force, bit for bit: point sets
with many points in few cells and many empty cells, ties and duplicates, sizes
around a block and around the greedy steps, and every kind of dimension."""
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


def clusters(N, d, seed):
    g = inputs.rng(seed)
    c = g.random((7, d))
    return c[g.integers(0, 7, N)] + g.standard_normal((N, d)) * 10.0 ** -g.uniform(1, 6, (N, 1))


def int_grid(side, d, seed):
    x = np.stack(np.meshgrid(*[np.arange(float(side))] * d, indexing="ij"), -1).reshape(-1, d)
    return x[inputs.rng(seed).permutation(len(x))]


CASES = [
    ("uniform129", lambda: inputs.uniform(129, 2, seed=21)),  # the greedy steps select all but the first
    ("uniform130", lambda: inputs.uniform(130, 2, seed=22)),  # one point is left to a band
    ("uniform257", lambda: inputs.uniform(257, 2, seed=1)),
    ("uniform258", lambda: inputs.uniform(258, 2, seed=2)),
    ("uniform4096", lambda: inputs.uniform(4096, 2, seed=3)),
    ("uniform4097", lambda: inputs.uniform(4097, 2, seed=4)),
    ("uniform20000", lambda: inputs.uniform(20000, 2, seed=5)),
    ("line5000", lambda: inputs.uniform(5000, 1, seed=6)),
    ("cube9000", lambda: inputs.uniform(9000, 3, seed=7)),
    ("d7", lambda: inputs.uniform(4500, 7, seed=8)),
    ("swiss9000", lambda: inputs.swiss_roll(9000, seed=9)),
    ("clusters2d", lambda: clusters(9000, 2, 10)),
    ("clusters3d", lambda: clusters(9000, 3, 11)),
    ("clusters6d", lambda: clusters(6000, 6, 12)),
    ("ties2d", lambda: int_grid(90, 2, 13)),
    ("ties3d", lambda: int_grid(19, 3, 14)),
    ("duplicates", lambda: np.repeat(inputs.uniform(40, 2, seed=15), 120, axis=0)),
    ("all_equal", lambda: np.ones((5000, 2))),
    ("collinear", lambda: np.outer(inputs.rng(16).random(6000), [1.0, 2.0, -1.0])),
    ("tiny_scale", lambda: inputs.uniform(5000, 2, seed=17) * 1e-160),
    ("huge_scale", lambda: inputs.uniform(5000, 2, seed=18) * 1e140),
]


@pytest.mark.parametrize("name,make", CASES, ids=[c[0] for c in CASES])
def test_order_is_the_greedy_one(name, make):
    x = np.ascontiguousarray(make())
    perm, l = oracle.maximin_brute(x)
    p, ll, xo = kc.order_points(torch.from_numpy(x).to(DEV))
    assert np.array_equal(p.cpu().numpy(), perm)
    assert np.array_equal(ll.cpu().numpy(), l)
    assert np.array_equal(xo.cpu().numpy(), x[perm])


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("at", [(0, 0), (4999, 2), (1234, 1)])
def test_points_that_are_not_finite_are_refused(bad, at):
    x = inputs.uniform(5000, 3, seed=19)
    x[at] = bad
    with pytest.raises(kc.KcError) as e:
        kc.order_points(torch.from_numpy(x).to(DEV))
    assert e.value.status == kc.KC_EINVAL
