"""The refined solve's product with Theta, entry by entry: with the identity as the
preconditioner two steps of conjugate gradients from b give x = a b + c (b - a Theta b
+ e b) with numbers a, c, e that follow from Theta and b, so x shows Theta b row by row.
Rows that carry little beside the largest values (one-hot vectors, far clusters of
other scales, steep ramps) keep FP64's accuracy relative to what they sum, a point that
is not finite spreads as in FP64 sums, and ordinary vectors are as close in the norm as
the split promises."""
import numpy as np
import pytest

from paper_1706_02205_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1706_02205_gb300 import kchol as kc  # noqa: E402

DEV = torch.device("cuda:0")
LD = np.longdouble
U = 2.0**-53


def T(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def theta(x, kern):
    r = np.sqrt(((x.astype(LD)[:, None, :] - x.astype(LD)[None, :, :]) ** 2).sum(-1))
    t = np.sqrt(LD(2 * kern.nu)) * r / LD(kern.ell)
    f = {0.5: LD(1), 1.5: 1 + t, 2.5: 1 + t + t * t / 3}[kern.nu]
    return LD(kern.sigma2) * f * np.exp(-t) + LD(kern.nugget) * np.eye(len(x), dtype=LD), t


def two_steps(x, kern, b, scale=1.0):
    """x of the GPU after two steps from b, and from 80-bit sums x, and what every row of x sums in magnitude.  The
    preconditioner is scale^2 times the identity: that changes no step, but a large one passes for large row weights."""
    N = len(x)
    rowptr, col = np.arange(N + 1, dtype=np.int64), np.arange(N, dtype=np.int32)
    pat = kc.schedule(T(rowptr), T(col))
    one = torch.ones(N, dtype=torch.float64, device=DEV)
    got, it, _, _ = kc.refine(pat, T(x), kern, kc.FP64, one, scale * one, T(col), T(b), rtol=1e-300, maxit=2)
    assert it == 2
    G, _ = theta(x, kern)
    want, size = [], []
    for v in b.astype(LD):
        q = G @ v
        a = (v @ v) / (v @ q)
        r = v - a * q
        e = (r @ r) / (v @ v)
        p = r + e * v
        c = (r @ r) / (p @ (G @ p))
        want.append(a * v + c * p)
        size.append((abs(a) + abs(c) * (1 + e)) * abs(v) + abs(c * a) * (np.abs(G) @ np.abs(v)))
    return got.cpu().numpy(), np.array(want), np.array(size)


def vectors(kind, x, seed):
    N, g = len(x), inputs.rng(seed)
    if kind == "one-hot":
        b = np.zeros((3, N))
        b[0, 0] = b[1, N // 2] = b[2, N - 1] = 1.0
        return b
    b = g.standard_normal((2, N))
    if kind == "clusters":
        b[:, x[:, 0] > 10] *= 2.0**-45
    elif kind == "ramp":
        b *= np.exp(12 * (x[:, 0] - x[:, 0].min()))
    return b


# what a row sums is at least its largest term, and FP64 evaluates an entry e^-t to (4 + t) units or so (t has four
# roundings before the exponential, which multiplies their sum by t); N sums add at most their square root in practice
def bound(N, t):
    return (8 + 2 * t + 2 * np.sqrt(N)) * U


@pytest.mark.parametrize("nu", [0.5, 1.5, 2.5])
@pytest.mark.parametrize("kind", ["one-hot", "clusters", "ramp"])
@pytest.mark.parametrize("d", [1, 2, 3, 5])
def test_rows_of_little_weight(kind, nu, d):
    N = 300
    x = inputs.uniform(N, d, seed=600 + d)
    if kind == "clusters":
        x[::2, 0] += 100.0  # neighbours in the order lie in different clusters
    kern = kc.Kernel(nu, 0.05, 1.0, 0.0)
    got, want, size = two_steps(x, kern, vectors(kind, x, 601))
    t = np.minimum(theta(x, kern)[1].max(), 745.0).astype(float)
    assert np.isfinite(got).all()
    ok = size > 1e-280
    assert np.max(np.abs(got - want)[ok] / size[ok]) <= bound(N, t)


@pytest.mark.parametrize("nu", [0.5, 1.5, 2.5])
@pytest.mark.parametrize("d", [1, 2, 3, 5])
@pytest.mark.parametrize("N", [129, 777])
def test_ordinary_vectors(N, d, nu):
    """x lies in the plane of b and Theta b whatever the numbers a, c, e (dot products, whose rounding a short residual
    magnifies): its distance from that plane is what the product and the vector steps rounded."""
    x = inputs.uniform(N, d, seed=610 + d)
    kern = kc.Kernel(nu, 0.2, 2.5, 0.01)
    b = inputs.rng(611).standard_normal((3, N))
    got, _, size = two_steps(x, kern, b, scale=2.0**20)
    G, _ = theta(x, kern)
    for g, v, s in zip(got, b.astype(LD), size):
        q = G @ v
        g, e1 = g.astype(LD), v / np.sqrt(v @ v)
        e2 = q - (q @ e1) * e1
        e2 /= np.sqrt(e2 @ e2)
        rest = g - (g @ e1) * e1 - (g @ e2) * e2
        share = abs((g @ e2) / (q @ e2))  # of Theta b in x
        # the product is up to 2.0e-16 |Theta b| off, each of the three vector steps half a unit of what it sums
        assert np.sqrt(rest @ rest) <= share * 2.0e-16 * np.sqrt(q @ q) + 3 * U * np.sqrt(s @ s)


def test_a_point_that_is_not_finite_shows():
    """A distance that is not a number makes the product one, as FP64 sums do; it is not a zero entry."""
    N = 200
    x, b = inputs.uniform(N, 2, seed=620), np.ones((1, N))
    x[7, 1] = np.nan
    rowptr, col = np.arange(N + 1, dtype=np.int64), np.arange(N, dtype=np.int32)
    one = torch.ones(N, dtype=torch.float64, device=DEV)
    got, _, rel, st = kc.refine(kc.schedule(T(rowptr), T(col)), T(x), kc.Kernel(0.5, 0.2), kc.FP64, one, one, T(col),
                                T(b), rtol=1e-10, maxit=1)
    assert st == kc.KC_EINDEF and not np.isfinite(rel[0])
