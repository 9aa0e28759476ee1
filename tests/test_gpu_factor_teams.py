"""Teams of warps where the CTA size or the rows of a task are asked for: every CTA
size, teams of any divisor of it, tasks of fewer rows than a team has rounds for: the
bits of the default, and no more time beside it than such tasks need."""
import time

import pytest

from paper_1706_02205_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1706_02205_gb300 import kchol as kc  # noqa: E402

DEV = torch.device("cuda:0")


def cube(N, rho):
    x = torch.from_numpy(inputs.uniform(N, 3, seed=500)).to(DEV)
    perm, l, xo = kc.order_points(x)
    return xo, kc.build_pattern(xo, l, rho)


@pytest.mark.parametrize("rho", [3.0, 5.0, 9.0])  # longest rows: tables of 2^9, 2^10 and 2^11 slots or more
@pytest.mark.parametrize("prec", [kc.FP32_FORM, kc.FP64])
def test_every_cta_size_same_bits(rho, prec):
    xo, pat = cube(3001, rho)
    kern = kc.Kernel(0.5, 0.3)
    ref = kc.factor(pat, xo, kern, prec)
    for warps in range(1, 9):
        for rows in (0, 1, 4, 7, 8, 16, 24, 100):
            got = kc.factor(pat, xo, kern, prec, kc.make_opts(warps_per_cta=warps, rows_per_task=rows))
            assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1]) and got[2] == ref[2], (warps, rows)


# 40,000 points of the cube, rho = 4, ms by default and as asked for: a warp a task of 4 rows 22 and 45 (FP32 form), 37
# and 124 (FP64), teams 75 and 183; a team of 3 warps 40 (FP64), a table a warp about 105
@pytest.mark.parametrize("prec,opts,bound", [(kc.FP32_FORM, dict(rows_per_task=4), 2.7),
                                             (kc.FP64, dict(rows_per_task=4), 3.9),
                                             (kc.FP64, dict(warps_per_cta=3), 1.7)])
def test_time_beside_the_default(prec, opts, bound):
    xo, pat = cube(40000, 4.0)
    best = []
    for o in (None, kc.make_opts(**opts)):
        kc.factor(pat, xo, kc.Kernel(1.5, 0.1), prec, o)
        ts = []
        for _ in range(3):
            torch.cuda.synchronize()
            t = time.perf_counter()
            kc.factor(pat, xo, kc.Kernel(1.5, 0.1), prec, o)
            torch.cuda.synchronize()
            ts.append(time.perf_counter() - t)
        best.append(min(ts))
    assert best[1] <= bound * best[0]
