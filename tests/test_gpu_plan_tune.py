"""A plan's tuner times every combination that differs and no other: the lanes of the
ring form, which has no staging depth, once, and reports the plan's depth with them."""
import pytest

from paper_1706_02205_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1706_02205_gb300 import kchol as kc  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("prec,ring,depth", [(kc.FP32_FORM, 8, 8), (kc.FP64, 4, 4)])
@pytest.mark.parametrize("aligned", [True, False])
def test_combinations(prec, ring, depth, aligned):
    x = torch.from_numpy(inputs.uniform(3000, 2, seed=700)).to(DEV)
    perm, l, xo = kc.order_points(x)
    pat = kc.build_pattern(xo, l, 3.0)
    kern = kc.Kernel(0.5, 0.2)
    dt = torch.float64 if prec == kc.FP64 else torch.float32
    val = torch.empty(pat.nnz + 1, dtype=dt, device=DEV)[0 if aligned else 1:][:pat.nnz]
    diag = torch.empty(3000, dtype=torch.float64, device=DEV)
    plan = kc.FactorPlan(pat, xo, [kern], prec=prec)
    n = kc.launch_count()
    best = plan.tune(val, diag)
    # a warm-up and the combinations, two kernels each; off the boundary no lanes take the ring form
    assert kc.launch_count() - n == 2 * (1 + (7 if aligned else 8))
    assert best["lanes_per_row"] in (2, 4, 8, 16) and best["unroll"] in (4, 8, 16)
    if aligned and best["lanes_per_row"] == ring:
        assert best["unroll"] == depth
    plan.launch(val, diag)
    assert plan.finish() == 0
    ref = kc.factor(pat, xo, kern, prec)
    assert float((val.double() - ref[0].double()).abs().max()) <= (1e-13 if prec == kc.FP64 else 1e-5)
