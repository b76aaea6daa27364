"""Tensor-core plans above L = 1024 with spins near the band-limit, against FP64 plans.

Such a plan has as few recursion tasks as one of small band-limit, but its first rows lie below the
FP64 range and carry exponents of their own.  Bound 2e-6 max-norm, that of the L = 2048 tests."""
import pytest
import torch

from paper_0807_4494_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("L,s", [(1100, 1040), (1280, 1200), (1280, -1200)])
def test_tensor_core_plans_with_few_tasks_above_L1024(L, s):
    from paper_0807_4494_gb300 import ssht
    x = torch.from_numpy(inputs.coeffs(L, s, 1, seed=1)).cuda()
    ref = ssht.Plan(L, s, 1, precision="fp64")
    f = ref.inverse(x)
    back = ref.forward(f)
    ref.check()
    ref.close()
    for precision in ("tf32x3", "bf16x6"):
        plan = ssht.Plan(L, s, 1, precision=precision)
        g = plan.inverse(x.to(torch.complex64))
        y = plan.forward(f.to(torch.complex64))
        plan.check()
        plan.close()
        assert float((g - f).abs().max() / f.abs().max()) < 2e-6, (precision, "inverse")
        assert float((y - back).abs().max() / back.abs().max()) < 2e-6, (precision, "forward")
