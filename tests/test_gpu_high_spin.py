"""Tensor-core plans with spins beyond the first block of columns, against FP64 plans: above L = 1024 near the
band-limit, where a plan has as few recursion tasks as one of small band-limit, but first rows below the FP64 range
that carry exponents of their own; and above L = 512, where plan creation makes only the part of the table that the
spin column reads.  Bound 2e-6 max-norm, that of the L = 2048 tests."""
import pytest
import torch

from paper_0807_4494_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("L,s", [(600, 31), (600, -70), (1100, 1040), (1280, 1200), (1280, -1200)])
def test_high_spins(L, s):
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
