"""FP32-class plans with so many fields that the torus passes run in slices of them: the memory they hold, and each
field's results bit for bit those of a plan that takes it in one slice (fields share nothing but launches)."""
import pytest
import torch

from paper_0807_4494_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


# three slices, the last one shorter, of band-limits whose operands are padded most
@pytest.mark.parametrize("precision", ["fp32", "tf32x3", "bf16x6"])
@pytest.mark.parametrize("L,s,B,fields", [(66, -1, 8300, 2767), (131, 2, 4000, 1334)])
def test_slices_of_fields(precision, L, s, B, fields):
    from paper_0807_4494_gb300 import ssht
    base = torch.from_numpy(inputs.coeffs(L, s, 5, seed=L)).to(torch.complex64).cuda()
    x = base[torch.arange(B, device="cuda") % 5].contiguous()
    plan = ssht.Plan(L, s, B, precision=precision)
    one = ssht.Plan(L, s, 5, precision=precision)
    f = plan.inverse(x)
    want = one.inverse(base)
    g = torch.randn(5, L, 2 * L - 1, dtype=torch.complex64, generator=torch.Generator().manual_seed(1)).cuda()
    gx = g[torch.arange(B, device="cuda") % 5].contiguous()
    fwd, adj = plan.forward(gx), plan.adjoint(gx)
    wf, wa = one.forward(g), one.adjoint(g)
    plan.check()
    for b in {0, 1, fields - 1, fields, fields + 3, 2 * fields - 1, 2 * fields, B - 2, B - 1}:
        assert torch.equal(f[b], want[b % 5]), b
        assert torch.equal(fwd[b], wf[b % 5]), b
        assert torch.equal(adj[b], wa[b % 5]), b


@pytest.mark.parametrize("L,B", [(65, 20000), (129, 8000), (300, 2000)])
def test_memory_of_many_fields(L, B):
    """An FP32 plan holds no more than two half rows [2L - 1][L] a field, and 2 GiB."""
    from paper_0807_4494_gb300 import ssht
    few = ssht.Plan(L, 0, 1, precision="fp32").workspace_bytes()
    assert ssht.Plan(L, 0, B, precision="fp32").workspace_bytes() - few <= 2 * B * (2 * L - 1) * L * 8 + (2 << 30)
