"""The powers of two of FP32-class plans' operands (one for 16 rows and 64 K in the torus products, one for a row
pair and 32 K in the split-FP16 contraction): scaling the data scales the results exactly, small magnitudes keep
their digits, and a field with a NaN or an infinity leaves the others as they are.

Bounds: those of the parity tests, 2e-6 (FP32) and 1e-6 (split FP16) max-norm."""
import pytest
import torch

from paper_0807_4494_gb300 import inputs

pytestmark = pytest.mark.gpu
SIZES = [(16, 3, 5), (70, 1, 5), (129, -2, 65), (257, 2, 3)]  # (L, s, B): one launch, products, two slices of fields


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def rel(a, b):
    return float((a - b).abs().max() / b.abs().max())


@pytest.mark.parametrize("precision", ["fp32", "tf32x3", "bf16x6"])
@pytest.mark.parametrize("L,s,B", SIZES)
def test_powers_of_two_and_non_finite_fields(precision, L, s, B):
    from paper_0807_4494_gb300 import ssht
    x = torch.from_numpy(inputs.coeffs(L, s, B, seed=3)).to(torch.complex64).cuda()
    plan = ssht.Plan(L, s, B, precision=precision)
    f = plan.inverse(x)
    y, a = plan.forward(f), plan.adjoint(f)
    for k in (-60, 37, 60):
        fk = plan.inverse(x * 2.0 ** k)
        assert torch.equal(fk, f * 2.0 ** k)
        assert torch.equal(plan.forward(fk), y * 2.0 ** k)
        assert torch.equal(plan.adjoint(fk), a * 2.0 ** k)
    bad = x.clone()
    at = s * s + L
    bad[1, at] = float("nan")
    bad[B - 1, at] = float("inf")
    fb = plan.inverse(bad)
    yb = plan.forward(fb)
    plan.check()
    keep = [b for b in range(B) if b not in (1, B - 1)]
    assert torch.equal(fb[keep], f[keep]) and torch.equal(yb[keep], y[keep])
    for b in (1, B - 1):
        assert not torch.isfinite(torch.view_as_real(fb[b])).any()
        assert not torch.isfinite(torch.view_as_real(yb[b])).all()


@pytest.mark.parametrize("precision,tol", [("fp32", 2e-6), ("tf32x3", 1e-6)])
@pytest.mark.parametrize("L,s,B", SIZES)
def test_small_magnitudes_keep_their_digits(precision, tol, L, s, B):
    from paper_0807_4494_gb300 import ssht
    x = torch.from_numpy(inputs.coeffs(L, s, B, seed=4)).to(torch.complex64).cuda()
    ref = ssht.Plan(L, s, B, precision="fp64")
    plan = ssht.Plan(L, s, B, precision=precision)
    for k in (-112, -116, -120):
        xk = x * 2.0 ** k
        fr = ref.inverse(xk.to(torch.complex128))
        fk = fr.to(torch.complex64)
        yr, ar = ref.forward(fk.to(torch.complex128)), ref.adjoint(fk.to(torch.complex128))
        assert rel(plan.inverse(xk).to(torch.complex128), fr) < tol, k
        assert rel(plan.forward(fk).to(torch.complex128), yr) < tol, k
        assert rel(plan.adjoint(fk).to(torch.complex128), ar) < tol, k
    plan.check()
