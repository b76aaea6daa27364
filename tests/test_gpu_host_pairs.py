"""Spin pairs from host memory: only the coefficients of spin s are copied to the device, and the results are
bit for bit those of device inputs, whatever the other half holds."""
import numpy as np
import pytest
import torch

from paper_0807_4494_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("precision", ["fp64", "fp32", "tf32x3"])
@pytest.mark.parametrize("pinned", [False, True])
@pytest.mark.parametrize("L,s,B", [(1, 0, 1), (33, 2, 1), (48, -1, 5)])
def test_host_input_equals_device_input(precision, pinned, L, s, B):
    from paper_0807_4494_gb300 import ssht
    dt = torch.complex128 if precision == "fp64" else torch.complex64
    flm = inputs.coeffs(L, s, B, seed=L)
    x = torch.from_numpy(np.stack([flm, np.full_like(flm, np.nan)], axis=1)).to(dt)
    plan = ssht.Plan(L, s, B, precision=precision, spin_pair=True)
    want = plan.inverse(x.cuda()).cpu()
    got = plan.inverse(x.pin_memory() if pinned else x)
    plan.check()
    assert not got.is_cuda and torch.equal(got, want) and torch.isfinite(torch.view_as_real(want)).all()
