"""The CUDA-core projection with few fields: against the oracle at the edges of its blocks of degrees and lanes, and
one field against two in time (the loads of the table are the same, so one never takes longer).

Bounds: 1e-12 (FP64) and 2e-6 (FP32) max-norm, those of the parity tests; a tenth above in time."""
import numpy as np
import pytest
import torch

from oracle import transforms as T

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 2e-6)])
@pytest.mark.parametrize("L,s", [(1, 0), (2, -1), (3, 0), (17, 2), (33, -32), (66, 1), (95, -2)])
@pytest.mark.parametrize("B", [1, 2, 3, 9])
def test_projection_matches_oracle(precision, tol, L, s, B):
    from paper_0807_4494_gb300 import ssht
    dt = torch.complex128 if precision == "fp64" else torch.complex64
    rng = np.random.default_rng(L)
    g = torch.from_numpy(rng.standard_normal((B, L, 2 * L - 1)) + 1j * rng.standard_normal((B, L, 2 * L - 1))).to(dt)
    plan = ssht.Plan(L, s, B, precision=precision)
    fwd, adj = plan.forward(g.cuda()).cpu().numpy(), plan.adjoint(g.cuda()).cpu().numpy()
    plan.check()
    g = g.numpy().astype(np.complex128)
    for got, want in ((fwd, T.forward(g, L, s)), (adj, T.adjoint(g, L, s))):
        assert np.abs(got - want).max() / np.abs(want).max() < tol


@pytest.mark.parametrize("L", [512, 1024])
def test_one_field_takes_no_longer_than_two(L):
    from paper_0807_4494_gb300 import ssht
    us = {}
    for B in (1, 2):
        plan = ssht.Plan(L, 0, B, precision="fp32", delta_mode="cache")
        f = torch.randn(B, L, 2 * L - 1, dtype=torch.complex64, device="cuda")
        out = plan.forward(f)
        best = np.inf
        for _ in range(5):
            plan.profile(True)
            for _ in range(3):
                plan.forward(f, out=out)
            best = min(best, plan.profile_read()[0]["project"][0])
        us[B] = best
        plan.close()
    assert us[1] < 1.1 * us[2], us
