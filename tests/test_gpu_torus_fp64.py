"""FP64 plans on both sides of the rule that chooses the torus stage -- products or FFTs (the batch and
the factors of N = 2L - 1 decide) -- against the FP64 oracle in all three directions.

Bound 1e-12 max-norm, that of the FP64 parity tests at L <= 256."""
import numpy as np
import pytest
import torch

from oracle import transforms as T
from paper_0807_4494_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


# (L, s, B): smallest sizes; edges of 32 rows; N = 199 prime with a large batch (products); N = 255 = 3 5 17
# and N = 189 = 3^3 7 with B L^3 just below and above 2^23 (products, FFTs); L = 209 (N = 3 139), above the line
@pytest.mark.parametrize("L,s,B", [(1, 0, 3), (2, -1, 2), (3, 2, 1), (32, 1, 2), (33, -2, 1), (65, 0, 2), (100, 2, 10),
                                   (128, 1, 4), (128, -1, 5), (95, 0, 9), (95, 2, 10), (203, 1, 1), (209, 0, 1)])
def test_both_torus_stages_match_oracle(L, s, B):
    from paper_0807_4494_gb300 import ssht
    flm = inputs.coeffs(L, s, B, seed=L + B)
    plan = ssht.Plan(L, s, B, precision="fp64")
    f = plan.inverse(torch.from_numpy(flm).cuda())
    rng = np.random.default_rng(L)
    g = rng.standard_normal(f.shape) + 1j * rng.standard_normal(f.shape)
    gd = torch.from_numpy(g).cuda()
    fwd, adj = plan.forward(gd).cpu().numpy(), plan.adjoint(gd).cpu().numpy()
    plan.check()
    assert rel(f.cpu().numpy(), T.inverse(flm, L, s)) < 1e-12
    assert rel(fwd, T.forward(g, L, s)) < 1e-12
    assert rel(adj, T.adjoint(g, L, s)) < 1e-12
