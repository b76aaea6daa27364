"""The torus stage of small band-limits (one launch a direction on CUDA cores) against the oracle in all three
directions and every precision, on both sides of the rule that chooses it, and the memory such plans hold.

Bounds: those of the parity tests, 1e-12 (FP64, L <= 256), 2e-6 (FP32), 1e-6 (tensor cores) max-norm."""
import numpy as np
import pytest
import torch

from oracle import transforms as T
from paper_0807_4494_gb300 import inputs

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-12, "fp32": 2e-6, "tf32x3": 1e-6, "bf16x6": 1e-6}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


# (L, s, B): the smallest sizes; edges of blocks of 8 and 16 rings and orders and of 32 m'; several fields a CTA with a last
# one not full; the rule's lines: L = 4 and 5 and 127 and 128 fields up to L = 32 (FP64), L = 48 and 49, L = 64 and 65, B L^3 = 2^24 at L = 49 (142 and 143
# fields) and L = 64 (64 and 65)
@pytest.mark.parametrize("L,s,B", [(1, 0, 2), (2, 1, 1), (3, -1, 33), (4, 1, 2), (5, 2, 3), (5, -4, 129), (8, 0, 1000), (8, -7, 2), (9, 1, 1), (15, -2, 309),
                                   (16, 3, 1250), (17, -1, 2), (24, 0, 609), (28, 1, 127), (28, -2, 128), (31, 30, 3), (32, 2, 613), (32, -1, 1), (33, 0, 5),
                                   (47, -3, 2), (48, 1, 4), (49, -3, 142), (49, 2, 143), (63, 1, 1), (64, 0, 64), (64, -2, 65),
                                   (65, 1, 2)])
@pytest.mark.parametrize("precision", ["fp64", "fp32", "tf32x3", "bf16x6"])
def test_small_band_limits_match_oracle(precision, L, s, B):
    from paper_0807_4494_gb300 import ssht
    dt = torch.complex128 if precision == "fp64" else torch.complex64
    flm = inputs.coeffs(L, s, B, seed=L + B)
    plan = ssht.Plan(L, s, B, precision=precision)
    f = plan.inverse(torch.from_numpy(flm).to(dt).cuda()).cpu().numpy()
    rng = np.random.default_rng(L)
    g = torch.from_numpy(rng.standard_normal(f.shape) + 1j * rng.standard_normal(f.shape)).to(dt)
    fwd, adj = plan.forward(g.cuda()).cpu().numpy(), plan.adjoint(g.cuda()).cpu().numpy()
    plan.check()
    g = g.numpy().astype(np.complex128)
    x = torch.from_numpy(flm).to(dt).numpy().astype(np.complex128)
    for b in sorted({0, 1 % B, B // 2, B - 1}):
        assert rel(f[b], T.inverse(x[b], L, s)) < TOL[precision]
        assert rel(fwd[b], T.forward(g[b], L, s)) < TOL[precision]
        assert rel(adj[b], T.adjoint(g[b], L, s)) < TOL[precision]


@pytest.mark.parametrize("L", [2, 8, 16, 33, 48])
def test_memory_a_field(L):
    """An FP32 plan holds no more than two half rows [2L - 1][L] a field."""
    from paper_0807_4494_gb300 import ssht
    held = [ssht.Plan(L, 0, B, precision="fp32").workspace_bytes() for B in (1024, 4096)]
    assert (held[1] - held[0]) / 3072 <= 2 * (2 * L - 1) * L * 8
