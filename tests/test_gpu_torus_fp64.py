"""FP64 plans on both sides of the rule that chooses the torus stage -- products on CUDA cores or of digits on
tensor cores -- and of the one that chooses the contractions, against the FP64 oracle in all three directions; the
digits' scaling over the exponent range.

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


# (L, s, B): smallest sizes; edges of 32 rows and k's and of 128 rows; B L^3 on both sides of 2^21 (128, 1 and 129, 1); data
# tiles of 16 and 32 columns with a last one not full; more than 512 k's (two segments of sums, and packing in two reads);
# contractions of digits (B L^3 > 2^23, 64 <= L <= 512): one to 33 fields in groups of four or eight, edges of 32 k's and 128 rows, |s|
# beyond the first row blocks
@pytest.mark.parametrize("L,s,B", [(1, 0, 3), (2, -1, 2), (3, 2, 1), (32, 1, 2), (33, -2, 1), (65, 0, 2), (100, 2, 10),
                                   (128, 1, 4), (128, -1, 5), (95, 0, 9), (95, 2, 10), (203, 1, 1), (209, 0, 1),
                                   (32, -1, 80), (33, 0, 64), (33, -2, 70), (127, 1, 2), (128, 0, 1), (129, 2, 1), (161, 1, 7),
                                   (513, 1, 1), (128, 0, 5), (128, 1, 8), (128, 2, 17), (129, 2, 4), (129, -64, 5), (64, 1, 33), (64, -63, 33), (100, 0, 9),
                                   (257, -2, 1), (384, 1, 1), (512, 0, 1)])
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


@pytest.mark.parametrize("recursion,delta_mode", [("risbo", "recompute"), ("risbo", "cache"), ("column", "cache")])
def test_digit_contractions_of_every_table(recursion, delta_mode):
    """The contractions of digits read the table of either recursion, made in the call or kept."""
    from paper_0807_4494_gb300 import ssht
    L, s, B = 140, -1, 4
    flm = inputs.coeffs(L, s, B, seed=5)
    plan = ssht.Plan(L, s, B, precision="fp64", recursion=recursion, delta_mode=delta_mode)
    f = plan.inverse(torch.from_numpy(flm).cuda())
    back = plan.forward(f).cpu().numpy()
    plan.check()
    assert rel(f.cpu().numpy(), T.inverse(flm, L, s)) < 1e-12
    assert rel(back, flm) < 1e-12


def test_powers_of_two_and_non_finite_rows():
    """Fixed point with a row's own power of two: scaling a field by 2^k scales the outputs exactly, and a field
    with a NaN or an infinity leaves the other fields' outputs as they are."""
    from paper_0807_4494_gb300 import ssht
    L, s, B = 140, 1, 5
    x = torch.from_numpy(inputs.coeffs(L, s, B, seed=3)).cuda()
    plan = ssht.Plan(L, s, B, precision="fp64")
    f = plan.inverse(x)
    y, a = plan.forward(f), plan.adjoint(f)
    for k in (-900, -300, 37, 800):
        fk = plan.inverse(x * 2.0 ** k)
        assert torch.equal(fk, f * 2.0 ** k)
        assert torch.equal(plan.forward(fk), y * 2.0 ** k)
        assert torch.equal(plan.adjoint(fk), a * 2.0 ** k)
    bad = x.clone()
    bad[1, 7] = float("nan")
    bad[3, 9] = float("inf")
    fb = plan.inverse(bad)
    yb = plan.forward(fb)
    plan.check()
    keep = [0, 2, 4]
    assert torch.equal(fb[keep], f[keep]) and torch.equal(yb[keep], y[keep])
    for b in (1, 3):
        assert not torch.isfinite(torch.view_as_real(fb[b])).any()
        assert not torch.isfinite(torch.view_as_real(yb[b])).all()


def test_real_pair_and_group_forms_of_digit_plans():
    """Real fields against the oracle; a group's buckets (concurrent, and replayed from a capture) bit for bit
    against plans of their own."""
    from paper_0807_4494_gb300 import ssht
    L, B = 140, 8
    flm = inputs.coeffs(L, 0, B, seed=9, real=True)
    plan = ssht.Plan(L, 0, B, precision="fp64", real=True)
    f = plan.inverse(torch.from_numpy(flm).cuda())
    back = plan.forward(f).cpu().numpy()
    plan.check()
    for b in range(B):
        assert rel(f[b].cpu().numpy(), T.inverse(flm[b], L, 0).real) < 1e-12
        assert rel(back[b], flm[b]) < 1e-12

    Ls, ss = [140] * 4 + [210] * 2 + [40] * 3 + [140] * 5, [0] * 4 + [-1] * 2 + [2] * 3 + [1] * 5
    x = [torch.from_numpy(inputs.coeffs(l, s, 1, seed=i)[0]).cuda() for i, (l, s) in enumerate(zip(Ls, ss))]
    g = ssht.Group(Ls, ss, precision="fp64", tune=False)
    flat = g.pack_coeffs(x)
    grid, out = g.inverse(flat), None
    out = g.forward(grid)
    grid2, out2 = g.empty_grid(), g.empty_coeffs()
    g.capture(flat, grid2, out2)
    g.replay()
    torch.cuda.synchronize()
    g.check()
    assert torch.equal(grid2, grid) and torch.equal(out2, out)
    fs, bs = g.unpack_grid(grid), g.unpack_coeffs(out)
    for l, s in set(zip(Ls, ss)):
        idx = [i for i in range(len(Ls)) if (Ls[i], ss[i]) == (l, s)]
        p = ssht.Plan(l, s, len(idx), precision="fp64")
        want = p.inverse(torch.stack([x[i] for i in idx]))
        wb = p.forward(want)
        for k, i in enumerate(idx):
            assert torch.equal(fs[i], want[k]) and torch.equal(bs[i], wb[k])
