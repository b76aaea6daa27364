"""The bounds-checked build on the kernels of FP64 plans and of small band-limits: every form of the torus stage (one
launch, CUDA-core products, digit products with tiles of 16 and 32 columns, one and two segments) and of the contractions (CUDA
cores, digits with items of four and eight fields, ragged groups, |s| beyond the first row blocks), in a child process on
that library; no access may fall outside its buffer, and the results match the oracle.

Bounds: those of the parity tests, 1e-12 (FP64, 1e-11 above L = 256), 2e-6 (FP32), 1e-6 (tensor cores)."""
import os
import re
import subprocess
import sys
import textwrap

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_0807_4494_gb300", "csrc")

CHILD = textwrap.dedent(r"""
    import numpy as np
    import torch
    from oracle import transforms as T
    from paper_0807_4494_gb300 import inputs, ssht

    TOL = {"fp64": 1e-12, "fp32": 2e-6, "tf32x3": 1e-6, "bf16x6": 1e-6}

    def rel(a, b):
        return float(np.abs(np.asarray(a) - np.asarray(b)).max() / np.abs(np.asarray(b)).max())

    def clean(what):
        n, site, idx, ext = ssht.ssht_debug_bounds()
        assert n == 0, "%s: %d accesses outside their buffers, first at site %d: index %d of %d" % (what, n, site, idx, ext)

    clean("start")
    cases = [(1, 0, 3, "fp64"), (17, 2, 2, "fp64"), (8, 1, 700, "fp64"), (40, 1, 3, "fp64"), (65, 0, 2, "fp64"), (129, 2, 1, "fp64"),
             (161, 1, 7, "fp64"), (33, -2, 70, "fp64"), (129, -64, 5, "fp64"), (64, -63, 33, "fp64"), (160, 3, 3, "fp64"),
             (257, -2, 1, "fp64"), (513, 1, 1, "fp64"), (2, 1, 33, "fp32"), (16, 1, 1250, "fp32"), (33, -5, 3, "tf32x3"),
             (48, 2, 300, "bf16x6"), (64, 0, 2, "tf32x3"), (9, 8, 609, "tf32x3")]
    for L, s, B, prec in cases:
        dt = torch.complex128 if prec == "fp64" else torch.complex64
        flm = inputs.coeffs(L, s, B, seed=L + B)
        plan = ssht.Plan(L, s, B, precision=prec)
        f = plan.inverse(torch.from_numpy(flm).to(dt).cuda())
        back, adj = plan.forward(f), plan.adjoint(f)
        plan.check()
        clean("L=%d s=%d B=%d %s" % (L, s, B, prec))
        tol = 1e-11 if prec == "fp64" and L > 256 else TOL[prec]
        fo, bo, ao = f.cpu().numpy(), back.cpu().numpy(), adj.cpu().numpy()
        x = torch.from_numpy(flm).to(dt).numpy().astype(np.complex128)
        for b in sorted({0, B - 1}):
            g = fo[b].astype(np.complex128)
            assert rel(fo[b], T.inverse(x[b], L, s)) < tol, (L, s, B, prec, "inverse", b)
            assert rel(bo[b], T.forward(g, L, s)) < tol, (L, s, B, prec, "forward", b)
            assert rel(ao[b], T.adjoint(g, L, s)) < tol, (L, s, B, prec, "adjoint", b)
        plan.close()
    # the triangular forward on a plan whose other directions use no FFT, real fields, spin pairs, the kept table
    for L, kw in ((24, {}), (140, {"real": True}), (140, {"spin_pair": True}), (140, {"delta_mode": "cache"})):
        plan = ssht.Plan(L, 0, 5, precision="fp64", **kw)
        x = torch.zeros(plan.coeff_shape(), dtype=plan.dtype, device="cuda")
        x[..., :4] = 1.0
        f = plan.inverse(x)
        plan.forward(f)
        if not plan.spin_pair:
            plan.forward_triangular(f)
        plan.check()
        clean(str((L, kw)))
        plan.close()
    print("bounds-checked build: clean")
""")


def test_kernels_with_index_checks():
    """Every source with transform kernels keeps a record of its index checks, and the library reads them all (the
    Risbo recursion, the triangular forward's kernels and the API have none)."""
    have = {}
    for name in os.listdir(CSRC):
        if name.endswith(".cu"):
            with open(os.path.join(CSRC, name)) as f:
                text = f.read()
            tag = re.findall(r"^SSHT_BOUNDS_TU\((\w+)\)", text, re.M)
            if tag or "__global__" in text:
                have[name] = tag
    assert {n for n, tag in have.items() if not tag} == {"delta.cu", "torus.cu", "triangular.cu"}
    with open(os.path.join(CSRC, "api.cu")) as f:
        read = set(re.findall(r"bounds_take_(\w+)", f.read()))
    assert read == {tag[0] for tag in have.values() if tag}


@pytest.mark.gpu
def test_bounds_checked_build_on_fp64_plans_and_small_band_limits():
    from paper_0807_4494_gb300 import build
    lib = build.build(debug=True)
    env = dict(os.environ, SSHT_LIBRARY=lib, PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True, timeout=1200)
    assert r.returncode == 0, r.stdout[-4000:] + r.stderr[-4000:]
    assert "bounds-checked build: clean" in r.stdout
