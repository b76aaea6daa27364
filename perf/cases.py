"""Workloads of the spin spherical harmonic transform whose speed is measured.

A case is what a user's program does over and over with one plan: a synthesis (inverse) followed
by an analysis (forward), a synthesis with its gradient (the adjoint), an uneven batch replayed as
one CUDA graph, or a round trip through host buffers.  ``prepare`` makes the plan and the inputs,
``run`` is one pass through the public entry points, ``exact`` the same outputs by direct sums
over Wigner functions d^l_{m,-s}(theta) in FP64, which share nothing with the library's method
(the three-term relation in l at every colatitude instead of a Fourier series).
"""
import math

import numpy as np
import torch

from paper_0807_4494_gb300 import ssht


def _case(name, kind, precision, L, s, batch, spectrum="flat", delta_mode="recompute", real=False, pair=False):
    return {"name": name, "kind": kind, "precision": precision, "L": L, "s": s, "batch": batch,
            "spectrum": spectrum, "delta_mode": delta_mode, "real": real, "pair": pair}


def listed():
    return [
        # One small spin-2 field in double precision: the interactive call, all latency.
        _case("fp64_single_L64", "roundtrip", "fp64", 64, 2, 1),
        # One scalar field at the largest band-limit that is held to 1e-11.
        _case("fp64_single_L512", "roundtrip", "fp64", 512, 0, 1),
        # A few double-precision fields at an odd band-limit, the plan kept with its Delta table
        # for many calls (an iterative solver).
        _case("fp64_batch_L129", "roundtrip", "fp64", 129, -1, 4, delta_mode="cache"),
        # Single precision on the CUDA cores: a handful of maps of moderate band-limit.
        _case("fp32_batch_L256", "roundtrip", "fp32", 256, 1, 8),
        # Small batched maps with a kept Delta table (training on many small spheres).
        _case("tf32x3_small_L128", "roundtrip", "tf32x3", 128, 0, 16, delta_mode="cache"),
        # A differentiable layer at an odd band-limit and batch: inverse, then its adjoint.
        _case("tf32x3_gradient_L257", "gradient", "tf32x3", 257, -2, 33),
        # Real scalar fields, two to a complex transform.
        _case("tf32x3_real_L512", "roundtrip", "tf32x3", 512, 0, 64, spectrum="cmb", real=True),
        # Spin pairs from and to pinned host memory: Monte Carlo maps kept on the host.
        _case("tf32x3_host_L512", "host", "tf32x3", 512, 2, 24, spectrum="cmb", pair=True),
        # The headline: a CMB-like ensemble, Delta recomputed in every call.
        _case("tf32x3_batch_L1024", "roundtrip", "tf32x3", 1024, 2, 64, spectrum="cmb"),
        # The same ensemble with the split-BF16 contraction.
        _case("bf16x6_batch_L1024", "roundtrip", "bf16x6", 1024, 2, 64, spectrum="cmb"),
        # The highest band-limit.
        _case("bf16x6_batch_L2048", "roundtrip", "bf16x6", 2048, 2, 16, spectrum="cmb"),
        # 256 fields of uneven band-limit and spin in one captured graph, tuned buckets.
        {"name": "group_uneven_256", "kind": "group", "precision": "fp32", "fields": 256, "Ls": "128,256,512,1024",
         "spins": "0,1,-1,2,-2", "pick": 0, "tune": True},
    ]


def _log_uniform(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["roundtrip"] * 6 + ["gradient"] * 2 + ["host", "group"])
    if kind == "group":
        Ls = sorted(rng.sample(range(48, 640), rng.randint(2, 4)))
        return {"kind": "group", "precision": rng.choice(["fp32", "tf32x3"]), "fields": _log_uniform(rng, 8, 128),
                "Ls": ",".join(str(x) for x in Ls), "spins": "0,1,-1,2,-2", "pick": rng.randrange(1 << 16),
                "tune": rng.random() < 0.5}
    precision = rng.choice(["fp64", "fp64", "fp32", "tf32x3", "tf32x3", "tf32x3", "bf16x6"])
    # the contraction's work B L^3 is bounded by that of the largest listed case of the precision
    top, most = {"fp64": (512, 512 ** 3), "fp32": (512, 8 * 512 ** 3)}.get(precision, (1536, 64 * 1024 ** 3))
    L = _log_uniform(rng, 32, top)
    batch = _log_uniform(rng, 1, max(1, min(96, most // L ** 3)))
    s = rng.choice([0, 0, 1, -1, 2, 2, -2])
    real = s == 0 and kind == "roundtrip" and rng.random() < 0.4
    pair = not real and kind == "roundtrip" and rng.random() < 0.15
    return {"kind": kind, "precision": precision, "L": L, "s": s, "batch": batch, "spectrum": rng.choice(["flat", "cmb"]),
            "delta_mode": rng.choice(["recompute", "recompute", "cache"]), "real": real, "pair": pair}


# ---- inputs ---------------------------------------------------------------------------------

def _device():
    return torch.device("cuda", torch.cuda.current_device()) if torch.cuda.is_available() else torch.device("cpu")


def _degrees(L, device):
    l = torch.repeat_interleave(torch.arange(L, device=device), 2 * torch.arange(L, device=device) + 1)
    m = torch.arange(L * L, device=device) - l * l - l
    return l, m


def _coeffs(gen, L, s, batch, spectrum, real, double):
    """Band-limited coefficients [batch, L*L]: iid N(0,1) parts, or the CMB-like spectrum 1/(l+1)^2."""
    device = gen.device
    x = torch.randn(batch, L * L, 2, generator=gen, device=device, dtype=torch.float64 if double else torch.float32)
    l, m = _degrees(L, device)
    scale = (l >= abs(s)).to(x.dtype)
    if spectrum == "cmb":
        scale = scale / (math.sqrt(2.0) * (l + 1).to(x.dtype))
    x *= scale[None, :, None]
    x = torch.view_as_complex(x)
    if real:
        sign = (1 - 2 * (m % 2)).to(x.dtype)
        mirror = x[:, l * l + l - m].conj() * sign
        x = torch.where(m > 0, x, torch.where(m < 0, mirror, x.real.to(x.dtype)))
    return x.contiguous()


def _pair(x, L, s):
    """[batch, L*L] spin-s coefficients -> [batch, 2, L*L] with those of the conjugate field."""
    l, m = _degrees(L, x.device)
    sign = (1 - 2 * ((s + m) % 2)).to(x.dtype)
    return torch.stack([x, x[:, l * l + l - m].conj() * sign], 1).contiguous()


def _inputs(case, seed):
    gen = torch.Generator(device=_device())
    gen.manual_seed(seed)
    L, s, batch, double = case["L"], case["s"], case["batch"], case["precision"] == "fp64"
    x = _coeffs(gen, L, s, batch, case["spectrum"], case["real"], double)
    g = None
    if case["kind"] == "gradient":
        # the cotangent that a loss on the samples sends back
        g = torch.randn(batch, L, 2 * L - 1, 2, generator=gen, device=gen.device,
                        dtype=torch.float64 if double else torch.float32)
        g = torch.view_as_complex(g)
    return (_pair(x, L, s) if case["pair"] else x), g


def _members(case):
    rng = np.random.default_rng(case["pick"])
    Ls = rng.choice([int(v) for v in case["Ls"].split(",")], size=case["fields"])
    ss = rng.choice([int(v) for v in case["spins"].split(",")], size=case["fields"])
    return [int(v) for v in Ls], [int(v) for v in ss]


def _group_inputs(case, seed):
    gen = torch.Generator(device=_device())
    gen.manual_seed(seed)
    Ls, ss = _members(case)
    return Ls, ss, [_coeffs(gen, L, s, 1, "flat", False, False)[0] for L, s in zip(Ls, ss)]


def prepare(case, seed):
    if case["kind"] == "group":
        Ls, ss, fields = _group_inputs(case, seed)
        group = ssht.Group(Ls, ss, precision=case["precision"], tune=case["tune"])
        flm = group.pack_coeffs(fields)
        f, back = group.empty_grid(), group.empty_coeffs()
        group.capture(flm, f, back)
        return {"kind": "group", "group": group, "flm": flm, "f": f, "back": back}
    x, g = _inputs(case, seed)
    plan = ssht.Plan(case["L"], case["s"], case["batch"], precision=case["precision"], delta_mode=case["delta_mode"],
                     real=case["real"], spin_pair=case["pair"])
    state = {"kind": case["kind"], "plan": plan, "flm": x, "g": g}
    if case["kind"] == "host":
        state["flm"] = x.cpu().pin_memory()
        state["f"] = torch.empty(plan.grid_shape(), dtype=plan.grid_dtype, device=plan.device)
        state["back"] = torch.empty(plan.coeff_shape(), dtype=plan.dtype, pin_memory=True)
    elif case["kind"] == "gradient":
        state["flm"].requires_grad_(True)
    return state


def run(state):
    if state["kind"] == "group":
        state["group"].replay()
        return {"f": state["f"], "flm": state["back"]}
    plan, flm = state["plan"], state["flm"]
    if state["kind"] == "gradient":
        f = ssht.inverse(flm, plan)
        grad, = torch.autograd.grad(f, flm, state["g"])
        return {"f": f.detach(), "grad": grad}
    if state["kind"] == "host":
        f = plan.inverse(flm, out=state["f"])
        return {"f": f, "flm": plan.forward(f, out=state["back"])}
    f = plan.inverse(flm)
    return {"f": f, "flm": plan.forward(f)}


# ---- what a pass cannot do without ------------------------------------------------------------

def _transform_work(L, batch, elem, recompute, calls=2):
    """Bytes and flops of `calls` transforms of `batch` complex fields (coefficients one way, samples the other)."""
    N = 2 * L - 1
    contraction = 4.0 * batch * sum((2 * l + 1) * (l + 1) for l in range(L))
    dfts = 5.0 * batch * N * math.log2(max(2, N)) * (L + N)
    recursion = 4.0 * L * (L + 1) * (2 * L + 1) / 6 if recompute else 0.0
    return calls * batch * (L * L + L * N) * elem, calls * (contraction + dfts + recursion)


def work(case):
    if case["kind"] == "group":
        Ls, _ = _members(case)
        total = [0.0, 0.0]
        for L in sorted(set(Ls)):
            b, f = _transform_work(L, Ls.count(L), 8, True)
            total[0] += b
            total[1] += f
        return {"bytes": total[0], "flops": total[1]}
    double = case["precision"] == "fp64"
    # a real field is half a complex one, in samples and in independent coefficients
    b, f = _transform_work(case["L"], case["batch"] * (0.5 if case["real"] else 1.0), 16 if double else 8,
                           case["delta_mode"] == "recompute")
    if case["real"]:
        b += 2 * 0.5 * case["batch"] * case["L"] ** 2 * (16 if double else 8)  # coefficients stay complex
    if case["pair"]:
        b += 2 * case["batch"] * case["L"] ** 2 * 8  # the second set of coefficients
    return {"bytes": b, "flops": f}


# ---- the same in 64 bits, by direct sums -------------------------------------------------------

def _wigner_blocks(L, s, device, most_bytes=5e9):
    """Blocks of orders m with d^l_{m,-s}(theta_t), theta_t = pi (2t+1)/(2L-1), as tables [l, m, t].

    The three-term relation in l from the closed form at l = max(|m|, |s|); a value is y 2^e with
    the exponent e <= 0 carried apart while the value is below the FP64 range."""
    N, n = 2 * L - 1, -s
    theta = math.pi * (2 * torch.arange(L, device=device, dtype=torch.float64) + 1) / N
    cos_t = torch.cos(theta)
    half_c, half_s = torch.cos(theta / 2), torch.sin(theta / 2)
    half_c[L - 1] = 0.0  # theta = pi
    log_c, log_s = torch.log2(half_c), torch.log2(half_s)
    per = max(1, min(N, int(most_bytes // (L * L * 8))))
    for first in range(-(L - 1), L, per):
        m = torch.arange(first, min(L, first + per), device=device)
        mf = m.to(torch.float64)
        j = torch.clamp(m.abs(), min=abs(n))
        jf = j.to(torch.float64)
        # d^j at one extreme index: sqrt(C(2j, j + q)) cos^{j+q} sin^{j-q} with a sign
        by_m = m.abs() >= abs(n)
        q = torch.where(by_m, torch.where(m >= 0, n, -n), torch.where(torch.full_like(m, n) >= 0, m, -m))
        odd = torch.where(by_m, torch.where(m >= 0, (j - n) % 2, 0), torch.where(torch.full_like(m, n) >= 0, 0, (j + m) % 2))
        qf = q.to(torch.float64)
        binom = 0.5 * (torch.lgamma(2 * jf + 1) - torch.lgamma(jf + qf + 1) - torch.lgamma(jf - qf + 1)) / math.log(2.0)

        def power(e, logs):  # e * log2, with 0 * -inf = 0
            return torch.where(e[:, None] == 0, torch.zeros((), device=device, dtype=torch.float64), e[:, None] * logs[None, :])

        lg = binom[:, None] + power(jf + qf, log_c) + power(jf - qf, log_s)
        zero = torch.isinf(lg)
        lg = torch.where(zero, torch.zeros_like(lg), lg)
        expo = torch.clamp(torch.floor(lg / 256.0) * 256.0, max=0.0)
        seed = torch.where(zero, torch.zeros_like(lg), torch.exp2(lg - expo)) * (1 - 2 * odd.to(torch.float64))[:, None]
        table = torch.zeros(L, len(m), L, device=device, dtype=torch.float64)
        prev, cur = torch.zeros_like(seed), torch.zeros_like(seed)
        big = 2.0 ** 256
        scale = torch.exp2(expo)
        for l in range(min(L, int(j.min())), L):
            start = j == l
            if l > 0:
                k = l - 1  # from degrees k and k - 1
                up = torch.sqrt(torch.clamp((l * l - mf * mf) * (l * l - n * n), min=0.0))
                down = torch.sqrt(torch.clamp((k * k - mf * mf) * (k * k - n * n), min=0.0))
                live = j < l
                div = torch.where(live, up * max(k, 1), torch.ones_like(up))
                a = torch.where(live, (2 * k + 1) * (k * (k + 1.0) if k else 1.0) / div, torch.zeros_like(up))
                shift = mf * n / (k * (k + 1.0)) if k else torch.zeros_like(mf)
                b = torch.where(live, l * down / div, torch.zeros_like(up))
                nxt = a[:, None] * (cos_t[None, :] - shift[:, None]) * cur - b[:, None] * prev
                prev, cur = cur, nxt
            if bool((l >= int(j.min())) and (l <= int(j.max()))):
                cur = torch.where(start[:, None], seed, cur)
            if l % 16 == 0 or l < int(j.min()) + 2:
                over = (cur.abs() > big) & (expo < 0)
                cur, prev = torch.where(over, cur / big, cur), torch.where(over, prev / big, prev)
                expo = torch.where(over, expo + 256.0, expo)
                scale = torch.exp2(expo)
            torch.mul(cur, scale, out=table[l])
        yield m, table


def _norms(L, device):
    l = torch.arange(L, device=device, dtype=torch.float64)
    return torch.sqrt((2 * l + 1) / (4 * math.pi))


def _synthesis(x, L, s):
    """Samples [B, L, N] of coefficients [B, L*L]."""
    B, N, device = x.shape[0], 2 * L - 1, x.device
    x = x.to(torch.complex128)
    hm = torch.zeros(B, N, L, device=device, dtype=torch.complex128)  # order m at m mod N
    l = torch.arange(L, device=device)
    sign = -1.0 if s % 2 else 1.0
    for m, table in _wigner_blocks(L, s, device):
        ok = (l[None, :] >= m.abs()[:, None]) & (l[None, :] >= abs(s))
        at = torch.where(ok, (l * l + l)[None, :] + m[:, None], torch.zeros_like(l)[None, :])
        v = torch.where(ok, x[:, at], torch.zeros((), device=device, dtype=x.dtype)) * (sign * _norms(L, device))
        v = torch.view_as_real(v).permute(1, 2, 0, 3).reshape(len(m), L, 2 * B)  # [m, l, 2B]
        r = torch.bmm(table.permute(1, 2, 0), v).reshape(len(m), L, B, 2)
        hm[:, m % N] = torch.view_as_complex(r.contiguous()).permute(2, 0, 1)
    phase = torch.arange(N, device=device)
    order = torch.where(phase < L, phase, phase - N).to(torch.float64)
    hm *= torch.polar(torch.ones_like(order), math.pi * order / N)[None, :, None]
    return (torch.fft.ifft(hm, dim=1) * N).permute(0, 2, 1).contiguous()


def _project(hm, L, s):
    """Coefficients sum_t d^l_{m,-s}(theta_t) hm[b, m, t] with the harmonics' norms, [B, L*L]."""
    B, N, device = hm.shape[0], 2 * L - 1, hm.device
    out = torch.zeros(B, L * L, device=device, dtype=torch.complex128)
    l = torch.arange(L, device=device)
    sign = -1.0 if s % 2 else 1.0
    for m, table in _wigner_blocks(L, s, device):
        v = torch.view_as_real(hm[:, m % N].contiguous()).permute(1, 2, 0, 3).reshape(len(m), L, 2 * B)
        r = torch.bmm(table.permute(1, 0, 2), v).reshape(len(m), L, B, 2)
        r = torch.view_as_complex(r.contiguous()) * (sign * _norms(L, device))[None, :, None]
        ok = (l[None, :] >= m.abs()[:, None]) & (l[None, :] >= abs(s))
        at = (l * l + l)[None, :] + m[:, None]
        out[:, at[ok]] = r[ok].permute(1, 0)
    return out


def _adjoint(g, L, s):
    """sum over the samples of g conj(sY_lm)."""
    N = 2 * L - 1
    hm = torch.fft.fft(g.to(torch.complex128), dim=2).permute(0, 2, 1).contiguous()
    k = torch.arange(N, device=g.device)
    order = torch.where(k < L, k, k - N).to(torch.float64)
    return _project(hm * torch.polar(torch.ones_like(order), -math.pi * order / N)[None, :, None], L, s)


def exact(case, seed):
    if case["kind"] == "group":
        Ls, ss, fields = _group_inputs(case, seed)
        # flat buffers in the group's documented order: by L, then s, then the caller's index
        order = sorted(range(len(Ls)), key=lambda i: (Ls[i], ss[i], i))
        f, at = [], 0
        while at < len(order):
            L, s = Ls[order[at]], ss[order[at]]
            same = [i for i in order if (Ls[i], ss[i]) == (L, s)]
            f.append(_synthesis(torch.stack([fields[i] for i in same]), L, s).to(torch.complex128).reshape(-1))
            at += len(same)
        return {"f": torch.cat(f), "flm": torch.cat([fields[i].to(torch.complex128) for i in order])}
    L, s = case["L"], case["s"]
    x, g = _inputs(case, seed)
    f = _synthesis(x[:, 0] if case["pair"] else x, L, s)
    if case["kind"] == "gradient":
        return {"f": f, "grad": _adjoint(g, L, s)}
    # the analysis of a band-limited field gives its coefficients back
    return {"f": f.real.contiguous() if case["real"] else f, "flm": x.to(torch.complex128)}
