"""A model of the torus passes' products (csrc/torus_gemm.cu), run on the CPU in FP64.

The model follows the kernels' index arithmetic: the units of every data operand (which unit, row and
64-K block an element lands in), the column tiles and the terms that an epilogue thread combines, and
the plan-time matrices.  Every write is checked against its operand's extent and for exactly-once
coverage; the results are compared with the oracle's inverse, forward and adjoint."""
import numpy as np
import pytest

from oracle import transforms as T


class Shape:
    def __init__(self, L):
        self.L, self.N = L, 2 * L - 1
        self.nI, self.nK, self.nKs = (L + 127) // 128, (L + 31) // 32, 2 * ((L + 63) // 64)
        nE, nO = (L + 1) // 2, L // 2
        self.gE, self.gO = (nE + 63) // 64, (nO + 63) // 64
        self.cE, self.cO = (nE + 31) // 32, (nO + 31) // 32
        self.nT = (L + 63) // 64
        self.G = self.gE + self.gO
        self.nKm = 2 * self.G


class Operand:
    def __init__(self, units, chunks):
        self.x = np.full((units, 128, 32 * chunks), np.nan)
        self.units, self.chunks = units, chunks
        self.written = np.zeros((units, 128, chunks // 2), int)

    def store(self, unit, kb, row, vals):
        assert 0 <= unit < self.units and 0 <= kb < self.chunks // 2 and 0 <= row < 128
        self.x[unit, row, 64 * kb:64 * kb + 64] = vals
        self.written[unit, row, kb] += 1
        assert self.written[unit, row, kb] == 1


def matrices(sh):
    L, N = sh.L, sh.N
    x = np.pi * (2 * np.arange(L) + 1) / N
    k = np.arange(L)
    cosm, sinm = np.cos(np.outer(x, k)), np.sin(np.outer(x, k))  # [node, order]
    sinm[L - 1] = 0.0
    w2 = np.where(k == 0, 1.0, 2.0)
    full = 128 * sh.nI

    def pad(a, ks):
        out = np.zeros((full, 32 * ks))
        out[:a.shape[0], :a.shape[1]] = a
        return out
    perm = np.full(64 * sh.G, -1)
    perm[:(L + 1) // 2] = np.arange(0, L, 2)
    perm[64 * sh.gE:64 * sh.gE + L // 2] = np.arange(1, L, 2)
    cp, sp = np.zeros((L, 64 * sh.G)), np.zeros((L, 64 * sh.G))
    cp[:, perm >= 0], sp[:, perm >= 0] = cosm[:, perm[perm >= 0]], sinm[:, perm[perm >= 0]]
    # the weight matrices by prefix sums over even p >= 0
    p = 2 * np.arange(L)
    pre = np.cumsum((2.0 / (1.0 - p[:, None] ** 2.0)) * np.exp(1j * p[:, None] * x[None, :]), axis=0)  # [q, t]
    up, dn = pre[(L - 1 - k) // 2], pre[(L - 1 + k) // 2]  # [m', t]
    sr, si = up.real + dn.real - 2.0, up.imag - dn.imag
    e = np.exp(1j * np.outer(k, x))
    c = w2[:, None] * 2 * np.pi * np.where(k == L - 1, 1.0, 2.0)[None, :] / (float(N) * N)
    we, wo = c * (e.real * sr - e.imag * si), c * (e.real * si + e.imag * sr)
    wo[:, L - 1] = 0.0
    wo[0] = 0.0
    assert max(np.abs(we).max(), np.abs(wo).max()) < 128.0 / N ** 2
    return {"theta": [pad(cosm * w2, sh.nKs), pad(2 * sinm * (k > 0), sh.nKs)], "phi_inv": [pad(cp, sh.nKm), pad(sp, sh.nKm)],
            "phi_fwd": [pad(cosm.T, sh.nKs), pad(sinm.T, sh.nKs)], "weight": [pad(we, sh.nKs), pad(wo, sh.nKs)],
            "adj": [pad((cosm * w2).T, sh.nKs), pad((2 * sinm * (k > 0)).T, sh.nKs)]}


def cols(A, op, units, chunks):
    """D[row, 256] of one column tile; only the chunks in use enter."""
    K = np.concatenate([np.arange(32 * c, 32 * c + 32) for c in chunks])
    X = np.concatenate([op.x[units[0]], op.x[units[1]]])[:, K]
    used = np.isfinite(X).all(axis=1)  # rows nothing writes: their columns are not used
    return np.where(used[None, :], A[:, K] @ np.where(used[:, None], X, 0.0).T, np.nan)


def order_group(sh, am):
    q = am >> 1
    return (sh.gE if am & 1 else 0) + (q >> 6), q & 63


def group_orders(sh, g):
    cls = 0 if g < sh.gE else 1
    gi = g - sh.gE if cls else g
    am = 2 * (64 * gi + np.arange(64)) + cls
    return cls, am, am < sh.L


def inverse(F, sh, s):
    B, L, N = F.shape[0], sh.L, sh.N
    M = matrices(sh)
    x = Operand(2 * B * sh.G, sh.nKs)
    Fp = np.zeros((B, N, 32 * sh.nKs), complex)
    Fp[:, :, :L] = F
    for b in range(B):
        for m in range(L):
            g, row = order_group(sh, m)
            p, n = Fp[b, L - 1 + m], Fp[b, L - 1 - m] * (m > 0)
            for kb in range(sh.nKs // 2):
                for eo, v in enumerate((p + n, (p - n) * (m > 0))):
                    x.store(2 * (b * sh.G + g), kb, 64 * eo + row, v[64 * kb:64 * kb + 64].real)
                    x.store(2 * (b * sh.G + g) + 1, kb, 64 * eo + row, v[64 * kb:64 * kb + 64].imag)
    y = Operand(2 * B * sh.nT, sh.nKm)
    for j in range(B * sh.G):
        b, g = divmod(j, sh.G)
        cls, am, live = group_orders(sh, g)
        odd = (cls + s) & 1
        D = cols(M["theta"][odd], x, (2 * j, 2 * j + 1), range(sh.nK))
        for cg in range(4):
            part, sg = (1 - (cg >> 1), -1.0 if cg >= 2 else 1.0) if odd else (cg >> 1, 1.0)
            for t in range(64 * sh.nT):  # the rows past L are written too (zeros)
                v = np.where(live, sg * D[t, 64 * cg:64 * cg + 64], 0.0)
                y.store(2 * (b * sh.nT + (t >> 6)) + (cg & 1), g, 64 * part + (t & 63), v)
    f = np.full((B, L, N), np.nan, complex)
    used = list(range(sh.cE)) + [2 * sh.gE + c for c in range(sh.cO)]
    for j in range(B * sh.nT):
        b, tg = divmod(j, sh.nT)
        E = cols(M["phi_inv"][0], y, (2 * j, 2 * j), used)[:, :128]
        O = cols(M["phi_inv"][1], y, (2 * j + 1, 2 * j + 1), used)[:, :128]
        for k in range(64):
            t = 64 * tg + k
            if t < L:
                a, c = E[:L, k] + 1j * E[:L, 64 + k], O[:L, k] + 1j * O[:L, 64 + k]
                f[b, t, :L] = a + 1j * c
                f[b, t, N - 1 - np.arange(L - 1)] = (a - 1j * c)[:L - 1]
    assert np.isfinite(f).all()
    return f


def analysis(f, sh, s, adjoint):
    """H[b][m + Lp][m'] of the projection."""
    B, L, N = f.shape[0], sh.L, sh.N
    M = matrices(sh)
    per = B * sh.nT
    x = Operand(2 * per, sh.nKs)
    for b in range(B):
        for t in range(L):
            e, d = np.zeros(32 * sh.nKs, complex), np.zeros(32 * sh.nKs, complex)
            mir = f[b, t, N - 1 - np.arange(L)]
            e[:L], d[:L] = f[b, t, :L] + mir, f[b, t, :L] - mir
            e[L - 1], d[L - 1] = f[b, t, L - 1], 0.0
            u, row = b * sh.nT + (t >> 6), t & 63
            for kb in range(sh.nKs // 2):
                sl = slice(64 * kb, 64 * kb + 64)
                x.store(u, kb, row, e[sl].real)
                x.store(u, kb, 64 + row, e[sl].imag)
                x.store(per + u, kb, row, d[sl].real)
                x.store(per + u, kb, 64 + row, d[sl].imag)
    y = Operand(2 * B * sh.G, sh.nKs)
    pairs = (per + 1) // 2
    for j in range(2 * pairs):
        eo = 0 if j < pairs else 1
        pr = j - eo * pairs
        u0 = eo * per + 2 * pr
        u1 = u0 + 1 if 2 * pr + 1 < per else u0
        D = cols(M["phi_fwd"][eo], x, (u0, u1), range(sh.nK))
        for cg in range(4):
            if cg >= 2 and u1 == u0:
                continue
            b, tg = divmod((u1 if cg >= 2 else u0) - eo * per, sh.nT)
            live = np.arange(64) < L - 64 * tg
            for row0 in range(0, 128 * sh.nI, 32):  # a warp's 32 orders: 16 rows of an even and of an odd group
                q0 = row0 >> 1
                for lane in range(32):
                    odd = lane & 1
                    if (q0 >> 6) >= (sh.gO if odd else sh.gE):
                        continue
                    g = (q0 >> 6) + (sh.gE if odd else 0)
                    y.store(2 * (b * sh.G + g) + eo, tg, 64 * (cg & 1) + (q0 & 63) + (lane >> 1),
                            np.where(live, D[row0 + lane, 64 * cg:64 * cg + 64], 0.0))
    H = np.full((B, N, L), np.nan, complex)
    for j in range(B * sh.G):
        b, g = divmod(j, sh.G)
        cls, am, live = group_orders(sh, g)
        odd = (cls + s) & 1
        D = cols(M["adj" if adjoint else "weight"][odd], y, (2 * j, 2 * j + 1), range(sh.nK))[:L]
        for cg in range(4):
            for k in range(16):
                m = am[16 * cg + k]
                if m >= L:
                    break
                P = D[:, 16 * cg + k] + 1j * D[:, 64 + 16 * cg + k]
                Q = D[:, 128 + 16 * cg + k] + 1j * D[:, 192 + 16 * cg + k]
                ph = -1j if odd else 1.0
                H[b, m + L - 1] = ph * (P - 1j * Q)
                if m > 0:
                    H[b, L - 1 - m] = ph * (P + 1j * Q)
    assert np.isfinite(H).all()
    return H


def spin_products(L, s):
    """A[l][m'][m] = sqrt((2l+1)/4pi) Delta^l_{m',-s} Delta^l_{m'm} for m' >= 0, all m, and the phases."""
    for l in range(abs(s), L):
        D = T.wigner_full(2 * l)
        yield l, np.sqrt((2 * l + 1) / (4 * np.pi)) * D[l:, l - s][:, None] * D[l:, :]


def rel(a, b):
    return np.abs(a - b).max() / np.abs(b).max()


@pytest.mark.parametrize("L,s,B", [(1, 0, 2), (2, 1, 1), (3, 0, 3), (5, -2, 1), (33, 2, 2), (64, 0, 1), (65, 1, 3), (129, -1, 1),
                                   (130, 0, 1)])
def test_products_match_oracle(L, s, B):
    rng = np.random.default_rng(L)
    sh = Shape(L)
    flm = rng.standard_normal((B, L * L)) + 1j * rng.standard_normal((B, L * L))
    flm[:, :s * s] = 0.0
    F = np.zeros((B, sh.N, L), complex)
    m = np.arange(-(L - 1), L)
    for l, A in spin_products(L, s):
        F[:, L - 1 - l:L + l, :l + 1] += flm[:, None, l * l:(l + 1) ** 2].transpose(0, 2, 1) * A.T[None]
    F *= ((-1.0) ** s * (1j) ** (-(m + s)))[None, :, None]
    f = inverse(F, sh, s)
    assert rel(f, T.inverse(flm, L, s)) < 1e-12
    g = rng.standard_normal(f.shape) + 1j * rng.standard_normal(f.shape)
    for adjoint, ref in ((0, T.forward(g, L, s)), (1, T.adjoint(g, L, s))):
        H = analysis(g, sh, s, adjoint)
        out = np.zeros((B, L * L), complex)
        for l, A in spin_products(L, s):
            mm = np.arange(-l, l + 1)
            out[:, l * l:(l + 1) ** 2] = np.einsum("km,bmk->bm", A, H[:, L - 1 - l:L + l, :l + 1]) * ((-1.0) ** s * (1j) ** (mm + s))
        assert rel(out, ref) < 1e-12
