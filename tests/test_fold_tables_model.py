"""CPU model of the factors of csrc/paco_fold.cuh: the tables that paco_route.cu
makes (tau_gen_kernel: levels, rows, powers; from a pair of root tables or not), the
places where a pass reads them for F1 and F2 in each of its modes, and the DFT that
comes of them.  And the one-launch form's passes with Phase III's factors taken
after the exchange, as its kernel does."""

import numpy as np
import pytest


def _rev(u, bits):
    r = 0
    for i in range(bits):
        r |= ((u >> i) & 1) << (bits - 1 - i)
    return r


def _tau_index(n, s):
    return 0 if n == 2 else n // 4 + s


def _fold(v, tau):
    """fold_dft with tau(q), q = tau_index(n, s)."""
    R = len(v)
    u = [v[_rev(i, R.bit_length() - 1)] for i in range(R)]
    n = 2
    while n <= R:
        Q = max(1, n // 4)
        for s in range(Q):
            t = tau(_tau_index(n, s))
            for b in range(0, R, n):
                for off, f in [(s, t)] + ([(s + Q, -1j * t)] if n >= 4 else []):
                    e, o = u[b + off], f * u[b + off + n // 2]
                    u[b + off], u[b + off + n // 2] = e + o, e - o
        n *= 2
    return np.array(u)


def _tau_gen(entries, kind, lgA, lgK, roots_lg=None):
    """tau_gen_kernel: entries << lgK places."""
    i = np.arange(entries << lgK)
    kap, q = i & ((1 << lgK) - 1), i >> lgK
    if kind == "levels":
        klo, t = q & ((1 << lgA) - 1), q >> lgA
        lgq = np.array([int(v).bit_length() - 1 if v else 0 for v in t])
        s = np.where(t > 0, t - (1 << lgq), 0)
        e = kap + (klo << lgK) + (s << (lgK + lgA))
        lgM = lgK + lgA + np.where(t > 0, lgq + 2, 1)
    else:
        e = kap * q if kind == "rows" else kap << q
        lgM = np.full_like(e, lgK + lgA)
    if roots_lg is None:
        return np.exp(-2j * np.pi * e / (1 << lgM))
    lo_bits = (roots_lg + 1) // 2
    lo = np.exp(-2j * np.pi * np.arange(1 << lo_bits) / (1 << roots_lg))
    hi = np.exp(-2j * np.pi * (np.arange(1 << (roots_lg - lo_bits)) << lo_bits) / (1 << roots_lg))
    x = e << (roots_lg - lgM)
    assert np.all(roots_lg >= lgM) and np.all(x < 1 << roots_lg)
    return lo[x & ((1 << lo_bits) - 1)] * hi[x >> lo_bits]


def _table(lgA, lgB, lgK, mode, fp64):
    """fold_table, in the order of its launches."""
    A, B = 1 << lgA, 1 << lgB
    nA, lgL = A if fp64 else A // 2, lgA + lgB
    if mode == 0 and (fp64 or lgB < 4):
        return np.exp(-2j * np.pi * np.arange(A * B) / (A * B))
    rt = None if fp64 or mode == 0 else lgK + lgL
    f1 = ("rows", A, lgA) if fp64 else ("levels", nA, 0)
    parts = []
    if mode == 1:
        parts = [_tau_gen(f1[1], f1[0], f1[2], lgK, rt), _tau_gen(A * B // 2, "levels", lgA, lgK, rt)]
    else:
        parts = [_tau_gen(A * B // 2, "levels", lgA, 0)]
        if mode == 2:
            parts += [_tau_gen(f1[1], f1[0], f1[2], lgK, rt), _tau_gen(lgB, "powers", lgL, lgK, rt)]
    return np.concatenate(parts)


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("lgA,lgB,lgK", [(4, 1, 5), (4, 2, 4), (3, 3, 3), (4, 3, 4), (4, 4, 3), (5, 4, 2), (5, 5, 3)])
def test_factors_of_a_pass(lgA, lgB, lgK, mode, fp64):
    A, B, K = 1 << lgA, 1 << lgB, 1 << lgK
    L, nA = A * B, A if fp64 else A // 2
    tau = _table(lgA, lgB, lgK, mode, fp64)
    rng = np.random.default_rng(lgA + 8 * lgB + mode)
    for kap in sorted({0, 1, K // 2, K - 1}):
        x = rng.normal(size=L) + 1j * rng.normal(size=L)
        f1 = {0: None, 1: lambda q: tau[kap + (q << lgK)], 2: lambda q: tau[L // 2 + (q << lgK) + kap]}[mode]
        pow_b = [tau[L // 2 + ((nA + i) << lgK) + kap] for i in range(lgB)] if mode == 2 else None
        ex = np.empty((A, B), complex)                       # [k_lo][j_lo]
        for jlo in range(B):
            v = x[jlo + B * np.arange(A)]
            if mode == 0:
                v = np.fft.fft(v)
                if fp64 or lgB < 4:
                    v = v * np.array([tau[k * jlo] for k in range(A)])
            elif fp64:
                v = np.fft.fft(v * np.array([1.0] + [f1(r) for r in range(1, A)]))
            else:
                v = _fold(list(v), f1)
            ex[:, jlo] = v
        y = np.empty(L, complex)
        for klo in range(A):
            if mode == 0 and (fp64 or lgB < 4):
                y[klo + A * np.arange(B)] = np.fft.fft(ex[klo])
                continue

            def f2(q):
                if mode == 1:
                    return tau[kap + ((nA + klo + q * A) << lgK)]
                w = tau[klo + q * A]
                if mode == 0:
                    return w
                lg, n = 0, 2 if q == 0 else 4 << (q.bit_length() - 1)
                while n << lg < B:
                    lg += 1
                return w * pow_b[lg]

            y[klo + A * np.arange(B)] = _fold(list(ex[klo]), f2)
        t = np.exp(-2j * np.pi * kap * np.arange(L) / (K * L)) if mode else 1.0
        ref = np.fft.fft(x * t)
        assert np.max(np.abs(y - ref)) <= 1e-12 * np.max(np.abs(ref))


@pytest.mark.parametrize("K", [8, 16])
@pytest.mark.parametrize("dims", [1, 2])
def test_one_launch_form_takes_its_factors_after_the_exchange(K, dims):
    """paco_cluster.cu: plain 16 x 16 passes over the input columns, the blocks
    [source][c][v], then folded butterflies over rows j = c whose factors
    (entries 128 on of the plan's table) hold w_N^{-v c}; none in 2-D."""
    L, W = 256, 256 // K
    one = _tau_gen(128, "levels", 4, 0)
    lgK = 8
    two = np.concatenate([_tau_gen(8, "levels", 0, lgK, 16), _tau_gen(128, "levels", 4, lgK, 16)])
    if dims == 2:                                            # kappa = 0 in every column
        two = np.repeat(np.concatenate([_tau_gen(8, "levels", 0, 0), _tau_gen(128, "levels", 4, 0)]), 1 << lgK)
    tab = np.concatenate([one, two])
    rng = np.random.default_rng(4)
    x = rng.normal(size=L * L) + 1j * rng.normal(size=L * L)
    X = x.reshape(L, L)

    def dft256(col, f1, f2):
        ex = np.empty((16, 16), complex)
        for t in range(16):
            v = col[t + 16 * np.arange(16)]
            ex[:, t] = np.fft.fft(v) if f1 is None else _fold(list(v), f1)
        out = np.empty(L, complex)
        for u in range(16):
            out[u + 16 * np.arange(16)] = _fold(list(ex[u]), lambda q: f2(q, u))
        return out

    cols = np.array([dft256(X[:, c], None, lambda q, u: tab[q * 16 + u]) for c in range(L)])      # [c][v]
    blocks = cols.reshape(K, W, K, W).transpose(2, 0, 1, 3)  # [destination][source][c][v]
    Y = np.empty((L, L), complex)
    for r in range(K):
        rows = blocks[r].reshape(L, W)                       # row j = c
        for vl in range(0, W, max(1, W // 4)):
            k1 = r * W + vl
            Y[:, k1] = dft256(rows[:, vl], lambda q: tab[128 + q * L + k1], lambda q, u: tab[128 + (8 + q * 16 + u) * L + k1])
    ref = (np.fft.fft(x).reshape(L, L) if dims == 1 else np.fft.fft2(X).T)
    done = [r * W + vl for r in range(K) for vl in range(0, W, max(1, W // 4))]
    assert np.max(np.abs(Y[:, done] - ref[:, done])) <= 1e-12 * np.max(np.abs(ref))
