"""CPU model of the address maps of csrc/paco_fold.cuh / paco_route.cu: the
passes' row maps (a per-thread term for j_lo plus a launch constant for j_hi),
the redistribution in the first pass's store addresses, the row blocks of the
later passes and the twiddles w_{K L}^{-kappa j} folded into their butterflies
(kappa = column), composed over every column to numpy's DFT.  Each pass reads
its whole input before it writes, which the kernel does tile by tile: the test
also checks that a tile writes exactly the places it read.  A second test
models one folded butterfly network with the kernel's twiddle list."""

import numpy as np
import pytest


def _rev(u, bits, t):
    r = 0
    for d in range(bits // t):
        r = (r << t) | ((u >> (d * t)) & ((1 << t) - 1))
    return r


@pytest.mark.parametrize("f,t,dims", [((3, 4), 1, 1), ((4, 4), 2, 1), ((4, 4), 4, 1), ((3, 3, 3), 1, 1),
                                      ((3, 3, 3), 3, 1), ((4, 3, 2), 1, 1), ((4, 2, 4), 2, 1), ((3, 3, 2, 2), 1, 1),
                                      ((2, 2, 2, 2), 2, 1), ((3, 4), 1, 2), ((2, 4, 3), 1, 3)])
def test_pass_address_maps(f, t, dims):
    n, lgN = len(f), sum(f)
    N = 1 << lgN
    rng = np.random.default_rng(0)
    x = rng.normal(size=N) + 1j * rng.normal(size=N)
    out, lgK = None, 0
    for i, lgL in enumerate(f):
        L, lgB = 1 << lgL, lgL // 2
        lgC = lgN - lgL if i == 0 else lgK                        # columns of a row block, and the row stride
        rb = 0 if i == 0 else lgL
        row_a = [(_rev(j << lgB, rb, t) if rb else j << lgB) << lgC for j in range(1 << (lgL - lgB))]

        def row(j):
            lo = j & ((1 << lgB) - 1)
            return row_a[j >> lgB] + ((_rev(lo, rb, t) if rb else lo) << lgC)

        src, dst = (x if i == 0 else out), np.full(N, np.nan, complex)
        for blk in range(1 << (lgN - lgL - lgC)):
            for c in range(1 << lgC):
                base = (blk << (lgK + lgL)) + c
                read = [base + row(j) for j in range(L)]
                tw = np.exp(-2j * np.pi * c * np.arange(L) / (L << lgK)) if i > 0 and dims == 1 else 1.0
                y = np.fft.fft(src[read] * tw)
                for k in range(L):
                    a = _rev(c, lgC, t) * L + k if i == 0 else base + (k << lgC)
                    assert np.isnan(dst[a].real)
                    dst[a] = y[k]
                if i > 0:
                    assert sorted(read) == sorted(base + (k << lgC) for k in range(L))
        out, lgK = dst, lgK + lgL
    ref = np.fft.fft(x) if dims == 1 else np.fft.fftn(x.reshape([1 << q for q in f])).transpose(range(n)[::-1]).reshape(-1)
    assert np.max(np.abs(out - ref)) <= 1e-13 * np.max(np.abs(ref)) * lgN


def _fold(v, tau):
    """fold_dft: bit-reversed input, levels n = 2, 4, .., with one twiddle per
    pair of butterflies (the second one of the pair takes -i times it)."""
    R = len(v)
    lg = R.bit_length() - 1
    u = [v[_rev(i, lg, 1)] for i in range(R)]
    n = 2
    while n <= R:
        q = max(1, n // 4)
        for s in range(q):
            for b in range(0, R, n):
                for off, t in [(s, tau(n, s))] + ([(s + q, -1j * tau(n, s))] if n >= 4 else []):
                    e, o = u[b + off], t * u[b + off + n // 2]
                    u[b + off], u[b + off + n // 2] = e + o, e - o
        n *= 2
    return np.array(u)


@pytest.mark.parametrize("lgA,lgB,lgK,lgN", [(4, 1, 6, 11), (3, 3, 5, 12), (4, 3, 7, 14), (5, 4, 3, 15), (5, 5, 2, 12)])
def test_folded_twiddles(lgA, lgB, lgK, lgN):
    """Both halves of a pass: the columns' list (as the kernel inverts its
    index), w_{K L}^{-kappa 2^i} times w_L^{-(k_lo + s A) 2^i}, and the result."""
    A, B, K, N = 1 << lgA, 1 << lgB, 1 << lgK, 1 << lgN
    L = A * B
    w = lambda m, e: np.exp(-2j * np.pi * e / m)  # noqa: E731
    rng = np.random.default_rng(1)
    for kap in {0, 1, K // 2, K - 1}:
        x = rng.normal(size=L) + 1j * rng.normal(size=L)
        lst, sizes = [], []
        for i in range(max(1, A // 2)):
            left = A // 2 - 1 - i
            lgq = left.bit_length() - 1 if left else 0
            lgn, s = (lgq + 2, (2 << lgq) - 1 - left) if left else (1, 0)
            e = ((kap + (s << lgK)) << (lgA - lgn)) << (lgN - lgK - lgA)
            assert 0 <= e < N
            lst.append(w(N, e))
            sizes.append((1 << lgn, s))
        index = {}
        n, i = A, 0
        while n >= 2:
            for s in range(max(1, n // 4)):
                index[n, s] = i
                i += 1
            n //= 2
        assert [index[z] for z in sizes] == list(range(len(sizes)))
        F1 = np.array([_fold([x[r * B + jlo] for r in range(A)], lambda n, s: lst[index[n, s]]) for jlo in range(B)])
        y = np.empty(L, complex)
        for klo in range(A):
            def tau(n, s):
                lg = (B // n).bit_length() - 1
                return w(L, (klo + s * A) * (B // n)) * w(N, (kap << lg) << (lgN - lgK - lgA - lgB))
            y[klo + A * np.arange(B)] = _fold(list(F1[:, klo]), tau)
        ref = np.fft.fft(x * w(K * L, kap * np.arange(L)))
        assert np.max(np.abs(y - ref)) <= 1e-12 * np.max(np.abs(ref))


@pytest.mark.parametrize("lg", range(4, 15))
def test_whole_transform_exchanges(lg):
    """paco_whole.cuh: the chain of register steps and exchanges -- every place
    in bounds and written once, at most two points of a half-warp in one bank
    (one from 2^6 points on, 2^9 aside), and the DFT as the result."""
    table = [[4, 4], [8, 4], [8, 8], [8, 16], [16, 16], [8, 8, 8], [16, 8, 8], [16, 16, 8], [16, 16, 16],
             [32, 16, 16], [32, 32, 16]]
    R, N = table[lg - 4], 1 << lg
    ept, nt = (16, 256) if lg <= 12 else (32, 256) if lg == 13 else (32, 512)
    G, K = ept * nt // N, [1]
    for r in R:
        K.append(K[-1] * r)

    def gs(i):
        b = N // K[i + 1] * (K[i + 1] + 1)
        return (b + 7) // 16 * 16 + 8 if K[i + 1] < 16 else b

    size = max(G * gs(i) for i in range(len(R) - 1))
    assert size * 8 <= 227 * 1024
    rng = np.random.default_rng(0)
    x = rng.normal(size=(G, N)) + 1j * rng.normal(size=(G, N))
    buf, out, conflicts = None, np.full((G, N), np.nan, complex), 0

    def banks(ad):
        return max(int(np.bincount(ad[h:h + 16, 0] % 16).max()) for h in range(0, len(ad), 16))

    for i, r in enumerate(R):
        sq, j = N // r, N // r // K[i]
        s, rr = np.arange(G * N // r), np.arange(r)
        g, idx = s // sq, s % sq
        kap, jlo = idx % K[i], idx // K[i]
        if i == 0:
            v = x[g[:, None], idx[:, None] + rr * sq]
        else:
            ad = (g * gs(i - 1) + kap + (K[i] + 1) * jlo)[:, None] + (K[i] + 1) * j * rr
            conflicts = max(conflicts, banks(ad))
            v = buf[ad]
        y = np.fft.fft(v * np.exp(-2j * np.pi * kap[:, None] * rr / (K[i] * r)), axis=1)
        if i < len(R) - 1:
            ad = (g * gs(i) + kap + (K[i] * r + 1) * jlo)[:, None] + K[i] * rr
            assert ad.max() < size and len(np.unique(ad)) == ad.size
            conflicts = max(conflicts, banks(ad))
            buf = np.full(size, np.nan, complex)
            buf[ad] = y
        else:
            out[g[:, None], kap[:, None] + K[i] * rr] = y
    ref = np.fft.fft(x, axis=1)
    assert np.max(np.abs(out - ref)) <= 1e-13 * np.max(np.abs(ref))
    assert conflicts <= (1 if lg >= 6 and lg != 9 else 2)


@pytest.mark.parametrize("K", [8, 16])
def test_cluster_block_exchange(K):
    """paco_cluster.cu: CTA q's results in [destination][c][v] blocks, one copy a
    pair of CTAs into [source][c][v], Phase III over rows j = c -- every place
    written once, runs of 16 places a half-warp, and the DFT as the result."""
    L, W = 256, 256 // K
    rng = np.random.default_rng(2)
    x = rng.normal(size=L * L) + 1j * rng.normal(size=L * L)
    X = x.reshape(L, L)
    tid = np.arange(4096 // K)
    send = np.full((K, K * W * W), np.nan, complex)
    for q in range(K):
        col_b, t_b = tid // 16, tid % 16
        A = np.fft.fft(X[:, q * W + col_b], axis=0)               # [v][thread]
        for k in range(16):
            v = t_b + 16 * k
            place = ((v // W) * W + col_b) * W + v % W
            assert all(len(set(place[h:h + 16] % 16)) == 16 for h in range(0, len(tid), 16))
            assert np.all(np.isnan(send[q, place].real))
            send[q, place] = A[v, tid] * np.exp(-2j * np.pi * v * (q * W + col_b) / L ** 2)
    assert not np.any(np.isnan(send.real))
    recv = send.reshape(K, K, W * W).transpose(1, 0, 2).reshape(K, K * W * W)
    y = np.empty((L, L), complex)                                 # [k2][k1]
    for q in range(K):
        vl, u = tid % W, tid // W
        cols = np.empty((L, W), complex)
        for s in range(16):
            place = (u + 16 * s) * W + vl
            assert all(len(set(place[h:h + 16] % 16)) == 16 for h in range(0, len(tid), 16))
            cols[u + 16 * s, vl] = recv[q, place]
        y[:, q * W:(q + 1) * W] = np.fft.fft(cols, axis=0)
    ref = np.fft.fft(x)
    assert np.max(np.abs(y.reshape(-1) - ref)) <= 1e-12 * np.max(np.abs(ref))
