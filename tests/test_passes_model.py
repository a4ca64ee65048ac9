"""CPU model of the address maps of csrc/paco_pass.cuh / paco_route.cu: the
passes' row maps (a per-thread term for j_lo plus a launch constant for j_hi),
the redistribution in the first pass's store addresses and the row blocks of
the middle pass, composed over every column to numpy's DFT.  Each pass reads
its whole input before it writes, which the kernel does tile by tile: the test
also checks that a tile writes exactly the places it read."""

import numpy as np
import pytest


def _rev(u, bits, t):
    r = 0
    for d in range(bits // t):
        r = (r << t) | ((u >> (d * t)) & ((1 << t) - 1))
    return r


@pytest.mark.parametrize("f,t,dims", [((3, 4), 1, 1), ((4, 4), 2, 1), ((4, 4), 4, 1), ((3, 3, 3), 1, 1),
                                      ((3, 3, 3), 3, 1), ((4, 3, 2), 1, 1), ((4, 2, 4), 2, 1), ((3, 4), 1, 2),
                                      ((2, 4, 3), 1, 3)])
def test_pass_address_maps(f, t, dims):
    n, lgN = len(f), sum(f)
    N = 1 << lgN
    rng = np.random.default_rng(0)
    x = rng.normal(size=N) + 1j * rng.normal(size=N)
    w = (lambda e: np.exp(-2j * np.pi * (e % N) / N)) if dims == 1 else (lambda e: 1.0)
    out = None
    for i, lgL in enumerate(f):
        L, lgB = 1 << lgL, lgL // 2
        lgC = lgN - lgL if i in (0, n - 1) else f[0]              # columns of a row block, and the row stride
        rb = 0 if i == 0 else lgL
        row_a = [_rev(j << lgB, rb, t) << lgC if rb else (j << lgB) << lgC for j in range(1 << (lgL - lgB))]

        def row(j):
            lo = j & ((1 << lgB) - 1)
            return row_a[j >> lgB] + ((_rev(lo, rb, t) if rb else lo) << lgC)

        src, dst = (x if i == 0 else out), np.full(N, np.nan, complex)
        for blk in range(1 if i in (0, n - 1) else 1 << (lgN - lgL - lgC)):
            for c in range(1 << lgC):
                base = (blk << (f[0] + f[1]) if blk else 0) + c
                read = [base + row(j) for j in range(L)]
                y = np.fft.fft(src[read])
                for k in range(L):
                    if i == 0:
                        v, a = y[k] * w(k * c), _rev(c, lgC, t) * L + k
                    else:
                        v, a = y[k], base + (k << lgC)
                        if i < n - 1:
                            v = v * w(k * _rev(blk, f[2], t) << f[0])
                    assert np.isnan(dst[a].real)
                    dst[a] = v
                if i > 0:
                    assert sorted(read) == sorted(base + (k << lgC) for k in range(L))
        out = dst
    ref = np.fft.fft(x) if dims == 1 else np.fft.fftn(x.reshape([1 << q for q in f])).transpose(range(n)[::-1]).reshape(-1)
    assert np.max(np.abs(out - ref)) <= 1e-13 * np.max(np.abs(ref)) * lgN
