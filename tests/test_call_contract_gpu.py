"""What a call owes its caller whichever kernels run it: data written by the
kernel just before it in the stream is what it reads, the scalar of a weighted
input multiplies the input, and a sum that overflows takes no other one with it."""

import math

import numpy as np
import pytest

import oracle
from paco_inputs import gaussian, weights

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2609_06449_gb300 as paco  # noqa: E402


@pytest.mark.parametrize("l1,l2,batch", [(10, 10, 8), (8, 8, 40), (6, 6, 500)])
def test_weights_and_scale_written_just_before_the_call(l1, l2, batch):
    """The weights and the scalar are rewritten by a kernel right before every
    call, twenty times without waiting; each result is that of a call which
    waited for everything."""
    N = 1 << (l1 + l2)
    plan = paco.Plan(1 << l1, 1 << l2, 2, batch, paco.C64)
    x = torch.from_numpy(gaussian(batch * N, 5, np.complex64).reshape(batch, N)).cuda()
    w0 = torch.from_numpy(weights(batch * N, 6).reshape(batch, N)).cuda()
    w, g = torch.empty_like(w0), torch.empty((), dtype=torch.float64, device="cuda")
    u, gx, loss = torch.empty_like(x), torch.empty_like(x), torch.empty((), dtype=torch.float64, device="cuda")

    def step(k):
        torch.mul(w0, 2.0 ** (k % 5), out=w)
        plan.execute_weighted_power(x, u, w, loss, -1, out_weighted=True)
        g.fill_(2.0 ** -(k % 7))
        plan.execute_weighted_input(u, gx, None, g, 2.0, +1)
        return gx[:: max(1, batch // 2)].clone()

    want = {}
    for k in range(20):
        torch.cuda.synchronize()
        want[k] = step(k)
        torch.cuda.synchronize()
    got = {k: step(k) for k in range(20)}
    torch.cuda.synchronize()
    plan.check()
    for k in range(20):
        assert torch.equal(got[k], want[k]), k


@pytest.mark.parametrize("size,mult,scale", [(1e37, 1e-10, None), (1e37, 0.5, 1e-9), (1e-41, 1e12, None), (1e-41, 4.0, 1e11)])
@pytest.mark.parametrize("l1,l2,batch", [(2, 2, 9), (3, 3, 5), (4, 4, 3), (6, 6, 3), (7, 6, 33), (7, 7, 2), (8, 8, 3), (9, 9, 2), (10, 10, 1),
                                         (11, 11, 1)])
def test_the_scalar_multiplies_the_input(l1, l2, batch, size, mult, scale):
    """Inputs whose sums overflow, or that are subnormal, before they are scaled
    and neither afterwards; bound of the complex64 transform."""
    N = 1 << (l1 + l2)
    x = (gaussian(batch * N, l1 + 5 * l2, np.complex64) * np.float32(size)).astype(np.complex64).reshape(batch, N)
    plan = paco.Plan(1 << l1, 1 << l2, 2, batch, paco.C64)
    xt = torch.from_numpy(x).cuda()
    y = torch.empty_like(xt)
    st = None if scale is None else torch.tensor(scale, dtype=torch.float64, device="cuda")
    plan.execute_weighted_input(xt, y, None, st, mult, -1)
    torch.cuda.synchronize()
    f = np.float32(mult) * np.float32(1.0 if scale is None else scale)
    ref = oracle.fft(x.astype(np.complex128) * float(f), threads=0)
    err = np.linalg.norm(y.cpu().numpy() - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert np.max(err) <= 5e-7 * math.log2(N)


ROUTES = [  # l1, l2, batch, dtype, plan options: whole transforms, two to three passes, the one-launch form, 2-D, 3-D
    (2, 2, 3, paco.C64, {}), (4, 3, 3, paco.C64, {}), (4, 4, 3, paco.C64, {}), (5, 4, 3, paco.C64, {}), (5, 5, 3, paco.C64, {}),
    (6, 5, 3, paco.C64, {}), (6, 6, 3, paco.C64, {}), (7, 6, 33, paco.C64, {}), (7, 7, 33, paco.C64, {}), (7, 6, 1, paco.C64, {}),
    (7, 7, 2, paco.C64, {}), (8, 7, 1, paco.C64, {}), (8, 8, 2, paco.C64, {}), (8, 8, 2, paco.C64, {"p": 4}), (9, 8, 1, paco.C64, {}),
    (9, 9, 1, paco.C64, {}), (10, 9, 1, paco.C64, {}), (10, 10, 1, paco.C64, {}), (11, 10, 1, paco.C64, {}), (12, 12, 1, paco.C64, {}),
    (13, 13, 1, paco.C64, {}), (5, 5, 2, paco.C128, {}), (6, 5, 2, paco.C128, {}), (7, 7, 2, paco.C128, {}), (9, 8, 1, paco.C128, {}),
    (9, 9, 1, paco.C128, {}), (10, 9, 1, paco.C128, {}), (11, 11, 1, paco.C128, {}), (12, 12, 1, paco.C128, {}),
    (8, 7, 2, paco.C64, {"dims": 2}), (9, 10, 1, paco.C64, {"dims": 2}), (6, 12, 1, paco.C64, {"dims": 3, "N3": 64})]


def _plan(l1, l2, batch, dtype, kw):
    n3 = kw.get("N3", 1)
    return paco.Plan(1 << l1, (1 << l2) // n3, 2, batch, dtype, **kw)


@pytest.mark.parametrize("sums", [1, 2, 4])
@pytest.mark.parametrize("l1,l2,batch,dtype,kw", ROUTES)
def test_an_overflowing_sum_leaves_the_other_bins(l1, l2, batch, dtype, kw, sums):
    """A constant input whose bin 0 is 1.2 * sums times the largest number: only
    the sums over N / sums points and more overflow, which are those of ``sums``
    bins; the other bins, whose sums are zero, stay finite and small."""
    N, real = 1 << (l1 + l2), np.float32 if dtype == paco.C64 else np.float64
    c = np.finfo(real).max / N * (1.2 * sums)
    x = np.full((batch, N), c, dtype=np.complex64 if dtype == paco.C64 else np.complex128)
    xt = torch.from_numpy(x).cuda()
    y = torch.empty_like(xt)
    plan = _plan(l1, l2, batch, dtype, kw)
    for d in (-1, 1):
        plan.execute(xt, y, d)
        torch.cuda.synchronize()
        plan.check()
        got = y.cpu().numpy()
        bad = ~(np.isfinite(got.real) & np.isfinite(got.imag))
        assert np.all(bad[:, 0]) and np.all(bad.sum(axis=1) <= sums)
        assert np.max(np.abs(got[~bad]) / np.finfo(real).max) <= (1e-6 if real is np.float32 else 1e-14)


@pytest.mark.parametrize("l1,l2,batch,dtype,kw", [r for r in ROUTES if "dims" not in r[4]])
def test_large_values_that_do_not_overflow(l1, l2, batch, dtype, kw):
    """Results of up to a quarter of the largest number (about), at the bounds of
    ordinary ones."""
    N, f64 = 1 << (l1 + l2), dtype == paco.C128
    x = gaussian(batch * N, l1 + 3 * l2, np.complex128) * (2.0 ** (1019 if f64 else 123) / math.sqrt(N))
    x = x.astype(np.complex128 if f64 else np.complex64).reshape(batch, N)
    xt = torch.from_numpy(x).cuda()
    y = torch.empty_like(xt)
    plan = _plan(l1, l2, batch, dtype, kw)
    for d in (-1, 1):
        plan.execute(xt, y, d)
        torch.cuda.synchronize()
        s = 2.0 ** (-600 if f64 else -64)                        # (norms within the range of a double)
        ref = oracle.fft(x.astype(np.complex128) * s, dir=d, threads=0)
        err = np.linalg.norm(y.cpu().numpy() * s - ref, axis=1) / np.linalg.norm(ref, axis=1)
        assert np.max(err) <= (1e-14 if f64 else 5e-7) * math.log2(N)


def test_uneven_batches_at_the_largest_values():
    lengths = [1 << lg for lg in (4, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16, 17, 18, 19, 20)]
    big = float(np.finfo(np.float32).max)
    x = np.concatenate([np.full(n, big / n * 1.2, np.complex64) for n in lengths])
    z = np.concatenate([(gaussian(n, n % 97, np.complex128) * (2.0 ** 123 / math.sqrt(n))).astype(np.complex64) for n in lengths])
    plan = paco.BatchedPlan(lengths, autotune=False)
    got = []
    for v in (x, z):
        vt = torch.from_numpy(v).cuda()
        y = torch.empty_like(vt)
        plan.execute(vt, y, -1)
        torch.cuda.synchronize()
        plan.check()
        got.append(y.cpu().numpy())
    o = 0
    for n in lengths:
        bad = ~np.isfinite(got[0][o:o + n].real) | ~np.isfinite(got[0][o:o + n].imag)
        assert bad[0] and bad.sum() == 1, n
        ref = oracle.fft(z[o:o + n].astype(np.complex128).reshape(1, n) * 2.0 ** -64)
        err = np.linalg.norm(got[1][o:o + n] * 2.0 ** -64 - ref[0]) / np.linalg.norm(ref)
        assert err <= 5e-7 * math.log2(n), n
        o += n
