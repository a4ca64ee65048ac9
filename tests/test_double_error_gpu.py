"""complex128: the passes of paco_execute are no further from the exact transform
than the stage kernels (which a plan with ctas_per_sm set runs).  The reference is
a long-double FFT, as an FP64 one is no closer than the transforms compared."""

import numpy as np
import pytest

from paco_inputs import uniform

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2609_06449_gb300 as paco  # noqa: E402


def _fft_long(x):
    """Radix-2 decimation in frequency over long doubles, as (re, im)."""
    n = x.size
    re, im = x.real.astype(np.longdouble)[:, None], x.imag.astype(np.longdouble)[:, None]
    pi = np.longdouble("3.14159265358979323846264338327950288")
    order, cur = np.zeros(1, dtype=np.int64), n
    while cur > 1:
        h, m = cur // 2, re.shape[1]
        ang = -2 * pi * np.arange(h, dtype=np.longdouble) / cur
        c, s = np.cos(ang)[:, None], np.sin(ang)[:, None]
        dr, di = re[:h] - re[h:], im[:h] - im[h:]
        re, im = (np.concatenate([re[:h] + re[h:], dr * c - di * s], axis=1),
                  np.concatenate([im[:h] + im[h:], dr * s + di * c], axis=1))
        order, cur = np.concatenate([order, order + n // cur]), h
        assert re.shape == (h, 2 * m)
    out = np.empty((2, n), np.longdouble)
    out[0, order], out[1, order] = re[0], im[0]
    return out


@pytest.mark.parametrize("l1,l2", [(6, 6), (9, 9), (10, 9), (10, 10), (11, 10), (11, 11)])
def test_passes_are_as_close_as_the_stages(l1, l2):
    N = 1 << (l1 + l2)
    x = uniform(N, l1 + 7 * l2, np.complex128)
    re, im = _fft_long(x)
    xt = torch.from_numpy(x).cuda()
    err = []
    for kw in ({}, {"ctas_per_sm": 1}):
        plan = paco.Plan(1 << l1, 1 << l2, 2, 1, paco.C128, **kw)
        assert (plan.info.passes > 0) == (not kw)
        y = torch.empty_like(xt)
        plan.execute(xt, y, -1)
        got = y.cpu().numpy()
        err.append(float(np.sqrt(np.sum((got.real - re) ** 2 + (got.imag - im) ** 2) / np.sum(re ** 2 + im ** 2))))
    print(l1 + l2, "passes %.4g, stages %.4g" % tuple(err))
    assert err[0] <= err[1], err
