"""What a call owes its caller whichever kernels run it: data written by the
kernel just before it in the stream is what it reads, and the scalar of a
weighted input multiplies the input."""

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
