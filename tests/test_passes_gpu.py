"""The passes of paco_execute (csrc/paco_fold.cuh, paco_whole.cuh, paco_power.cuh,
paco_route.cu): every length held whole in a CTA, every pass length as first,
middle and last pass, both directions, ragged batches, the 2-D form, and the
stages of the weighted power, whose arithmetic is that of the stage kernels."""

import math

import numpy as np
import pytest

import oracle
import oracle2d
from paco_inputs import gaussian, uniform, weights

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2609_06449_gb300 as paco  # noqa: E402


def _err(got, ref):
    got = np.asarray(got, dtype=np.complex128).reshape(ref.shape)
    return float(np.max(np.linalg.norm(got - ref, axis=-1) / np.linalg.norm(ref, axis=-1)))


def _run(plan, x, d):
    xt = torch.from_numpy(x).cuda()
    y = torch.full_like(xt, float("nan"))
    plan.execute(xt, y, d)
    torch.cuda.synchronize()
    plan.check()
    return y.cpu().numpy()


@pytest.mark.parametrize("d", [-1, 1])
@pytest.mark.parametrize("l1,l2,b,batch,passes", [
    (2, 2, 2, 3000, 1), (3, 2, 2, 1000, 1), (3, 3, 8, 333, 1), (4, 3, 2, 77, 1), (4, 4, 16, 50, 1), (1, 8, 2, 21, 1),
    (5, 5, 2, 9, 1), (5, 6, 2, 5, 1), (6, 6, 8, 7, 1), (7, 6, 2, 3, 2), (7, 6, 2, 33, 1), (7, 7, 2, 5, 2), (7, 7, 2, 33, 1), (8, 7, 2, 3, 2), (8, 8, 16, 17, 2),
    (8, 9, 2, 3, 2), (9, 9, 8, 2, 2), (10, 9, 2, 2, 2), (10, 10, 4, 3, 2), (14, 4, 2, 1, 2), (4, 14, 2, 1, 2),
    (11, 10, 2, 2, 3), (12, 10, 2, 2, 3), (11, 12, 2, 1, 3), (12, 12, 16, 1, 3), (13, 12, 2, 1, 3)])
def test_passes_against_oracle(l1, l2, b, batch, passes, d):
    N = 1 << (l1 + l2)
    plan = paco.Plan(1 << l1, 1 << l2, b, batch, paco.C64)
    assert plan.info.passes == passes
    x = uniform(batch * N, l1 + 31 * l2, np.complex64).reshape(batch, N)
    ref = oracle.fft(x.astype(np.complex128), dir=d, threads=0)
    assert _err(_run(plan, x, d), ref) <= 5e-7 * math.log2(N)


@pytest.mark.parametrize("d", [-1, 1])
@pytest.mark.parametrize("l1,l2,b,batch,passes", [
    (5, 5, 2, 5, 2), (6, 5, 2, 5, 2), (6, 6, 8, 7, 2), (7, 7, 2, 3, 2), (9, 9, 2, 2, 2), (9, 10, 2, 2, 3), (11, 10, 2, 1, 3),
    (12, 12, 4, 1, 3)])
def test_double_passes_against_oracle(l1, l2, b, batch, passes, d):
    N = 1 << (l1 + l2)
    plan = paco.Plan(1 << l1, 1 << l2, b, batch, paco.C128)
    assert plan.info.passes == passes
    x = uniform(batch * N, l1 + 31 * l2, np.complex128).reshape(batch, N)
    ref = oracle.fft(x, dir=d, threads=0)
    assert _err(_run(plan, x, d), ref) <= 1e-14 * math.log2(N)


@pytest.mark.parametrize("d", [-1, 1])
@pytest.mark.parametrize("form,tol", [(paco.C64_TC_BF16X3, None), (paco.C64_TC_FP16, 1e-3)])
@pytest.mark.parametrize("l1,l2,b,batch", [(8, 8, 16, 3), (8, 9, 2, 2), (9, 9, 8, 1), (10, 9, 2, 1), (10, 10, 2, 3),
                                           (11, 10, 2, 1), (11, 11, 2, 1), (12, 11, 2, 1), (12, 12, 4, 1), (13, 12, 2, 1)])
def test_tensor_core_passes(l1, l2, b, batch, form, tol, d):
    """Every length and place of a tensor-core pass (16 x 2, 4, 8, 16; first,
    middle, last; F2 contracted and plain), the forms' own bounds."""
    N = 1 << (l1 + l2)
    plan = paco.Plan(1 << l1, 1 << l2, b, batch, form)
    assert plan.info.passes == (l1 + l2 + 7) // 8
    x = gaussian(batch * N, l1 + 31 * l2, np.complex64).reshape(batch, N)
    ref = oracle.fft(x.astype(np.complex128), dir=d, threads=0)
    assert _err(_run(plan, x, d), ref) <= (tol or 5e-7 * math.log2(N))


@pytest.mark.parametrize("d", [-1, 1])
@pytest.mark.parametrize("l1,l2,b", [(5, 6, 2), (6, 5, 2), (7, 8, 2), (8, 4, 4), (10, 9, 2), (9, 10, 2)])
def test_passes_2d(l1, l2, b, d):
    batch, N1, N2 = 3, 1 << l1, 1 << l2
    plan = paco.Plan(N1, N2, b, batch, paco.C64, dims=2)
    assert plan.info.passes in (0, 2)
    x = gaussian(batch * N1 * N2, l1 + l2, np.complex64).reshape(batch, N1 * N2)
    ref = oracle2d.fft2_transposed(x.astype(np.complex128), N1, N2, d).reshape(batch, -1)
    assert _err(_run(plan, x, d), ref) <= 5e-7 * (l1 + l2)


@pytest.mark.parametrize("l1,l2,b,batch", [(10, 10, 4, 2), (8, 8, 16, 5), (6, 6, 8, 7), (5, 6, 2, 7), (9, 7, 2, 5),
                                           (7, 9, 2, 5), (10, 5, 2, 5), (12, 8, 2, 2), (4, 9, 2, 3), (11, 10, 2, 1)])
def test_weighted_power_keeps_the_stage_arithmetic(l1, l2, b, batch):
    """Spectrum bit by bit, and the 64-bit sum, as the stage kernels give them
    (a plan with ctas_per_sm set runs those)."""
    N = 1 << (l1 + l2)
    x = torch.from_numpy(gaussian(batch * N, 3, np.complex64).reshape(batch, N)).cuda()
    w = torch.from_numpy(weights(batch * N, 4).reshape(batch, N)).cuda()
    res = []
    for kw in ({}, {"ctas_per_sm": 2}):
        plan = paco.Plan(1 << l1, 1 << l2, b, batch, paco.C64, **kw)
        y, loss = torch.empty_like(x), torch.empty((), dtype=torch.float64, device="cuda")
        plan.execute_weighted_power(x, y, w, loss, -1, out_weighted=True)
        torch.cuda.synchronize()
        res.append((y, loss.item()))
    assert torch.equal(res[0][0], res[1][0])
    assert abs(res[0][1] - res[1][1]) <= 1e-13 * abs(res[1][1])
