"""The stage kernels through their own entry points (paco_execute_stage1, _stage2),
which plans that run as passes in paco_execute reach in no other way: the 2^14
panel pipeline with its ring wrapping and after a wait that gave up, the stages in
two passes, the tensor-core stages.  And the complex128 route of four passes."""

import math

import numpy as np
import pytest

import oracle
from paco_inputs import gaussian, loguniform, uniform

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2609_06449_gb300 as paco  # noqa: E402


def _err(got, ref):
    got = np.asarray(got, dtype=np.complex128).reshape(ref.shape)
    return float(np.max(np.linalg.norm(got - ref, axis=-1) / np.linalg.norm(ref, axis=-1)))


def _stages(plan, x, d=-1):
    xt = torch.from_numpy(x).cuda()
    w = torch.full_like(xt, float("nan"))
    plan.execute_stage1(xt, w, d)
    plan.execute_stage2(w, w, d)
    torch.cuda.synchronize()
    plan.check()
    return w.cpu().numpy()


@pytest.mark.parametrize("N1,N2,b", [(16384, 2048, 2), (2048, 16384, 2), (16384, 4096, 4), (4096, 16384, 4)])
@pytest.mark.parametrize("d", [-1, 1])
def test_panel_ring_wraps_in_the_stages(N1, N2, b, d):
    """16 or 32 panels of 128 columns a transform, batch 2: the three panel buffers
    are used many times over."""
    batch, N = 2, N1 * N2
    x = uniform(batch * N, N1 + 3 * N2 + b, np.complex64).reshape(batch, N)
    plan = paco.Plan(N1, N2, b, batch, paco.C64)
    assert plan.info.passes > 0
    ref = oracle.fft(x.astype(np.complex128), dir=d, threads=0)
    assert _err(_stages(plan, x, d), ref) <= 5e-7 * math.log2(N)


def test_panel_stages_of_the_largest_size():
    """2^14 x 2^14, both stages the panel pipeline: against paco_execute, whose
    result the parity tests compare with the oracle."""
    N = 1 << 28
    plan = paco.Plan(16384, 16384, 4, 1, paco.C64, p=64)
    x = torch.from_numpy(uniform(N, 3, np.complex64)).cuda()
    y, w = torch.empty_like(x), torch.empty_like(x)
    for d in (-1, 1):
        plan.execute(x, y, d)
        plan.execute_stage1(x, w, d)
        plan.execute_stage2(w, w, d)
        torch.cuda.synchronize()
        plan.check()
        err = torch.linalg.vector_norm(w - y) / torch.linalg.vector_norm(y)
        assert err.item() <= 5e-7 * 28


@pytest.mark.parametrize("N1,N2", [(16384, 128), (128, 16384)])
def test_panel_stages_after_a_wait_that_gave_up(N1, N2):
    x = gaussian(N1 * N2, 41, np.complex64).reshape(1, -1)
    plan = paco.Plan(N1, N2, 2, 1, paco.C64)
    xt = torch.from_numpy(x).cuda()
    w = torch.zeros_like(xt)
    plan.debug_set_waits(spin_limit=20000, wait_bias=1)
    plan.execute_stage1(xt, w)
    plan.execute_stage2(w, w)
    torch.cuda.synchronize()
    with pytest.raises(paco.PacoError) as ei:
        plan.check()
    assert ei.value.status == 5                            # PACO_ERR_TIMEOUT
    plan.debug_set_waits(0, 0)
    assert _err(_stages(plan, x), oracle.fft(x.astype(np.complex128))) <= 5e-7 * math.log2(N1 * N2)


@pytest.mark.parametrize("N1,N2,b,batch,split", [
    (4096, 4096, 4, 1, (1, 1)), (4096, 4096, 8, 1, (1, 1)), (8192, 4096, 2, 1, (1, 1)), (4096, 8192, 2, 1, (1, 1)),
    (8192, 256, 2, 3, (1, 0)), (256, 8192, 2, 3, (0, 1)), (4096, 64, 4, 5, (1, 0)), (4096, 4096, 16, 1, (0, 0))])
@pytest.mark.parametrize("d", [-1, 1])
def test_stages_in_two_passes(N1, N2, b, batch, split, d):
    N = N1 * N2
    plan = paco.Plan(N1, N2, b, batch, paco.C64)
    assert tuple(plan.info.stage_split) == split
    x = uniform(batch * N, N1 + 3 * N2 + b, np.complex64).reshape(batch, N)
    ref = oracle.fft(x.astype(np.complex128), dir=d, threads=0)
    assert _err(_stages(plan, x, d), ref) <= 5e-7 * math.log2(N)


@pytest.mark.parametrize("form,tol", [(paco.C64_TC_BF16X3, None), (paco.C64_TC_FP16, 1e-3)])
@pytest.mark.parametrize("N1,N2,b,batch,gen", [(256, 256, 4, 3, uniform), (1024, 256, 4, 2, loguniform),
                                               (256, 4096, 16, 1, uniform), (512, 2048, 2, 1, loguniform),
                                               (4096, 4096, 4, 1, loguniform), (16384, 256, 2, 1, uniform)])
@pytest.mark.parametrize("d", [-1, 1])
def test_tensor_core_stages(N1, N2, b, batch, gen, form, tol, d):
    N = N1 * N2
    plan = paco.Plan(N1, N2, b, batch, form)
    assert plan.info.passes > 0                            # paco_execute runs other kernels
    x = gen(batch * N, N1 + N2 + batch, np.complex64).reshape(batch, N)
    ref = oracle.fft(x.astype(np.complex128), dir=d, threads=0)
    assert _err(_stages(plan, x, d), ref) <= (tol or 5e-7 * math.log2(N))


@pytest.mark.parametrize("d", [-1, 1])
def test_four_double_passes(d):
    """2^28 in complex128: eight points of random size, whose transform is a sum of
    eight tones at every one of the 2^28 results."""
    N = 1 << 28
    plan = paco.Plan(16384, 16384, 2, 1, paco.C128)
    assert plan.info.passes == 4
    rng = np.random.default_rng(7)
    at, size = rng.integers(0, N, 8), rng.normal(size=8) + 1j * rng.normal(size=8)
    x = torch.zeros(N, dtype=torch.complex128, device="cuda")
    x[torch.from_numpy(at).cuda()] = torch.from_numpy(size).cuda()
    y = torch.empty_like(x)
    plan.execute(x, y, d)
    torch.cuda.synchronize()
    num = den = 0.0
    for k0 in range(0, N, 1 << 24):
        k = torch.arange(k0, k0 + (1 << 24), device="cuda")
        ref = torch.zeros(1 << 24, dtype=torch.complex128, device="cuda")
        for p, a in zip(at, size):
            ang = (k * int(p) % N).to(torch.float64) * (d * 2.0 * math.pi / N)
            ref += complex(a) * torch.polar(torch.ones_like(ang), ang)
        num += torch.linalg.vector_norm(y[k0:k0 + (1 << 24)] - ref).item() ** 2
        den += torch.linalg.vector_norm(ref).item() ** 2
    assert math.sqrt(num / den) <= 1e-14 * 28
