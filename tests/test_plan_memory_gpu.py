"""What a plan holds on the device: nothing for kernels it does not run, until a
call needs them, which may be one that a stream capture records."""

import numpy as np
import pytest

from paco_inputs import gaussian

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2609_06449_gb300 as paco  # noqa: E402

MIB = 1 << 20


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("N1,N2,b,batch,kw,scratch", [
    (4096, 4096, 4, 16, {}, 2048), (16384, 2048, 2, 1, {}, 48), (64, 64, 2, 64, {"dims": 3, "N3": 64}, 128)])
def test_stage_scratch_comes_with_the_first_stage_call(N1, N2, b, batch, kw, scratch):
    N = N1 * N2 * kw.get("N3", 1)
    x = torch.zeros(batch, N, dtype=torch.complex64, device="cuda")
    y = torch.empty_like(x)
    paco.Plan(N1, N2, b, batch, paco.C64, **kw).execute(x, y)    # (module loading aside)
    free = _free()
    plan = paco.Plan(N1, N2, b, batch, paco.C64, **kw)
    assert plan.info.passes > 0
    plan.execute(x, y)
    assert free - _free() <= 24 * MIB
    plan.execute_stage1(x, y)
    assert free - _free() >= scratch * MIB
    plan.close()
    assert free - _free() <= 8 * MIB


@pytest.mark.parametrize("N1,N2,b,kw", [(4096, 4096, 4, {}), (16384, 2048, 2, {}), (256, 8192, 2, {}),
                                        (64, 64, 2, {"dims": 3, "N3": 64})])
def test_first_stage_calls_inside_a_capture(N1, N2, b, kw):
    N = N1 * N2 * kw.get("N3", 1)
    x = torch.from_numpy(gaussian(N, 17, np.complex64)).cuda()
    ys, plans = [], [paco.Plan(N1, N2, b, 1, paco.C64, **kw) for _ in range(2)]
    for captured, plan in enumerate(plans):
        w, y = torch.empty_like(x), torch.zeros_like(x)
        torch.cuda.synchronize()
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                plan.execute_stage1(x, w)
                plan.execute_stage2(w, y)
            g.replay()
        else:
            plan.execute_stage1(x, w)
            plan.execute_stage2(w, y)
        torch.cuda.synchronize()
        plan.check()
        ys.append(y)
    assert torch.count_nonzero(ys[0]) > 0 and torch.equal(ys[0], ys[1])
