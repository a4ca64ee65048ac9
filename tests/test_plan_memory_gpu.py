"""What a plan holds on the device: nothing for kernels it does not run, until a
call needs them, which may be one that a stream capture records; and one set of
factors for all plans of a length."""

import threading

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


@pytest.mark.parametrize("l1,l2,dtype,one", [(10, 10, paco.C64, 8), (12, 12, paco.C64, 10), (10, 10, paco.C128, 16)])
def test_plans_of_one_length_hold_one_set_of_factors(l1, l2, dtype, one):
    paco.Plan(1 << l1, 1 << l2, 2, 1, dtype).close()
    free = _free()
    plans = [paco.Plan(1 << l1, 1 << l2, 2, batch, dtype) for batch in range(1, 17)]
    assert free - _free() <= (one + 8) * MIB
    for p in plans:
        p.close()
    assert free - _free() <= 2 * MIB


def test_factors_outlive_the_plan_that_made_them():
    """Plans made, run and closed by several threads on streams of their own, in
    any order: each result is that of a plan alone."""
    shapes = [(6, 6), (7, 7), (8, 8), (9, 9), (10, 10), (11, 10)]
    xs = [torch.from_numpy(gaussian(1 << (a + b), a, np.complex64)).cuda() for a, b in shapes]
    want = []
    for (a, b), x in zip(shapes, xs):
        y = torch.empty_like(x)
        paco.Plan(1 << a, 1 << b, 2, 1, paco.C64).execute(x, y)
        want.append(y)
    torch.cuda.synchronize()
    bad = []

    def work(seed):
        rng, stream = np.random.default_rng(seed), torch.cuda.Stream()
        for _ in range(25):
            i = int(rng.integers(len(shapes)))
            a, b = shapes[i]
            plan = paco.Plan(1 << a, 1 << b, 2, 1, paco.C64)
            y = torch.full_like(xs[i], float("nan"))
            torch.cuda.synchronize()
            plan.execute(xs[i], y, -1, stream)
            stream.synchronize()
            if not torch.equal(y, want[i]):
                bad.append((seed, a, b))
            plan.close()

    threads = [threading.Thread(target=work, args=(s,)) for s in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
