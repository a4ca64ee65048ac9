"""The work that a user of this framework has it do, as cases that can be timed.

Every case goes through the package's public entry points (``Plan``,
``BatchedPlan``, ``PacoFFT``, ``fft``, ``fft2``, ``fft3``,
``weighted_power_loss``).  Sizes come from the benchmark's workloads (the
2^16, 2^28, 16 x 2^24, 256 x 2^20, uneven and 64 x 256 x 64 x 64 ones), from
the parity tests, or are the generic sizes between them; batches that are not
powers of two stand for what a caller's data happens to hold.

A case is a dict of plain values; ``kind`` says which entry point it takes:

* ``plan``    one ``Plan.execute`` into a buffer the caller keeps;
* ``grad``    ``PacoFFT`` forward and backward (a layer inside a model);
* ``loss``    ``weighted_power_loss`` forward and backward (a training step);
* ``uneven``  one ``BatchedPlan.execute`` over transforms of many lengths;
* ``fft2`` / ``fft3``  the functional 2-D and 3-D forms.
"""

from __future__ import annotations

import random

import torch

import paper_2609_06449_gb300 as paco

_DTYPES = {"c64": paco.C64, "c128": paco.C128, "bf16x3": paco.C64_TC_BF16X3, "fp16": paco.C64_TC_FP16}


def listed():
    return [
        # one short transform: a filter or a spectrum inside a real-time loop,
        # where launches and latency are all there is
        dict(name="one_64k", kind="plan", lg1=8, lg2=8, b=2, p=4, batch=1, dtype="c64", dir=-1, dist="uniform"),
        # one transform of a million points, backwards
        dict(name="one_1m_inverse", kind="plan", lg1=10, lg2=10, b=4, p=0, batch=1, dtype="c64", dir=1,
             dist="normal"),
        # many short rows, a count that divides nothing, as a layer of a model
        # (forward and the gradient)
        dict(name="rows_4k_layer", kind="grad", lg1=6, lg2=6, b=4, p=0, batch=3001, dtype="c64", dir=-1,
             dist="normal"),
        # a few rows of medium length, factors of different size
        dict(name="rows_256k", kind="plan", lg1=10, lg2=8, b=4, p=0, batch=77, dtype="c64", dir=-1, dist="uniform"),
        # the long batched rows whose magnitudes span eight decades
        dict(name="rows_16m", kind="plan", lg1=12, lg2=12, b=4, p=0, batch=16, dtype="c64", dir=-1, dist="loguniform"),
        # the headline: one transform of 2^28 points
        dict(name="one_256m", kind="plan", lg1=14, lg2=14, b=4, p=64, batch=1, dtype="c64", dir=-1, dist="uniform"),
        # the double-precision form at the size it is quoted on
        dict(name="one_128m_double", kind="plan", lg1=13, lg2=14, b=2, p=0, batch=1, dtype="c128", dir=-1,
             dist="uniform"),
        # the split-precision tensor-core form
        dict(name="rows_4m_bf16x3", kind="plan", lg1=12, lg2=10, b=2, p=0, batch=6, dtype="bf16x3", dir=-1,
             dist="loguniform"),
        # thousands of transforms of uneven length in one launch, with a
        # regular part of 4096-point ones
        dict(name="uneven", kind="uneven", count=1024, lg_min=8, lg_max=18, regular=4096, regular_lg=12, dir=-1),
        # a training step: weighted power of the spectrum and its gradient
        dict(name="loss_256x1m", kind="loss", lg1=10, lg2=10, b=4, p=0, batch=256),
        # images
        dict(name="images_1024", kind="fft2", lg1=10, lg2=10, b=4, batch=23, dtype="c64", dir=-1),
        # volumes
        dict(name="volumes_256x64x64", kind="fft3", lg1=8, lg2=6, lg3=6, b=2, batch=64, dtype="c64", dir=-1),
    ]


def draw(rng: random.Random):
    """One more case: the kinds as often as they are listed, sizes spread over
    the logarithm of the whole range, odd batches among them."""
    kind = rng.choice(["plan"] * 6 + ["grad", "grad", "loss", "uneven", "fft2", "fft3"])
    if kind == "uneven":
        return dict(kind=kind, count=int(2 ** rng.uniform(5, 10)), lg_min=rng.randint(4, 10),
                    lg_max=rng.randint(12, 18), regular=rng.choice([0, int(2 ** rng.uniform(6, 12))]),
                    regular_lg=rng.randint(8, 13), dir=rng.choice([-1, 1]))
    if kind == "fft3":
        lg2, lg3 = rng.randint(5, 7), rng.randint(5, 7)
        lg1 = rng.randint(4, 9)
        lgb = rng.uniform(0, 26 - lg1 - lg2 - lg3)
        return dict(kind=kind, lg1=lg1, lg2=lg2, lg3=lg3, b=2, batch=max(1, int(2 ** lgb)), dtype="c64",
                    dir=rng.choice([-1, 1]))
    if kind == "fft2":
        lg1, lg2 = rng.randint(5, 11), rng.randint(5, 11)
        lgb = rng.uniform(0, max(0.0, 26 - lg1 - lg2))
        return dict(kind=kind, lg1=lg1, lg2=lg2, b=2, batch=max(1, int(2 ** lgb)),
                    dtype=rng.choice(["c64", "c64", "c64", "c128"]), dir=rng.choice([-1, 1]))
    if kind == "loss":
        lg1, lg2 = rng.randint(6, 12), rng.randint(6, 12)
        lgb = rng.uniform(0, max(0.0, 27 - lg1 - lg2))
        return dict(kind=kind, lg1=lg1, lg2=lg2, b=2, p=0, batch=max(1, int(2 ** lgb)))
    if kind == "grad":
        lg1, lg2 = rng.randint(4, 12), rng.randint(4, 12)
        lgb = rng.uniform(0, max(0.0, 26 - lg1 - lg2))
        return dict(kind=kind, lg1=lg1, lg2=lg2, b=2, p=0, batch=max(1, int(2 ** lgb)),
                    dtype=rng.choice(["c64", "c64", "c64", "c128"]), dir=-1, dist="normal")
    dtype = rng.choice(["c64"] * 7 + ["c128", "c128", "bf16x3", "fp16"])
    lg1, lg2 = rng.randint(8, 14), rng.randint(8, 14)
    if rng.random() < 0.3:                                   # a plan with a larger radix
        b = rng.choice([4, 16])
        t = 2 if b == 4 else 4
        lg1, lg2 = max(8, lg1 // t * t), max(8, lg2 // t * t)
    else:
        b = 2
    if dtype != "c64":
        lg2 = min(lg2, 8 if lg1 == 14 else 12)
    lgb = rng.uniform(0, max(0.0, (28 if dtype == "c64" else 24) - lg1 - lg2))
    return dict(kind="plan", lg1=lg1, lg2=lg2, b=b, p=0, batch=max(1, int(2 ** lgb)), dtype=dtype,
                dir=rng.choice([-1, 1]), dist=rng.choice(["uniform", "normal", "loguniform"]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _values(shape, dist, double, gen):
    """Complex inputs: U[-1, 1) or N(0, 1) parts, or magnitudes 10^U[-4, 4)
    with uniform phase (the precision workload)."""
    rdt = torch.float64 if double else torch.float32
    cdt = torch.complex128 if double else torch.complex64
    x = torch.empty(shape, dtype=cdt, device="cuda")
    r = torch.view_as_real(x)
    if dist == "normal":
        r.normal_(generator=gen)
    elif dist == "uniform":
        r.uniform_(-1.0, 1.0, generator=gen)
    else:
        mag = torch.empty(shape, dtype=rdt, device="cuda").uniform_(-4.0, 4.0, generator=gen)
        mag = torch.pow(10.0, mag)
        ph = torch.empty(shape, dtype=rdt, device="cuda").uniform_(0.0, 6.283185307179586, generator=gen)
        x.copy_(torch.polar(mag, ph))
    return x


def _lengths(case):
    """The uneven workload's lengths: exponents uniform over the range, the
    same for every seed (a caller's data changes, its plan's shape does not),
    with the regular part after them."""
    rng = random.Random(1234)
    lens = [1 << rng.randint(case["lg_min"], case["lg_max"]) for _ in range(case["count"])]
    return lens + [1 << case["regular_lg"]] * case["regular"]


def _elems(case):
    if case["kind"] == "uneven":
        return sum(_lengths(case))
    return case["batch"] << (case["lg1"] + case["lg2"] + case.get("lg3", 0))


def _inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    n = _elems(case)
    if kind == "uneven":
        return dict(x=_values((n,), "normal", False, gen))
    rows = (case["batch"], n // case["batch"])
    double = case.get("dtype") == "c128"
    d = dict(x=_values(rows, case.get("dist", "normal"), double, gen))
    if kind == "loss":
        d["w"] = torch.empty(rows, dtype=torch.float32, device="cuda").uniform_(0.0, 1.0, generator=gen)
    if kind == "grad":
        d["g"] = _values(rows, "normal", double, gen)
    return d


def prepare(case, seed):
    state = _inputs(case, seed)
    state["case"] = case
    kind = case["kind"]
    if kind == "plan":
        state["plan"] = paco.Plan(1 << case["lg1"], 1 << case["lg2"], case["b"], case["batch"],
                                  _DTYPES[case["dtype"]], p=case["p"])
        state["y"] = torch.empty_like(state["x"])
    elif kind == "uneven":
        state["plan"] = paco.BatchedPlan(_lengths(case))
        state["y"] = torch.empty_like(state["x"])
    elif kind in ("loss", "grad"):
        state["x"].requires_grad_(True)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    x = state["x"]
    if kind in ("plan", "uneven"):
        state["plan"].execute(x, state["y"], case["dir"])
        return state["y"]
    N1, N2, b = 1 << case["lg1"], 1 << case["lg2"], case["b"]
    if kind == "fft2":
        return paco.fft2(x, N1, N2, b, dir=case["dir"])
    if kind == "fft3":
        return paco.fft3(x, N1, N2, 1 << case["lg3"], b, dir=case["dir"])
    if kind == "grad":
        y = paco.PacoFFT.apply(x, N1, N2, b, case["p"])
        (gx,) = torch.autograd.grad(y, x, state["g"])
        return y.detach(), gx
    loss = paco.weighted_power_loss(x, state["w"], N1, N2, b, case["p"])
    (gx,) = torch.autograd.grad(loss, x)
    return loss.detach(), gx


def _dft(x, direction):
    """The unnormalised DFT of the last dimension, in 64 bits."""
    if direction == -1:
        return torch.fft.fft(x.to(torch.complex128))
    return torch.fft.ifft(x.to(torch.complex128), norm="forward")


def exact(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    x = d.pop("x")
    if kind == "plan":
        return _dft(x, case["dir"])
    if kind == "grad":
        return _dft(x, -1), _dft(d["g"], 1)
    if kind == "loss":
        # in blocks of rows: the whole batch in 64 bits is many times the inputs
        w, loss, gx = d["w"], torch.zeros((), dtype=torch.float64, device="cuda"), torch.empty(
            x.shape, dtype=torch.complex128, device="cuda")
        step = max(1, (1 << 24) // x.shape[1])
        for i in range(0, x.shape[0], step):
            y = _dft(x[i:i + step], -1)
            wi = w[i:i + step].to(torch.float64)
            loss += (wi * (y.real ** 2 + y.imag ** 2)).sum()
            gx[i:i + step] = _dft(2.0 * wi * y, 1)
        return loss, gx
    if kind == "uneven":
        y = torch.empty(x.shape, dtype=torch.complex128, device="cuda")
        groups, off = {}, 0
        for n in _lengths(case):
            groups.setdefault(n, []).append(off)
            off += n
        for n, offs in groups.items():
            step = max(1, (1 << 24) // n)
            for s in range(0, len(offs), step):
                idx = torch.tensor(offs[s:s + step], device="cuda")[:, None] + torch.arange(n, device="cuda")
                y[idx] = _dft(x[idx], case["dir"])
        return y
    N1, N2 = 1 << case["lg1"], 1 << case["lg2"]
    if kind == "fft2":
        a = x.to(torch.complex128).reshape(-1, N1, N2)
        y = torch.fft.fft2(a) if case["dir"] == -1 else torch.fft.ifft2(a, norm="forward")
        return y.transpose(1, 2).reshape(x.shape)
    a = x.to(torch.complex128).reshape(-1, N1, N2, 1 << case["lg3"])
    y = torch.fft.fftn(a, dim=(1, 2, 3)) if case["dir"] == -1 else torch.fft.ifftn(a, dim=(1, 2, 3), norm="forward")
    return y.permute(0, 3, 2, 1).reshape(x.shape)


def work(case):
    """Each input read once, each output written once; 5 N log2 N flops a
    transform (the usual count for a complex DFT of N points)."""
    n = _elems(case)
    kind = case["kind"]
    size = 16 if case.get("dtype") == "c128" else 8
    if kind == "uneven":
        return {"bytes": 2 * size * n, "flops": sum(5 * m * (m.bit_length() - 1) for m in _lengths(case))}
    lg = case["lg1"] + case["lg2"] + case.get("lg3", 0)
    flops = 5 * n * lg
    if kind == "grad":                      # x and g in, y and gx out
        return {"bytes": 4 * size * n, "flops": 2 * flops}
    if kind == "loss":                      # x and w in, gx and the loss out
        return {"bytes": 2 * size * n + 4 * n + 8, "flops": 2 * flops + 5 * n}
    return {"bytes": 2 * size * n, "flops": flops}
