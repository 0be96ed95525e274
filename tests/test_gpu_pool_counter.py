"""The tail pool's claim counters when something went wrong before: whatever
overlapping calls left in theirs spoils no later call, and what a launch that
gave up left is cleared with its status.  The leftovers are written by the
host (mpadam_debug_spoil_pool); nothing overlaps or gives up here."""
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

TILE, CTAS = 3840, 152
N_POOLED = 10 * CTAS * TILE  # ten tiles a CTA: a quarter of them in the pool


@pytest.fixture(scope="module")
def N():
    from paper_2607_10611_gb300 import _native, build
    build()
    return _native


def _arrays(sizes):
    specs = tuple(W.TensorSpec(f"t{i}", n, "flat") for i, n in enumerate(sizes))
    wl = W.Workload(name="counter", specs=specs, weight_dtype="bf16", grad_dtype="bf16", moment_dtype="bf16",
                    rounding="stochastic", steps=2, seed=9, grad=("normal_logu", 1e-6, 1e-2))
    mt = W.materialize(wl, "cuda", warm_state=True)
    return [{k: [t.clone() for t in getattr(mt, k)] for k in ("w", "g", "m", "v", "ve")} for _ in range(2)]


FMT = dict(weight_dtype="bf16", grad_dtype="bf16", moment_dtype="bf16", rounding="stochastic", seed=9)


def _same(a, b):
    for key in ("w", "m", "v", "ve"):
        for x, y in zip(a[key], b[key]):
            assert torch.equal(x.view(torch.uint8), y.view(torch.uint8)), key


# N_POOLED makes a pool of one chunk per CTA, whose claims end at 2 x 152
@pytest.mark.parametrize("value", [1, 100, 200, 0x7FFFFFFF])
@pytest.mark.parametrize("how", ["calls", "status", "grid", "pool"])
def test_state(N, value, how):
    from paper_2607_10611_gb300.optimizer import MPAdam
    a, b = _arrays([N_POOLED, 777])
    oa, ob = (MPAdam(x["w"], x["m"], x["v"], x["ve"], **FMT) for x in (a, b))
    ob.set_tail_pool(1024, 1)
    for t in (1, 2):
        oa.step(a["g"], t)
        ob.step(b["g"], t)
    N.mpadam_debug_spoil_pool(oa.state, value, 0 if how == "calls" else 2)
    if how == "status":
        assert oa.device_status() == 2 and oa.device_status() == 0
    elif how == "grid":
        oa.set_grid(0)
    elif how == "pool":
        oa.set_tail_pool(768, 4)
    for t in range(3, 10):
        oa.step(a["g"], t)
        ob.step(b["g"], t)
    torch.cuda.synchronize()
    _same(a, b)
    oa.close(); ob.close()


@pytest.mark.parametrize("value", [1, 100, 200, 0x7FFFFFFF])
@pytest.mark.parametrize("how", ["calls", "status"])
@pytest.mark.parametrize("extra", [1, 8])  # tables with the launch, and in the library's array
def test_noalloc(N, value, how, extra):
    from paper_2607_10611_gb300.optimizer import MPAdam
    a, b = _arrays([N_POOLED] + [777] * extra)
    ob = MPAdam(b["w"], b["m"], b["v"], b["ve"], **FMT)
    ob.set_tail_pool(1024, 1)
    cfg = N.make_config(**FMT)
    ptrs = [tuple(x.data_ptr() for x in t) + (t[0].numel(),) for t in zip(a["w"], a["m"], a["v"], a["ve"])]
    grads = [g.data_ptr() for g in a["g"]]
    stream = torch.cuda.current_stream().cuda_stream
    for t in range(1, 10):
        N.mpadam_step_noalloc(ptrs, grads, cfg, t, stream=stream)
        ob.step(b["g"], t)
        if t == 2:
            N.mpadam_debug_spoil_pool(0, value, 0 if how == "calls" else 2)
            if how == "status":
                assert N.mpadam_noalloc_status(stream) == 2
    assert N.mpadam_noalloc_status(stream) == 0
    _same(a, b)
    ob.close()
