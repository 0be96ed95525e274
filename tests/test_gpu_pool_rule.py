"""The library's own choice of tile runs and pool chunks (by tiles per CTA and
tiles per tensor) changes no bit: lists on either side of every limit of the
rule, with few and with many tensors, stepped by the default and by static
runs."""
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

TILE, CTAS = 3840, 152


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2607_10611_gb300 import build
    build()


def _sizes(per_cta, many):
    n = per_cta * CTAS * TILE
    if not many:  # a large tensor, an empty one, one that ends inside a tile
        return (n - 2 * TILE, 0, TILE + 7)
    k = per_cta * CTAS // 3
    return tuple([2 * TILE + 5, 0] * k) + (9,)  # three tiles each, the last of 5 elements


@pytest.mark.parametrize("many", [False, True])
@pytest.mark.parametrize("per_cta", [7, 8, 15, 16, 127, 128])
@pytest.mark.parametrize("formats", [("bf16",), ("e4m3",), ("bf16", "e4m3_b32")])
def test_default_rule_equals_static_runs(per_cta, many, formats):
    from paper_2607_10611_gb300.optimizer import MPAdam
    if per_cta > 100 and len(formats) == 1 and formats[0] == "e4m3" and many:
        pytest.skip("long, and covered by the others")
    sizes = _sizes(per_cta, many)
    fmts = [formats[i % len(formats)] for i in range(len(sizes))] if not many else \
        [formats[(i // 2) % len(formats)] for i in range(len(sizes))]
    wl = W.Workload(name="rule", specs=tuple(W.TensorSpec(f"t{i}", n, "matrix") for i, n in enumerate(sizes)),
                    weight_dtype="bf16" if len(formats) > 1 else formats[0], grad_dtype="bf16", moment_dtype="bf16",
                    rounding="stochastic", steps=2, seed=3, grad=("normal_logu", 1e-6, 1e-2),
                    format_list=tuple(fmts) if len(formats) > 1 else ())
    mt = W.materialize(wl, "cuda", warm_state=True)
    outs = []
    for static in (False, True):
        w, m, v, ve, sc = ([t.clone() if t is not None else None for t in x] for x in (mt.w, mt.m, mt.v, mt.ve, mt.bscale))
        ext = len(formats) > 1
        o = MPAdam(w, m, v, ve, weight_dtype=fmts if ext else formats[0], grad_dtype="bf16", moment_dtype="bf16",
                   rounding="stochastic", seed=3, fp8_exp=mt.fp8_exp, block_scales=sc if ext else None)
        if static:
            o.set_tail_pool(1024, 1)
        for t in (1, 2, 3):
            o.step(mt.g, t)
        assert o.device_status() == 0
        rings = [o.fp8_exp_ring, o.fp8_amax_ring] if o.fp8_exp_ring is not None else []
        outs.append([torch.cat([t.view(torch.uint8).view(-1) for t in x if t is not None]) for x in (w, m, v, ve)] +
                    [t.view(torch.uint8).view(-1) for t in sc if t is not None] + rings)
        o.close()
    for x, y in zip(*outs):
        assert torch.equal(x, y)
