"""The library's own choice of tile runs and pool chunks (by tiles per CTA,
tiles per tensor and formats) changes no bit: lists with exactly the tiles on
either side of every limit of the rule, in every weight format and with long
and with short tensors, stepped by the default and by static runs."""
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

TILE = 3840


@pytest.fixture(scope="module")
def N():
    from paper_2607_10611_gb300 import _native, build
    build()
    return _native


def _sizes(tiles, many):
    """Tensors of `tiles` tiles in all."""
    if not many:  # a long tensor, an empty one, one that ends inside a tile
        sizes = [(tiles - 2) * TILE, 0, TILE + 7]
    else:  # three tiles each, the last of 5 elements, empty ones between, and what is left over
        sizes = [2 * TILE + 5, 0] * (tiles // 3)
        if tiles % 3:
            sizes.append((tiles % 3 - 1) * TILE + 9)
    assert sum(-(-n // TILE) for n in sizes) == tiles
    return sizes


def _outputs(wl, mt, fmts, ctas, static):
    from paper_2607_10611_gb300.optimizer import MPAdam
    w, m, v, ve, sc = ([t.clone() if t is not None else None for t in x]
                       for x in (mt.w, mt.m, mt.v, mt.ve, mt.bscale or [None] * len(mt.w)))
    plain = set(fmts) <= {"bf16", "e4m3"} and len(set(fmts)) == 1
    o = MPAdam(w, m, v, ve, weight_dtype=fmts[0] if plain else fmts, grad_dtype="bf16", moment_dtype=wl.moment_dtype,
               rounding="stochastic", seed=3, fp8_exp=mt.fp8_exp, block_scales=None if plain else sc,
               global_scales=None if plain else mt.gscale)
    o.set_grid(ctas)
    if static:
        o.set_tail_pool(1024, 1)
    for t in (1, 2, 3):
        o.step(mt.g, t)
    assert o.device_status() == 0
    rings = [o.fp8_exp_ring, o.fp8_amax_ring] if o.fp8_exp_ring is not None else []
    out = [torch.cat([t.view(torch.uint8).view(-1) for t in x if t is not None]) for x in (w, m, v, ve)] + \
        [t.view(torch.uint8).view(-1) for t in sc if t is not None] + rings
    o.close()
    return out


@pytest.mark.parametrize("md", ["bf16", "f32"])
@pytest.mark.parametrize("many", [False, True])
@pytest.mark.parametrize("limit,ctas", [(8, 152), (8, 24), (16, 24), (128, 24)])
@pytest.mark.parametrize("formats", [("bf16",), ("e4m3",), ("e4m3_b32",), ("nvfp4",), ("bf16", "e4m3_b32")])
def test_default_rule_equals_static_runs(N, formats, limit, ctas, many, md):
    rules = []
    for tiles in (limit * ctas - 1, limit * ctas):
        one = _sizes(tiles, many)  # each format's own tensors, interleaved
        sizes = [n for n in one for _ in formats]
        fmts = list(formats) * len(one)
        wl = W.Workload(name="rule", specs=tuple(W.TensorSpec(f"t{i}", n, "matrix") for i, n in enumerate(sizes)),
                        weight_dtype="bf16" if len(formats) > 1 else formats[0], grad_dtype="bf16", moment_dtype=md,
                        rounding="stochastic", steps=2, seed=3, grad=("normal_logu", 1e-6, 1e-2),
                        format_list=tuple(fmts) if len(formats) > 1 else ())
        mt = W.materialize(wl, "cuda", warm_state=True)
        for x, y in zip(*(_outputs(wl, mt, fmts, ctas, static) for static in (False, True))):
            assert torch.equal(x, y)
        rules.append([N.mpadam_debug_pool_rule(tiles, len(one), ctas, N.DTYPE[f], N.DTYPE[md]) for f in formats])
    for f, below, at in zip(formats, *rules):  # the two sides are two ways of dealing out
        assert below != at or f == "e4m3", f
