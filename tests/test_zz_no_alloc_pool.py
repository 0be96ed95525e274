"""mpadam_step_noalloc on lists long enough for its tail pool (chunks from the
end of the list, their first tensor found by search) and on lists short enough
to carry their tables with the launch: bit for bit what mpadam_step gives,
over calls that follow one another without synchronisation."""
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

E = W.TensorSpec("empty", 0, "flat")


@pytest.fixture(scope="module")
def N():
    from paper_2607_10611_gb300 import _native, build
    build()
    return _native


def _flat(*sizes):
    return tuple(W.TensorSpec(f"t{i}", n, "flat") for i, n in enumerate(sizes))


LISTS = {
    "ragged": W.ragged_specs(3000, 13, 4),                                  # tiny tensors, many to a chunk
    "empties": tuple(x for s in W.ragged_specs(700, 15, 6) for x in (E, s, E)) + (E, E),
    "large_then_tiny": _flat(5_000_001, *([1] * 400), 700_000, *([257] * 300)),
    "one": _flat(152 * 8 * 3840),                                           # the first size with a pool, tables inline
    "four": _flat(3840, 6_000_000, 1, 77_777),
    "below": _flat(152 * 8 * 3840 - 3840, 9),
}


@pytest.mark.parametrize("fmt", [("bf16", "bf16", "f32", "stochastic"), ("e4m3", "bf16", "bf16", "nearest")])
@pytest.mark.parametrize("name", list(LISTS))
def test_pool_matches_mpadam_step(N, name, fmt):
    from paper_2607_10611_gb300.optimizer import MPAdam
    wd, gd, md, rnd = fmt
    wl = W.Workload(name=name, specs=LISTS[name], weight_dtype=wd, grad_dtype=gd, moment_dtype=md, rounding=rnd,
                    steps=3, seed=5, zero_frac=0.1, grad=("normal_logu", 1e-6, 1e-1))
    mt = W.materialize(wl, "cuda", warm_state=True)
    a, b = ({k: [t.clone() for t in getattr(mt, k)] for k in ("w", "g", "m", "v", "ve")} for _ in range(2))
    ref = MPAdam(a["w"], a["m"], a["v"], a["ve"], weight_dtype=wd, grad_dtype=gd, moment_dtype=md, rounding=rnd,
                 seed=wl.seed, fp8_exp=mt.fp8_exp)
    cfg = N.make_config(weight_dtype=wd, grad_dtype=gd, moment_dtype=md, rounding=rnd, seed=wl.seed)
    exp = amax = None
    if wd == "e4m3":
        exp, amax = ref.fp8_exp_ring.clone(), ref.fp8_amax_ring.clone()
    ptr = lambda t: t.data_ptr() if t.numel() else 0
    tensors = [(ptr(w), ptr(m), ptr(v), ptr(ve), w.numel()) for w, m, v, ve in zip(b["w"], b["m"], b["v"], b["ve"])]
    stream = torch.cuda.current_stream().cuda_stream
    for t in (1, 2, 3):
        ref.step(a["g"], t)
        N.mpadam_step_noalloc(tensors, [ptr(g) for g in b["g"]], cfg, t, exp.data_ptr() if exp is not None else 0,
                              amax.data_ptr() if amax is not None else 0, stream)
    assert N.mpadam_noalloc_status(stream) == 0 and ref.device_status() == 0
    for key in ("w", "m", "v", "ve"):
        for k, (x, y) in enumerate(zip(a[key], b[key])):
            assert torch.equal(x.view(torch.uint8), y.view(torch.uint8)), (key, k)
    if exp is not None:
        assert torch.equal(exp, ref.fp8_exp_ring) and torch.equal(amax, ref.fp8_amax_ring)
    ref.close()
