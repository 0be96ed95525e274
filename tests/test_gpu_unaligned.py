"""Gradients that start at any element (packed in one bucket) and one-byte
weights at multiples of 8 bytes: read through the stage like aligned ones,
bit for bit, at every offset modulo 16 bytes, around tile and warp
boundaries, and where a tensor's first or last bytes fall outside the whole
16-byte lines that are copied."""
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

SIZES = (256, 3840, 3841, 1, 7680, 255, 257, 512, 3839, 3848, 11521, 2, 5120, 8, 15, 4096 + 256, 7, 3840 * 3, 1024)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2607_10611_gb300 import build
    build()


def _workload(wd, gd, md, rnd):
    specs = tuple(W.TensorSpec(f"t{i}", n, "matrix" if i % 3 else "norm") for i, n in enumerate(SIZES))
    return W.Workload(name="unaligned", specs=specs, weight_dtype=wd, grad_dtype=gd, moment_dtype=md, rounding=rnd,
                      steps=2, seed=17, zero_frac=0.02, grad=("normal_logu", 1e-6, 1e-1), compute_copy=wd != "bf16")


def _run(wl, start=None, **kw):
    import parity
    r = parity.Run(wl, warm=True, **kw)
    if start is not None:  # gradients packed from element `start` of a bucket, NaN around and nowhere between
        g = r.dev["g"]
        total = sum(x.numel() for x in g)
        bucket = torch.full((start + total + 64,), float("nan"), dtype=g[0].dtype, device="cuda")
        o, views = start, []
        for x in g:
            views.append(bucket[o:o + x.numel()])
            views[-1].copy_(x)
            o += x.numel()
        r.dev["g"] = views
    for t in (1, 2):
        r.step(t)
        parity.assert_exact(r.compare(t + 1), f"step {t}")
    r.close()


@pytest.mark.parametrize("start", [0, 1, 2, 3, 5, 6, 7])
@pytest.mark.parametrize("gd", ["bf16", "f32"])
@pytest.mark.parametrize("wd,md,rnd", [("bf16", "f32", "stochastic"), ("bf16", "bf16", "nearest"),
                                       ("e4m3", "f32", "stochastic"), ("e4m3", "bf16", "nearest"),
                                       ("mixed_b32", "bf16", "stochastic"), ("mixed_fp4", "f32", "nearest"),
                                       ("mixed_fp4", "bf16", "stochastic")])
def test_bucketed_gradients(wd, md, rnd, gd, start):
    _run(_workload(wd, gd, md, rnd), start)


@pytest.mark.parametrize("start", [None, 1, 4])
@pytest.mark.parametrize("md,rnd", [("f32", "stochastic"), ("bf16", "nearest"), ("bf16", "stochastic")])
def test_one_byte_weights_at_multiples_of_eight(md, rnd, start):
    wl = _workload("e4m3", "bf16", md, rnd)
    _run(W.replace(wl, compute_copy=False), start, layout="flat")
    _run(_workload("mixed_b32", "bf16", md, rnd), start, misalign=8)


@pytest.mark.parametrize("hp", [dict(lr_mul=4.0, lr_add=0.3), dict(wd_add=0.1, g_max=0.7, w_max=0.05)])
@pytest.mark.parametrize("wd", ["bf16", "e4m3", "mixed_b32", "mixed_fp4"])
def test_exact_branch_reads_the_shifted_stage(wd, hp):
    """Large rates leave many elements undecided: their gradients are read again from the stage."""
    _run(_workload(wd, "bf16", "bf16", "stochastic"), 3, hp=hp)
