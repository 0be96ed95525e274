"""The certified fast path at the edges of what it accepts: the approximate
reciprocal's error bound, the host's conditions on eps, and the E4M3 encoders
where codes stop being certifiable (subnormal codes, saturation at the largest
scale)."""
import ctypes
import subprocess
from pathlib import Path

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu
HERE = Path(__file__).resolve().parent


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2607_10611_gb300 import build
    build()


def P():
    import parity
    return parity


def test_reciprocal_within_certificate_bound(tmp_path):
    out = tmp_path / "librcp_probe.so"
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "--ftz=false",
                    "-Xcompiler", "-fPIC", "-shared", str(HERE / "cuda" / "rcp_probe.cu"), "-o", str(out)], check=True)
    lib = ctypes.CDLL(str(out))
    lib.rcp_probe.argtypes = [ctypes.c_void_p, ctypes.c_int64, ctypes.c_void_p]
    g = torch.Generator(device="cuda").manual_seed(0)
    # every mantissa in one binade, then all exponents with a normal reciprocal
    one = (torch.arange(1 << 23, dtype=torch.int32, device="cuda") + 0x3F800000).view(torch.float32)
    e = torch.randint(-125, 126, (1 << 26,), device="cuda", generator=g).float()
    wide = (torch.rand(1 << 26, device="cuda", generator=g) + 1) * torch.exp2(e)
    for b in (one, wide):
        worst = torch.zeros(1, device="cuda")
        assert lib.rcp_probe(b.data_ptr(), b.numel(), worst.data_ptr()) == 0
        assert worst.item() < 2.0 ** -21


def _steps(r, steps, what):
    p = P()
    for t in range(1, steps + 1):
        r.step(t)
        p.assert_exact(r.compare(t + 1), f"{what} step {t}")
    r.close()


# eps from the smallest certified one to past the largest (2^60: beyond it a
# finite denominator could leave the reciprocal's normal range)
@pytest.mark.parametrize("eps", [2.0 ** -28, 2.0 ** 60, 2.0 ** 61, 2.0 ** 126])
@pytest.mark.parametrize("name", ["llama_7b", "llama_1p5b"])
def test_eps_at_the_certificate_limits(name, eps):
    _steps(P().Run(W.SMALL[name], warm=True, hp=dict(eps=eps)), 2, f"{name} eps {eps}")


# Infinite moments with finite gradients: both sides divide by infinity
@pytest.mark.parametrize("name", ["gpt2_124m", "llama_1p5b", "llama_1p5b_mixed", "llama_1p5b_nvfp4"])
def test_infinite_moments(name):
    mt = W.materialize(W.SMALL[name], "cpu", warm_state=True)
    for k in range(len(mt.v)):
        mt.v[k][::37] = float("inf")
        mt.ve[k][::41] = float("inf")
        mt.m[k][5::1009] = -float("inf")
    _steps(P().Run(W.SMALL[name], mt=mt), 2, name)


# Block-scaled codes at both ends of the range: blocks at the largest scale
# whose weights grow past 448 2^15 (codes saturate), and blocks of subnormal
# codes and codes next to them
@pytest.mark.parametrize("rnd", ["nearest", "stochastic"])
@pytest.mark.parametrize("md", ["f32", "bf16"])
def test_block_codes_at_the_ends_of_the_range(md, rnd):
    wl = W.replace(W.SMALL["llama_1p5b_mixed"], moment_dtype=md, rounding=rnd, name="ends")
    mt = W.materialize(wl, "cpu", warm_state=True)
    gen = torch.Generator().manual_seed(3)
    for k, f in enumerate(mt.formats):
        if f != "e4m3_b32":
            continue
        n = mt.w[k].numel()
        small = torch.randint(0, 20, (n,), generator=gen, dtype=torch.uint8)  # subnormal codes are 0..7
        large = torch.randint(118, 127, (n,), generator=gen, dtype=torch.uint8)
        pick = (torch.arange(n) // W.BLOCK) % 2 == 0
        mt.w[k].copy_(torch.where(pick, small, large) | (torch.randint(0, 2, (n,), generator=gen, dtype=torch.uint8) << 7))
        sc = torch.where((torch.arange(mt.bscale[k].numel()) % 2) == 0, torch.tensor(2.0 ** -10), torch.tensor(2.0 ** 15))
        mt.bscale[k].copy_(sc.to(torch.float16))
    _steps(P().Run(wl, mt=mt, hp=dict(lr_mul=0.5, lr_add=1e-3)), 3, f"ends {md}/{rnd}")


# The options' certified path in every weight format: clamps that bind for
# many elements (so that intervals straddle them), decay up to and past the
# largest the certificate takes (eta_a lambda = 1), and non-finite inputs,
# which a clamp would hide
OPTIONS = [dict(g_max=0.7, w_max=0.02, wd_add=0.1), dict(g_max=1e-3), dict(w_max=1e-3), dict(lr_add=0.5, wd_add=2.0),
           dict(lr_add=0.5, wd_add=2.5), dict(lr_mul=4.0, lr_add=0.3, wd_add=0.3, g_max=2.0, w_max=0.5)]


@pytest.mark.parametrize("hp", OPTIONS)
@pytest.mark.parametrize("rnd", ["nearest", "stochastic"])
@pytest.mark.parametrize("name", ["llama_7b", "llama_1p5b", "llama_1p5b_mixed", "llama_1p5b_nvfp4"])
def test_options_in_every_format(name, rnd, hp):
    mt = W.materialize(W.replace(W.SMALL[name], moment_dtype="bf16", rounding=rnd), "cpu", warm_state=True)
    big = max(range(len(mt.g)), key=lambda k: mt.g[k].numel())
    for i, x in enumerate((float("nan"), float("inf"), -float("inf"))):
        mt.g[big][100 * i::977] = x
    mt.ve[big][17::1009] = float("inf")
    wl = mt.workload
    _steps(P().Run(wl, mt=mt, hp=hp), 2, f"{name}/{rnd}/{hp}")


# Stochastic E2M1 codes read off binary32's bits, where that can go wrong:
# weights that a small step leaves beside a code (so beside zero, beside 1,
# where 1 + x takes over from x, beside the binade edges 2 and 4 and the
# saturation point 6), steps from far below a tick of 2^-22 to several codes
# (an error bound ei from under 2^-24, one constant, to past 2^-3, nothing
# certified), and enough elements that some random bits lie at the decision
@pytest.mark.parametrize("md", ["f32", "bf16"])
@pytest.mark.parametrize("lr", [1e-7, 1e-4, 1e-2, 1e2, 1e5])
def test_stochastic_e2m1_codes_beside_the_grid(lr, md):
    wl = W.Workload(name="grid", specs=tuple(W.TensorSpec(f"t{i}", n, "matrix") for i, n in enumerate((200000, 3840, 97))),
                    weight_dtype="nvfp4", grad_dtype="bf16", moment_dtype=md, rounding="stochastic", steps=2, seed=23,
                    zero_frac=0.0, grad=("normal_logu", 1e-6, 1e-1), compute_copy=True)
    mt = W.materialize(wl, "cpu", warm_state=True)
    gen = torch.Generator().manual_seed(5)
    for k in range(len(mt.w)):
        mt.w[k].copy_(torch.randint(0, 256, (mt.w[k].numel(),), generator=gen, dtype=torch.uint8))
        if mt.g[k].numel() % 2:
            mt.w[k][-1] &= 0x0F  # the spare nibble is zero
    _steps(P().Run(wl, mt=mt, hp=dict(lr_add=lr, lr_mul=min(lr, 0.5))), 2, f"grid lr={lr}/{md}")
