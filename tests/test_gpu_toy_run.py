"""mpadam_toy_run (many steps inside one cooperative kernel) against the oracle,
weights and every step's loss bit for bit: all regimes and rules at the full
size, and the smallest and largest batches it splits over CTAs (one warp, one
CTA, all CTAs at their most threads)."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

LR = {"additive": dict(lr_add=1024.0), "multiplicative": dict(lr_mul=1024.0),
      "combined": dict(lr_add=1024.0, lr_mul=1024.0)}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2607_10611_gb300 import build
    build()


def _setup(regime, mode, n, batch):
    from paper_2607_10611_gb300.toy import ToyDiagnostic
    p = W.toy_problem(regime, n=n, seed=5)
    lr = {k: v * batch / 65536 for k, v in LR[mode].items()}
    kw = dict(batch=batch, c_lo=p.c_lo, c_hi=p.c_hi, split=p.split, seed=11, **lr)
    w = p.w0.to("cuda")
    return p, w, ToyDiagnostic(w, p.wstar.to("cuda"), mode=mode, **kw), oracle.toy_config(mode, **kw)


def _compare(regime, mode, n, batch, runs):
    p, w, d, cfg = _setup(regime, mode, n, batch)
    losses = torch.zeros(sum(runs), dtype=torch.float64, device="cuda")
    t = 0
    for k in runs:  # consecutive calls continue one another
        d.run(t + 1, k, losses[t:t + k])
        t += k
    assert d.device_status() == 0
    hw, hs = W.to_numpy_bits(p.w0), p.wstar.numpy()
    want = np.array([oracle.toy_step(cfg, hw, hs, i) for i in range(1, t + 1)])
    bad = int((W.to_numpy_bits(w) != hw).sum())
    assert bad == 0, f"{regime}/{mode}: {bad} weights differ"
    np.testing.assert_array_equal(losses.cpu().numpy().view(np.uint64), want.view(np.uint64))
    d.close()


@pytest.mark.parametrize("mode", ["additive", "multiplicative", "combined"])
@pytest.mark.parametrize("regime", W.TOY_REGIMES)
def test_full_size(regime, mode):
    _compare(regime, mode, W.TOY_N, 65536, [5, 1])


@pytest.mark.parametrize("regime,n,batch", [
    ("mixed", 64, 64), ("large", 64, 64), ("mixed", 64, 128), ("small", 64, 128),
    ("sign_flip", 64, 256), ("mixed", 128, 512), ("mixed", 256, 16384), ("large", 256, 32768),
    ("mixed", 512, 131072)])
def test_batches_over_ctas(regime, n, batch):
    _compare(regime, "combined", n, batch, [1, 70, 2])


def test_run_under_capture_replays():
    """A captured run replays: each replay repeats the same step numbers."""
    p, w, d, cfg = _setup("sign_flip", "combined", 64, 1024)
    losses = torch.zeros(3, dtype=torch.float64, device="cuda")
    s = torch.cuda.Stream()
    d.run(1, 1)  # warm-up outside the capture
    torch.cuda.synchronize()
    w.copy_(p.w0)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        d.run(1, 3, losses, stream=s)
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    assert d.device_status() == 0
    hw, hs = W.to_numpy_bits(p.w0), p.wstar.numpy()
    for _ in range(2):
        want = np.array([oracle.toy_step(cfg, hw, hs, i) for i in range(1, 4)])
    assert (W.to_numpy_bits(w) == hw).all()
    np.testing.assert_array_equal(losses.cpu().numpy().view(np.uint64), want.view(np.uint64))
    d.close()
