"""How steps follow one another on a stream: programmatic dependent launches
(a step's entry overlaps the end of the work ahead of it) and the tail pool's
self-resetting counter.  Back-to-back steps among kernels that write their
gradients and read their weights, and captured steps replayed, equal separate
synchronised steps bit for bit."""
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

NAMES = ["flat_1m", "llama_7b", "llama_1p5b", "llama_1p5b_mixed", "llama_1p5b_nvfp4"]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2607_10611_gb300 import build
    build()


def _pair(name, pooled):
    import parity
    wl = W.SMALL[name] if not pooled else W.replace(W.CONFIGS["gpt2_124m"], specs=W.gpt2_specs(2, 768, 3000, 64))
    mt = W.materialize(wl, "cpu", warm_state=True)
    return [parity.Run(wl, mt=mt) for _ in range(2)]


def _same(a, b):
    for key in ("w", "m", "v", "ve", "bscale", "cc"):
        for x, y in zip(a.dev[key], b.dev[key]):
            if x is not None:
                assert torch.equal(x.view(torch.uint8), y.view(torch.uint8)), key


@pytest.mark.parametrize("name,pooled", [(n, False) for n in NAMES] + [("gpt2_124m", True)])
def test_back_to_back_steps(name, pooled):
    a, b = _pair(name, pooled)
    base = [g.clone() for g in a.dev["g"]]
    sums = []
    for t in range(1, 9):  # a: no synchronisation; gradients rewritten before and weights read after every step
        for g, g0 in zip(a.dev["g"], base):
            torch.mul(g0, 1.0 + 0.25 * t, out=g)
        a.opt.step(a.dev["g"], t)
        sums.append(torch.stack([w.view(torch.uint8).long().sum() for w in a.dev["w"]]).sum())
    for t in range(1, 9):
        for g, g0 in zip(b.dev["g"], base):
            torch.mul(g0, 1.0 + 0.25 * t, out=g)
        torch.cuda.synchronize()
        b.opt.step(b.dev["g"], t)
        torch.cuda.synchronize()
        assert torch.stack([w.view(torch.uint8).long().sum() for w in b.dev["w"]]).sum() == sums[t - 1]
    assert a.opt.device_status() == 0 and b.opt.device_status() == 0
    _same(a, b)
    a.close(); b.close()


@pytest.mark.parametrize("name,pooled", [(n, False) for n in NAMES] + [("gpt2_124m", True)])
def test_captured_steps_replay(name, pooled):
    a, b = _pair(name, pooled)
    for r in (a, b):  # the gradient table goes up outside the capture
        r.opt.step(r.dev["g"], 1)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        a.opt.step(a.dev["g"], 2)
        a.opt.step(a.dev["g"], 3)
    for _ in range(3):
        graph.replay()
    for _ in range(3):
        for t in (2, 3):
            b.opt.step(b.dev["g"], t)
            torch.cuda.synchronize()
    torch.cuda.synchronize()
    assert a.opt.device_status() == 0
    _same(a, b)
    a.close(); b.close()


@pytest.mark.parametrize("name,pooled", [("flat_1m", False), ("llama_1p5b_mixed", False), ("gpt2_124m", True)])
def test_captured_behind_a_copy_and_behind_a_join(name, pooled):
    """The work ahead of a captured step need not be a kernel: the first step of
    a state copies its gradient table inside the capture, and the next waits
    for gradients written on another captured stream."""
    a, b = _pair(name, pooled)
    base = [g.clone() for g in a.dev["g"]]
    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        a.opt.step(a.dev["g"], 1)
        main = torch.cuda.current_stream()
        side.wait_stream(main)
        with torch.cuda.stream(side):
            for g, g0 in zip(a.dev["g"], base):
                torch.mul(g0, 1.5, out=g)
        main.wait_stream(side)
        a.opt.step(a.dev["g"], 2)
    for _ in range(2):
        for g, g0 in zip(a.dev["g"], base):
            g.copy_(g0)
        graph.replay()
    torch.cuda.synchronize()
    for _ in range(2):
        for t, f in ((1, 1.0), (2, 1.5)):
            for g, g0 in zip(b.dev["g"], base):
                torch.mul(g0, f, out=g)
            b.opt.step(b.dev["g"], t)
            torch.cuda.synchronize()
    assert a.opt.device_status() == 0
    _same(a, b)
    a.close(); b.close()
