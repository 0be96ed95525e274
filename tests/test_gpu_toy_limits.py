"""The branches of mpadam_toy_run that an ordinary run does not take: launches
after the first 8192 steps, the step-by-step way where a cooperative launch
does not fit (the refusal is made on the host), and waits that give up (a
build whose waits poll once)."""
import ctypes
import subprocess
from pathlib import Path

import numpy as np
import pytest
import torch

import oracle
import workloads as W

pytestmark = pytest.mark.gpu
HERE = Path(__file__).resolve().parent
LR, SEED = 3.0, 11


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2607_10611_gb300 import build
    build()


def _probe(tmp_path_factory, name, *defines):
    from paper_2607_10611_gb300 import builder as B
    out = tmp_path_factory.mktemp(name) / f"lib{name}.so"
    subprocess.run([B.nvcc(), *B.NVCC_FLAGS, *defines, "-shared", str(HERE / "cuda" / "toy_run_probe.cu"), "-o", str(out)],
                   check=True)
    f = ctypes.CDLL(str(out)).toy_run_probe
    p, i64, f32 = ctypes.c_void_p, ctypes.c_longlong, ctypes.c_float
    f.argtypes = [p, p, i64, i64, ctypes.c_int, f32, f32, f32, ctypes.c_ulonglong, i64, i64, p, p]
    return f


@pytest.fixture(scope="module")
def refused(tmp_path_factory):
    return _probe(tmp_path_factory, "toy_refused", "-DREFUSE_COOPERATIVE")


@pytest.fixture(scope="module")
def impatient(tmp_path_factory):
    return _probe(tmp_path_factory, "toy_impatient", "-DMPADAM_TOY_SPIN_LIMIT=1")


def _oracle(p, batch, first, steps):
    kw = dict(batch=batch, c_lo=p.c_lo, c_hi=p.c_hi, split=p.split, seed=SEED, lr_add=LR, lr_mul=LR)
    cfg = oracle.toy_config("combined", **kw)
    hw, hs = W.to_numpy_bits(p.w0), p.wstar.numpy()
    return kw, hw, np.array([oracle.toy_step(cfg, hw, hs, i) for i in range(first, first + steps)])


def _check(w, losses, hw, want):
    assert (W.to_numpy_bits(w) == hw).all()
    np.testing.assert_array_equal(losses.cpu().numpy().view(np.uint64), want.view(np.uint64))


@pytest.mark.parametrize("regime", ["mixed", "large"])
def test_more_steps_than_a_launch_holds(regime):
    from paper_2607_10611_gb300.toy import ToyDiagnostic
    p = W.toy_problem(regime, n=8, seed=5)
    steps = 2 * 8192 + 5
    kw, hw, want = _oracle(p, 64, 3, steps)
    w = p.w0.to("cuda")
    d = ToyDiagnostic(w, p.wstar.to("cuda"), mode="combined", **kw)
    losses = torch.zeros(steps, dtype=torch.float64, device="cuda")
    d.run(3, steps, losses)
    assert d.device_status() == 0
    _check(w, losses, hw, want)
    d.close()


def _run_probe(f, p, batch, first, steps):
    w, ws = p.w0.to("cuda"), p.wstar.to("cuda")
    losses = torch.zeros(steps, dtype=torch.float64, device="cuda")
    err = ctypes.c_int(-1)
    torch.cuda.synchronize()
    assert f(w.data_ptr(), ws.data_ptr(), w.numel(), batch, int(p.split), LR, p.c_lo, p.c_hi, SEED, first, steps,
             losses.data_ptr(), ctypes.byref(err)) == 0
    return w, losses, err.value


@pytest.mark.parametrize("regime,batch", [("mixed", 64), ("sign_flip", 512)])
def test_step_by_step_where_the_launch_does_not_fit(refused, regime, batch):
    p = W.toy_problem(regime, n=64, seed=5)
    _, hw, want = _oracle(p, batch, 7, 20)
    w, losses, err = _run_probe(refused, p, batch, 7, 20)
    assert err == 0
    _check(w, losses, hw, want)


@pytest.mark.parametrize("regime,batch", [("mixed", 512), ("sign_flip", 16384)])
def test_a_wait_that_gives_up_ends_the_run_with_a_status(impatient, regime, batch):
    """Several CTAs that have to wait for one another, and poll once: the run returns, and says so."""
    p = W.toy_problem(regime, n=64, seed=5)
    _, _, err = _run_probe(impatient, p, batch, 1, 10)
    assert err == 1
