"""What MPAdam.step hands to the C ABI, checked on the host (no GPU): each
gradient's own data_ptr(), whatever kind of object it is, and the current
stream, also where torch does not offer its raw handle."""
import types

import pytest
import torch

from paper_2607_10611_gb300 import _native as N
from paper_2607_10611_gb300 import optimizer as O


@pytest.fixture
def step(monkeypatch):
    calls = []
    monkeypatch.setattr(N, "mpadam_step", lambda state, grads, t, stream=0: calls.append((list(grads), stream)))
    monkeypatch.setattr(O, "_get_raw_stream", lambda index: 100 + index)  # as torch's, it wants a number
    opt = object.__new__(O.MPAdam)
    opt.state, opt.device = None, torch.device("cuda", 3)

    def run(grads, **kw):
        opt.step(grads, 1, **kw)
        return calls[-1]
    run.opt = opt
    return run


class Moved(torch.Tensor):
    """A tensor whose data lies elsewhere."""

    def data_ptr(self):
        return 0x7000


def test_pointers_of_every_kind_of_gradient(step):
    a, b = torch.zeros(3), torch.nn.Parameter(torch.zeros(5))
    c, d = torch.zeros(2).as_subclass(Moved), types.SimpleNamespace(data_ptr=lambda: 0x9000)
    want = [a.data_ptr(), b.data_ptr(), 0x7000, 0x9000]
    for grads in ([a, b, c, d], (a, b, c, d), (x for x in (a, b, c, d))):
        assert step(grads)[0] == want
    with pytest.raises(AttributeError):
        step([a, None])


def test_current_stream(step, monkeypatch):
    assert step([])[1] == 103
    assert step([], stream=types.SimpleNamespace(cuda_stream=7))[1] == 7
    seen = []
    monkeypatch.setattr(torch.cuda, "current_stream", lambda d: seen.append(d) or types.SimpleNamespace(cuda_stream=55))
    step.opt.device = torch.device("cuda")  # no index: the current device's
    assert step([])[1] == 55 and seen == [torch.device("cuda")]
    step.opt.device = torch.device("cuda", 3)
    monkeypatch.setattr(O, "_get_raw_stream", None)  # a torch without it
    assert step([])[1] == 55 and seen[-1] == torch.device("cuda", 3)
