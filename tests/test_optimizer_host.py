"""What MPAdam.step hands to the C ABI, checked on the host (no GPU): each
gradient's own data_ptr(), whatever kind of object it is, and the current
stream, also where torch does not offer its raw handle."""
import gc
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


def _moved(mixin):
    """A kind of tensor whose data lies elsewhere: its own method, or one from another base."""
    class Elsewhere:
        def data_ptr(self):
            return 0x7000
    if mixin:
        return type("Moved", (Elsewhere, torch.Tensor), {})
    return type("Moved", (torch.Tensor,), {"data_ptr": Elsewhere.data_ptr})


@pytest.mark.parametrize("n", [1, 2 * O._MANY])  # by the tensors' types, and by the classes that are loaded
@pytest.mark.parametrize("mixin", [False, True])
def test_pointers_of_every_kind_of_gradient(step, mixin, n):
    gc.collect()  # classes of earlier tests
    assert not O._own_data_ptr()
    a, b = torch.zeros(3), torch.nn.Parameter(torch.zeros(5))
    d = types.SimpleNamespace(data_ptr=lambda: 0x9000)
    assert step([a, b] * n)[0] == [a.data_ptr(), b.data_ptr()] * n
    assert step([a, d] * n)[0] == [a.data_ptr(), 0x9000] * n
    c = torch.zeros(2).as_subclass(_moved(mixin))
    assert O._own_data_ptr()
    want = [a.data_ptr(), b.data_ptr(), 0x7000, 0x9000]
    for grads in ([a, b, c, d] * n, (a, b, c, d) * n, (x for x in [a, b, c, d] * n)):
        assert step(grads)[0] == want * n
    with pytest.raises(AttributeError):
        step([a, None] * n)


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
