"""binding.py: tensors that a kernel could not read or write are refused before the library is entered."""
import importlib

import pytest


@pytest.fixture()
def binding():
    return importlib.import_module("paper_2609_10937_b200.binding")


class OnDevice:
    """A CUDA tensor as far as the argument checks look at one."""

    is_cuda = True

    def __init__(self, torch, *shape, device=0, dtype=None, contiguous=True):
        self.shape, self.dtype = torch.Size(shape), dtype or torch.bfloat16
        self.device, self._contiguous = torch.device("cuda", device), contiguous

    def is_contiguous(self):
        return self._contiguous

    def dim(self):
        return len(self.shape)

    def numel(self):
        return self.shape.numel()

    def get_device(self):
        return self.device.index

    def data_ptr(self):
        return 4096


def _calls(binding, monkeypatch):
    torch = importlib.import_module("torch")
    entered = []
    monkeypatch.setattr(binding, "_call", lambda *args, **kwargs: entered.append(args[1]))
    monkeypatch.setattr(binding, "_stream", lambda dev: 0)
    monkeypatch.setattr(binding, "_torch", torch, raising=False)
    return torch, (lambda *shape, **kwargs: OnDevice(torch, *shape, **kwargs)), entered


def test_forward_qk_refuses_outputs_that_its_result_does_not_fit(binding, monkeypatch):
    torch, t, entered = _calls(binding, monkeypatch)
    q, k, v = t(2, 3, 40, 64), t(2, 3, 90, 64), t(2, 3, 90, 64)
    for o in (t(2, 3, 39, 64), t(2, 3, 41, 64), t(2, 3, 40, 64, contiguous=False), t(2, 3, 40, 64, dtype=torch.float32), t(2, 3, 40, 64, dtype=torch.float16),
              t(2, 3, 40, 64, device=1), torch.empty(2, 3, 40, 64, dtype=torch.bfloat16)):
        with pytest.raises(ValueError):
            binding.forward_qk(q, k, v, o)
    assert entered == []
    for o in (t(2, 3, 40, 64), t(6, 40 * 64)):               # the same elements in a row, as gemm takes its c
        assert binding.forward_qk(q, k, v, o) is o
    assert entered == ["attn_forward_qk"] * 2


def test_operands_on_another_device_are_refused(binding, monkeypatch):
    torch, t, entered = _calls(binding, monkeypatch)
    here, there = t(2, 3, 40, 64), t(2, 3, 40, 64, device=1)
    for q, k, v in ((here, there, here), (here, here, there), (there, here, here)):
        for call in (binding.forward, binding.forward_qk):
            with pytest.raises(ValueError):
                call(q, k, v, t(2, 3, 40, 64))
    for a, b in ((t(40, 64), t(64, 48, device=1)), (t(40, 64, device=1), t(64, 48))):
        with pytest.raises(ValueError):
            binding.gemm(a, b, t(40, 48))
    assert entered == []
    o = t(2, 3, 40, 64)
    assert binding.forward(here, here, here, o) is o and binding.gemm(t(40, 64), t(64, 48), c := t(40, 48)) is c
    assert entered == ["attn_forward", "gemm_forward"]


@pytest.mark.gpu
def test_refused_outputs_are_not_written(binding):
    torch = importlib.import_module("torch")
    q, k, v = (torch.randn(2, 3, n, 64, device="cuda").to(torch.bfloat16) for n in (40, 90, 90))
    good = binding.forward_qk(q, k, v)
    strided = torch.zeros(2, 3, 40, 128, dtype=torch.bfloat16, device="cuda")[..., :64]
    for o in (q[:, :, :39].contiguous(), strided, torch.zeros_like(q, dtype=torch.float32), torch.zeros(2, 3, 40, 64, dtype=torch.bfloat16)):
        before = o.clone()
        with pytest.raises(ValueError):
            binding.forward_qk(q, k, v, o)
        assert torch.equal(o, before)
    flat = torch.empty(6, 40 * 64, dtype=torch.bfloat16, device="cuda")
    assert binding.forward_qk(q, k, v, flat) is flat and torch.equal(flat.view_as(good).view(torch.int16), good.view(torch.int16))
    assert binding.last_device_status()[0] == 0
