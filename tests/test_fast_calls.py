"""csrc/py_fast.cpp: the usual calls without the interpreter give what binding.py gives, and what is not usual is left to binding.py."""
import importlib

import pytest


@pytest.fixture()
def binding():
    return importlib.import_module("paper_2609_10937_b200.binding")


def _calls(torch, binding, device):
    gen = torch.Generator(device=device).manual_seed(5)
    t = lambda *shape: torch.randn(*shape, generator=gen, device=device).to(torch.bfloat16)
    q, k, v, x = t(2, 3, 200, 64), t(2, 3, 200, 64), t(2, 3, 200, 64), t(2, 3, 90, 64)
    a, b, s = t(2, 130, 72), t(2, 72, 136), t(50, 128)
    return [
        lambda: binding.forward(q, k, v), lambda: binding.forward(q, k, v, torch.empty_like(q), causal=True), lambda: binding.forward_qk(x, k, v),
        lambda: binding.forward_qk(x, k, v, torch.empty_like(x)), lambda: binding.gemm(a, b), lambda: binding.gemm(a[0], b[0], torch.empty_like(a[0] @ b[0])),
        lambda: binding.gemm(a[1], b[1].T.contiguous(), b_layout="nk"), lambda: binding.softmax_rows(s, 0.125), lambda: binding.softmax_rows(s, 1, torch.empty_like(s)),
        # refused by both: shapes, types, strides, a name, a size the library does not have
        lambda: binding.forward(q, k, x), lambda: binding.forward(q.float(), k, v), lambda: binding.forward(q.transpose(1, 2), k, v), lambda: binding.forward(q[0], k[0], v[0]),
        lambda: binding.forward(q, k, v, x), lambda: binding.forward_qk(x[:, :2], k, v), lambda: binding.forward_qk(x[:1], k, v), lambda: binding.gemm(a, a),
        lambda: binding.gemm(a, b, b_layout="kk"), lambda: binding.gemm(a, b, torch.empty_like(a)), lambda: binding.gemm(a, b.transpose(1, 2)), lambda: binding.softmax_rows(s.T, 0.5),
        lambda: binding.softmax_rows(s, 0.5, s[:3]), lambda: binding.softmax_rows(s, -1.0), lambda: binding.forward(t(1, 1, 8, 32), t(1, 1, 8, 32), t(1, 1, 8, 32)),
        lambda: binding.forward(q, k, v, q), lambda: binding.softmax_rows(t(3, 12), 0.5), lambda: binding.forward(q[:0], k[:0], v[:0]), lambda: binding.forward(None, k, v),
    ]


def _outcome(call):
    try:
        return call()
    except Exception as e:
        return type(e), str(e)


def test_without_a_gpu_the_same_errors(binding, monkeypatch):
    torch = importlib.import_module("torch")
    direct = [_outcome(c) for c in _calls(torch, binding, "cpu")]
    monkeypatch.setattr(binding, "_fast", binding._NoFast)
    assert direct == [_outcome(c) for c in _calls(torch, binding, "cpu")]
    assert all(isinstance(x, tuple) for x in direct)


@pytest.mark.gpu
def test_the_usual_calls_give_what_binding_gives(binding, monkeypatch):
    torch = importlib.import_module("torch")
    direct = [_outcome(c) for c in _calls(torch, binding, "cuda")]
    fast = binding._fast
    assert not isinstance(fast, binding._LazyFast) and fast is not binding._NoFast
    monkeypatch.setattr(binding, "_fast", binding._NoFast)
    for i, (x, y) in enumerate(zip(direct, [_outcome(c) for c in _calls(torch, binding, "cuda")])):
        assert torch.equal(x.view(torch.int16), y.view(torch.int16)) if torch.is_tensor(x) else x == y, i
    assert sum(map(torch.is_tensor, direct)) == 9
    assert binding.last_device_status()[0] == 0


@pytest.mark.gpu
def test_what_is_not_usual_is_left_to_binding(binding):
    """Non-contiguous, other types, subclasses, wrapped tensors, a mode that watches operations: None, and nothing launched."""
    torch = importlib.import_module("torch")
    from torch.utils._python_dispatch import TorchDispatchMode

    class Watch(TorchDispatchMode):
        def __torch_dispatch__(self, func, types, args=(), kwargs=None):
            return func(*args, **(kwargs or {}))

    class Sub(torch.Tensor):
        pass

    q = torch.zeros(1, 2, 64, 64, dtype=torch.bfloat16, device="cuda")
    binding.forward(q, q, q)
    before, fast = binding.last_kernel(), binding._fast
    assert fast.attn(q, q, q, None, False, False).shape == q.shape
    for bad in (q.transpose(1, 2), q.float(), q.cpu(), q.as_subclass(Sub), q[0], q[..., :32], torch.empty(0, 2, 64, 64, dtype=torch.bfloat16, device="cuda"), None, 3):
        assert fast.attn(bad, q, q, None, False, False) is None and fast.attn(q, bad, q, None, False, False) is None
        assert bad is None or fast.attn(q, q, q, bad, False, False) is None
    with Watch():
        assert fast.attn(q, q, q, None, False, False) is None and fast.softmax(q, 1.0, None) is None and fast.gemm(q[0], q[0], None, "kn") is None
    seen = []
    torch.vmap(lambda x: (seen.append(fast.attn(x, x, x, None, False, False)), x)[1])(torch.stack([q, q]))
    assert seen == [None]
    assert fast.softmax(q, 1, None) is None and fast.gemm(q[0], q[0], None, 0) is None
    assert binding.last_kernel() == before and binding.last_device_status()[0] == 0


@pytest.mark.gpu
def test_a_refusal_is_raised_by_the_entry_that_met_it(binding):
    """The library is entered once: a second entry could succeed where the first one met, and took, an error of CUDA's."""
    import ctypes

    torch = importlib.import_module("torch")
    q, a = torch.zeros(1, 2, 64, 64, dtype=torch.bfloat16, device="cuda"), torch.zeros(64, 64, dtype=torch.bfloat16, device="cuda")
    binding.forward(q, q, q)                                  # (loads the module)
    handle, entered = binding.lib(), []
    fail = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p)(lambda call: entered.append(call) or binding.ERR_CUDA)
    address = lambda f: ctypes.cast(f, ctypes.c_void_p).value
    binding._fast.bind(address(fail), address(fail), address(fail), binding._refused)
    try:
        before = binding.last_kernel(), binding.last_grid()
        for call, where in ((lambda: binding.forward(q, q, q), "attn_forward"), (lambda: binding.forward(q, q, q, causal=True), "attn_forward_causal"),
                            (lambda: binding.forward_qk(q, q, q), "attn_forward_qk"), (lambda: binding.gemm(a, a), "gemm_forward"),
                            (lambda: binding.softmax_rows(a, 1.0), "softmax_rows_forward")):
            entered.clear()
            with pytest.raises(binding.AttnError) as err:
                call()
            assert err.value.code == binding.ERR_CUDA and where in str(err.value) and len(entered) == 1
        assert before == (binding.last_kernel(), binding.last_grid())
    finally:
        binding._fast.bind(address(handle.attn_forward_call), address(handle.gemm_forward_call), address(handle.softmax_rows_forward_call), binding._refused)
    assert binding.forward(q, q, q).shape == q.shape and binding.last_device_status()[0] == 0
