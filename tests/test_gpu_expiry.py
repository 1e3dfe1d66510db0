"""The way out of an expired wait in the kernels of whole tiles: nothing is issued and nothing passed on after it."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("own_status", [False, True])
def test_a_warp_whose_wait_expired_issues_nothing(own_status):
    """A warp of the library's self-test waits, as the warps that issue products do, on a barrier nothing arrives at (half a second).
    None of its lanes may issue afterwards, its next wait ends at once, and the expiry is reported in the caller's status words or in the
    device-wide record; a warp whose phase had completed issues a product, whose drain leaves it complete.  The kernels that wait this way then compute as before."""
    torch = pytest.importorskip("torch")
    from paper_2609_10937_b200 import binding

    assert binding.last_device_status()[0] == 0
    status = torch.zeros(4, dtype=torch.int32, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    assert binding.lib().attn_selftest_issue_expiry_to(status.data_ptr() if own_status else None, stream) == 0
    code, detail = binding.status_read(status, None) if own_status else binding.last_device_status()
    assert code == binding.ERR_DEVICE_TIMEOUT
    assert detail[0] == 1 and detail[1] == (5 << 24) | (10 << 16) | 0x7E57 and detail[2] == 0
    assert binding.last_device_status()[0] == 0 and binding.status_read(status, None) == (0, [0, 0, 0, 0])
    gen = torch.Generator(device="cuda").manual_seed(3)
    for d, H, L, causal in ((64, 148, 600, False), (64, 20, 700, True), (128, 148, 600, False), (128, 148, 600, True)):
        q, k, v = (torch.randn(1, H, L, d, generator=gen, device="cuda").to(torch.bfloat16) for _ in range(3))
        s = q[0, 7].double() @ k[0, 7].double().T / d ** 0.5
        if causal:
            s = s.masked_fill(torch.ones(L, L, dtype=torch.bool, device="cuda").triu(1), float("-inf"))
        ref = torch.softmax(s, dim=-1) @ v[0, 7].double()
        got = binding.forward(q, k, v, causal=causal)[0, 7].double()
        assert float((got - ref).norm() / ref.norm()) <= 5e-3
    assert binding.last_device_status()[0] == 0
