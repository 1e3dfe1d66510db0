"""The softmax weights of the attention kernels: how exact they are, seen through outputs that lie beside a rounding boundary."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_10937_b200 import binding

    binding.lib()   # must load: there is no fallback
    return torch, binding


@pytest.mark.parametrize("d,H,L,causal,below", [(64, 148, 1024, False, 3), (64, 74, 6144, False, 18), (64, 4, 4096, False, 12), (64, 1, 8192, False, 24),
                                                (128, 148, 1024, False, 3), (128, 4, 4096, False, 12), (128, 16, 512, False, 2),
                                                (128, 128, 1024, True, 1), (128, 148, 2048, True, 1)])
def test_equal_weights_are_as_exact_as_their_shares(env, d, H, L, causal, below):
    """Scores of zero: every weight is 1, and the last row is the mean of V.  V holds 1 and 1 + 2^-7 so often that the mean lies
    `below` counts (2^-7 / L each, 7.6e-6 at L = 1024) under the midpoint of the two, and rounds to 1; sums and products of these values are exact in
    fp32.  A weight that the cubic for 2^f gives is 7.1e-5 too small (in the sum; as bf16 it is 1), so the mean comes out too large by that
    times the cubic's share of the keys: 1.8e-5 at a quarter, which stays below, 2.7e-5 at three eighths, which does not.
    Causal at d = 128: none of the keys ahead of the diagonal tile, a quarter of that tile's 128 (1.8e-5 * 128 / L)."""
    torch, binding = env
    q = torch.zeros(1, H, L, d, dtype=torch.bfloat16, device="cuda")
    k = torch.randn(1, H, L, d, generator=torch.Generator(device="cuda").manual_seed(L), device="cuda").to(torch.bfloat16)
    v = torch.ones_like(q)
    high = torch.randperm(L, generator=torch.Generator(device="cuda").manual_seed(d), device="cuda")[: L // 2 - below]
    v[:, :, high] = 1.0 + 2.0 ** -7
    out = binding.forward(q, k, v, causal=causal)
    torch.cuda.synchronize()
    assert binding.last_device_status()[0] == 0
    rows = out[0, :, L - 1] if causal else out[0]
    assert (rows == 1.0).all()
