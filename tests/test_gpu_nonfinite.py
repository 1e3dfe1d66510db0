"""Scores that are no numbers: a row of the result is NaN exactly where plain softmax attention in 64 bits gives NaN."""
import math

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


# whole tiles of 256 and of 128 rows, clusters, tiles cut over the machine, few rows; ragged last key tiles
@pytest.mark.parametrize("d,H,Lq,Lk,causal", [
    (64, 148, 1024, 1024, False), (64, 148, 300, 513, False), (64, 4, 2048, 2048, False), (64, 1, 256, 256, False), (64, 300, 256, 200, False), (64, 1, 4096, 4096, False),
    (64, 20, 1111, 1111, True), (64, 128, 700, 700, True), (64, 9, 1111, 1111, True), (64, 2, 6144, 6144, True),
    (128, 148, 1024, 1024, False), (128, 300, 129, 129, False), (128, 4, 2048, 2048, False), (128, 16, 512, 512, False), (128, 1, 4096, 4096, False),
    (128, 128, 1024, 1024, True), (128, 16, 1024, 1024, True), (128, 3, 4096, 4096, True), (128, 20, 1111, 1111, True),
    (64, 32, 3, 900, False), (128, 32, 16, 900, False)])
def test_rows_are_nan_where_plain_attention_is(env, d, H, Lq, Lk, causal):
    """One element of K is NaN or infinite, in a key of each residue mod 16 in turn (the kernels evaluate the exponentials of a
    group of 16 keys in two ways), in the first, a middle or the last key tile.  An infinite element gives scores of +inf (NaN
    rows) and -inf (weight 0) by the sign of the query's element."""
    torch, binding = env
    gen = torch.Generator(device="cuda").manual_seed(H + Lq + Lk + d)
    q, k0, v = (torch.randn(1, H, n, d, generator=gen, device="cuda").to(torch.bfloat16) for n in (Lq, Lk, Lk))
    keep = torch.ones((Lq, Lk), dtype=torch.bool, device="cuda").tril() if causal else None
    head = H // 2
    tiles = (Lk + 127) // 128
    for what in (math.nan, math.inf, -math.inf):
        for r in range(16):
            tile = (0, tiles // 2, tiles - 1)[r % 3]
            key = min(tile * 128 + (r * 5 % 8) * 16 + r, Lk - 1)
            k = k0.clone()
            k[0, head, key, 0] = what
            out = binding.forward(q, k, v, causal=True) if causal else binding.forward_qk(q, k, v)
            s = q[0, head].double() @ k[0, head].double().T / d ** 0.5
            if causal:
                s = s.masked_fill(~keep, -math.inf)
            ref = torch.softmax(s, dim=-1) @ v[0, head].double()
            bad, got = ref.isnan().any(-1), out[0, head].double()
            assert torch.equal(got.isnan().all(-1), bad) and torch.equal(got.isfinite().all(-1), ~bad), (what, key)
            if not bad.all():
                assert float((got[~bad] - ref[~bad]).norm() / ref[~bad].norm()) <= 5e-3, (what, key)
            out[0, head] = 0
            assert out.isfinite().all(), (what, key)
    assert binding.last_device_status()[0] == 0
