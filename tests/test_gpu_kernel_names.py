"""Which kernel a call ran as, by its name: the lines of the dispatch rules, and kernels that share an attn_kernel number."""
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


PIPE, NARROW, FWD = "attn_pipe_kernel", "attn_narrow_kernel", "attn_fwd_kernel"


@pytest.mark.parametrize("d,H,Lq,Lk,causal,name", [
    # d = 128, not causal: waves of whole tiles; one wave from four key steps on three quarters of 148 SMs; tiles the plan would cut
    (128, 300, 129, 129, False, f"{PIPE}<128,0>"), (128, 160, 257, 1, False, f"{PIPE}<128,0>"), (128, 150, 300, 128, False, f"{PIPE}<128,0>"),
    (128, 152, 640, 640, False, f"{PIPE}<128,0>"), (128, 111, 200, 900, False, f"{PIPE}<128,0>"), (128, 111, 256, 512, False, f"{PIPE}<128,0>"),
    (128, 110, 256, 900, False, f"{FWD}<128,128,2,0,0,0>"), (128, 111, 256, 384, False, f"{FWD}<128,128,2,0,0,0>"), (128, 222, 640, 640, False, f"{PIPE}<128,0>"),
    (128, 16, 512, 512, False, f"{NARROW}<128,0,1>"), (128, 4, 4096, 4096, False, f"{FWD}<128,128,2,0,1,1>"), (128, 1, 16384, 16384, False, f"{FWD}<128,128,2,0,0,0>"),
    # d = 64: the same up to the steps from which the plan's kernel is the faster one
    (64, 74, 900, 900, False, f"{PIPE}<64,0>"), (64, 148, 1024, 1024, False, f"{PIPE}<64,0>"), (64, 60, 300, 449, False, f"{PIPE}<64,0>"),
    (64, 148, 256, 1280, False, f"{PIPE}<64,0>"), (64, 148, 256, 1281, False, f"{FWD}<64,128,2,0,0,0>"), (64, 74, 1024, 2100, False, f"{PIPE}<64,0>"),
    (64, 74, 1024, 2304, False, f"{FWD}<64,128,2,0,0,0>"), (64, 160, 3500, 3500, False, f"{PIPE}<64,0>"), (64, 160, 3500, 4000, False, f"{FWD}<64,128,2,0,0,0>"),
    (64, 148, 640, 640, False, f"{FWD}<64,128,2,0,0,0>"), (64, 148, 640, 600, False, f"{PIPE}<64,0>"), (64, 148, 640, 256, False, f"{PIPE}<64,0>"),
    (64, 148, 600, 1500, False, f"{FWD}<64,128,2,0,0,0>"), (64, 148, 600, 1300, False, f"{PIPE}<64,0>"), (64, 148, 641, 640, False, f"{PIPE}<64,0>"), (64, 128, 896, 896, False, f"{PIPE}<64,0>"),
    (64, 148, 896, 896, False, f"{FWD}<64,128,2,0,0,0>"), (64, 111, 1300, 1300, False, f"{PIPE}<64,0>"), (64, 37, 6144, 6144, False, f"{NARROW}<64,0,2>"),
    (64, 296, 300, 300, False, f"{NARROW}<64,0,2>"), (64, 16, 512, 512, False, f"{NARROW}<64,0,1>"), (64, 8, 1000, 1000, False, f"{FWD}<64,128,2,0,1,1>"),
    # causal
    (128, 152, 640, 640, True, f"{PIPE}<128,1>"), (128, 20, 1111, 1111, True, f"{NARROW}<128,1,1>"), (128, 8, 1000, 1000, True, f"{FWD}<128,128,2,1,1,1>"),
    (128, 3, 4096, 4096, True, f"{FWD}<128,128,2,1,0,0>"), (64, 128, 700, 700, True, f"{NARROW}<64,1,2>"), (64, 20, 1111, 1111, True, f"{NARROW}<64,1,1>"),
    # few rows
    (64, 32, 3, 900, False, "attn_decode_kernel<64,1,1>"), (128, 32, 16, 900, False, "attn_decode_kernel<128,1,0>")])
def test_a_call_runs_as_the_kernel_of_its_rule(env, d, H, Lq, Lk, causal, name):
    """On the 148 SMs that the rules' lines were measured on.  Every element of some heads against fp64; the bound per element is that of
    test_causal_whole_tiles_match_the_reference."""
    torch, binding = env
    if binding.hw_desc_query(0).num_units != 148:
        pytest.skip("the lines are those of 148 SMs")
    gen = torch.Generator(device="cuda").manual_seed(H + Lq + Lk + d)
    q, k, v = (1.5 * torch.randn(1, H, n, d, generator=gen, device="cuda") for n in (Lq, Lk, Lk))
    q, k, v = (x.to(torch.bfloat16) for x in (q, k, v))
    out = binding.forward(q, k, v, causal=True) if causal else binding.forward_qk(q, k, v)
    assert binding.last_kernel_name() == name
    assert binding.last_device_status()[0] == 0
    for h in sorted({0, H // 2, H - 1}):
        s = q[0, h].double() @ k[0, h].double().T / d ** 0.5
        if causal:
            s = s.masked_fill(torch.ones((Lq, Lk), dtype=torch.bool, device="cuda").triu(1), -math.inf)
        p, vd, got = torch.softmax(s, dim=-1), v[0, h].double(), out[0, h].double()
        ref, spread = p @ vd, p @ vd.abs()
        assert ((got - ref).abs() <= (2.0 ** -8 + 2.0 ** -13) * spread + 2.0 ** -8 * ref.abs() + 1e-6).all(), h
        assert float((got - ref).norm() / ref.norm()) <= 5e-3, h


@pytest.mark.parametrize("H,L", [(152, 640), (300, 257), (148, 385), (64, 2048), (128, 1111)])
def test_causal_whole_tiles_whose_references_move_in_every_step(env, H, L):
    """attn_pipe_kernel, causal: blocks of 64 keys each 7 above the one before.  Every element of some heads against fp64, NaN-filled
    output, the same bits again; the bound per element is that of test_causal_whole_tiles_match_the_reference."""
    torch, binding = env
    d = 128
    gen = torch.Generator(device="cuda").manual_seed(H + L)
    q, k, v = (1.5 * torch.randn(1, H, L, d, generator=gen, device="cuda") for _ in range(3))
    q[..., 0] = 8.0
    k[..., 0] = 7.0 * (torch.arange(L, device="cuda") // 64) * d ** 0.5 / 8.0
    q, k, v = (x.to(torch.bfloat16) for x in (q, k, v))
    out = binding.forward(q, k, v, torch.full_like(q, float("nan")), causal=True)
    assert binding.last_kernel_name() == "attn_pipe_kernel<128,1>" and binding.last_kernel() == binding.KERNEL_CAUSAL_TILES
    keep = torch.ones((L, L), dtype=torch.bool, device="cuda").tril()
    for h in sorted({0, 1, H // 2, H - 1}):
        p = torch.softmax((q[0, h].double() @ k[0, h].double().T / d ** 0.5).masked_fill(~keep, -math.inf), dim=-1)
        vd, got = v[0, h].double(), out[0, h].double()
        ref, spread = p @ vd, p @ vd.abs()
        assert ((got - ref).abs() <= (2.0 ** -8 + 2.0 ** -13) * spread + 2.0 ** -8 * ref.abs() + 1e-6).all(), h
        assert float((got - ref).norm() / ref.norm()) <= 5e-3, h
    for _ in range(3):
        assert torch.equal(binding.forward(q, k, v, causal=True).view(torch.int16), out.view(torch.int16))
    assert binding.last_device_status()[0] == 0


def test_products_and_row_softmax_are_named(env):
    torch, binding = env
    a = torch.zeros(512, 512, dtype=torch.bfloat16, device="cuda")
    binding.gemm(a, a)
    assert binding.last_kernel_name() == "gemm_small_kernel<1>"
    big = torch.zeros(4096, 1024, dtype=torch.bfloat16, device="cuda")
    binding.gemm(big, big, b_layout="nk")
    assert binding.last_kernel_name() == "gemm_pair_kernel<0,256>" and binding.last_kernel() == binding.KERNEL_GEMM_PAIR
    binding.softmax_rows(a, 1.0)
    assert binding.last_kernel_name() == "softmax_rows" and binding.last_kernel() == binding.KERNEL_SOFTMAX
