"""GroupNorm statistics of several samples in one pass, against 64 bits: samples that do not fill a chunk, widths that do not divide
a stage, more than 32 chunks per block, a tensor off the 16-byte grid, an offset; and a sample alone gives the same bits."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vd():
    from paper_2602_00608_b200 import binding
    return binding


@pytest.mark.parametrize("B,H,W,C,G,bf16,offset,shifted", [
    (2, 1, 5, 20, 5, False, False, False), (3, 33, 41, 36, 3, False, True, False), (2, 67, 71, 1000, 250, False, False, False),
    (34, 64, 74, 20, 5, False, False, False),                   # 296 chunks of 16 pixels: 34 chunks per block
    (5, 97, 101, 24, 3, True, True, False), (3, 150, 170, 128, 32, True, True, False), (2, 90, 100, 512, 32, True, False, False),
    (3, 50, 61, 20, 5, True, False, False), (3, 50, 61, 24, 3, True, False, True),      # pieces of 8 bytes: the other kernel
    (3, 130, 140, 256, 32, False, True, False),
])
def test_gn_stats_of_several_samples(vd, B, H, W, C, G, bf16, offset, shifted):
    import torch
    g = torch.Generator(device="cuda").manual_seed(C + B)
    rnd = lambda *s: torch.randn(*s, device="cuda", generator=g)
    x = (rnd(B, H, W, C) * 1.5 + 3.0).to(torch.bfloat16 if bf16 else torch.float32)
    if shifted:                                                  # 8 bytes off the 16-byte grid
        store = torch.empty(x.numel() + 8, dtype=x.dtype, device="cuda")
        x = store[4:4 + x.numel()].view(x.shape).copy_(x)
        assert x.data_ptr() % 16 == 8
    gamma, beta, off = 1 + 0.1 * rnd(C), 0.1 * rnd(C), rnd(C) if offset else None
    sc, sh = vd.op_gn_stats(x, gamma, beta, G, 1e-6, offset=off)
    t = (x.double() + (off.double() if offset else 0.0)).view(B, H * W, G, C // G)
    mean, var = t.mean(dim=(1, 3)), t.var(dim=(1, 3), unbiased=False)
    want = gamma.double() * (var + 1e-6).rsqrt().repeat_interleave(C // G, dim=1)
    wsh = beta.double() - mean.repeat_interleave(C // G, dim=1) * want + (off.double() * want if offset else 0.0)
    assert torch.allclose(sc.double(), want, rtol=2e-5, atol=0)  # fp32 sums of up to 1e6 terms about a reference value, in blocks
    assert torch.allclose(sh.double(), wsh, rtol=2e-5, atol=2e-5)
    if not shifted:
        one = vd.op_gn_stats(x[B - 1:].contiguous(), gamma, beta, G, 1e-6, offset=off)
        assert torch.equal(sc[B - 1:], one[0]) and torch.equal(sh[B - 1:], one[1])
