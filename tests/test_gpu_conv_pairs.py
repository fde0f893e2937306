"""3x3 layers large enough to run as CTA pairs, with an odd number of tiles per frame, ragged edges and one or several channel
blocks: small whole numbers, whose sums are exact in any order, so the result equals the FFMA kernel's bit for bit."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,W,Cin,Cout", [
    (3, 130, 310, 64, 128),        # 128-channel blocks: 3 x 351 tiles
    (1, 250, 505, 128, 128),       # 1024 tiles, the last row and column cut
    (1, 165, 361, 64, 384),        # three blocks of 128 channels
    (2, 170, 550, 64, 256),        # a 256-channel block: 2 x 759 tiles
])
@pytest.mark.parametrize("in_bf16", [False, True])
def test_pair_layers_are_exact(B, H, W, Cin, Cout, in_bf16):
    import torch
    from paper_2602_00608_b200 import binding as vd
    g = torch.Generator(device="cuda").manual_seed(B * 1000 + H)
    x = torch.randint(-4, 5, (B, H, W, Cin), device="cuda", generator=g).to(torch.bfloat16 if in_bf16 else torch.float32)
    w = torch.randint(-2, 3, (Cout, Cin, 3, 3), device="cuda", generator=g).to(torch.bfloat16)
    kw = dict(out_dtype=vd.VD_F32, bf16_operands=True)
    got = vd.op_conv2d(x, w, impl=vd.VD_IMPL_TC, **kw)
    want = vd.op_conv2d(x, w, impl=vd.VD_IMPL_SIMT, **kw)
    assert torch.equal(got, want)
