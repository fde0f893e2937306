"""Attention on the FP32 pipes at the edges of its key tile, its queries per CTA and its loads."""
import math

import pytest

pytestmark = pytest.mark.gpu


# T: one token, around the 64-key tile, the last size of two queries per CTA (592) and the first of four; C: one lane group,
# a partly used one, all four.  The sums of C products and of T weights are fp32: 2e-6 covers sqrt(C + T) roundings of 6e-8.
@pytest.mark.parametrize("B,T,C", [(1, 1, 32), (2, 63, 96), (1, 64, 512), (1, 65, 160), (1, 592, 32), (1, 593, 512), (3, 300, 128)])
def test_attention_matches_double(B, T, C):
    torch = pytest.importorskip("torch")
    from paper_2602_00608_b200 import binding as vd

    torch.manual_seed(T * 7 + C)
    qkv = torch.randn(B, T, 3 * C, device="cuda")
    qkv[:, :, :C] *= 2.0
    scale = 1.0 / math.sqrt(C)
    got = vd.op_attention(qkv, C, scale, vd.VD_IMPL_SIMT).double()
    q, k, v = qkv.double().split(C, dim=2)
    want = torch.softmax(q @ k.transpose(1, 2) * scale, dim=2) @ v
    err = ((got - want).norm() / want.norm()).item()
    assert err <= 2e-6, err
