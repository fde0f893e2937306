"""The register-tiled fp32 convolution against the oracle's plain operators, at the sizes where it can go wrong: tiles cut by
the image edge, images smaller than a tile, channel counts that leave a chunk part empty, K divided among thread groups
and clusters, the four parities of the phase-collapsed upsampling form, the frame head."""
import pytest

from tests.test_gpu_ops import _conv_case, env                      # noqa: F401  (env is a fixture)
from tests.util import rel_l2

pytestmark = pytest.mark.gpu

CASES = [
    dict(B=1, H=1, W=1, Cin=16, Cout=32, k=3, upsample=False, prologue=True, silu=True, residual=False),
    dict(B=1, H=8, W=8, Cin=512, Cout=64, k=3, upsample=False, prologue=True, silu=True, residual=True),    # 8-row tile, cluster of 8
    dict(B=2, H=17, W=9, Cin=36, Cout=96, k=3, upsample=False, prologue=True, silu=True, residual=True),    # part-empty chunk
    dict(B=3, H=33, W=50, Cin=32, Cout=32, k=3, upsample=False, prologue=True, silu=True, residual=True),   # no cluster
    dict(B=1, H=9, W=7, Cin=4, Cout=512, k=3, upsample=False, prologue=False, silu=False, residual=False),
    dict(B=3, H=33, W=21, Cin=4, Cout=256, k=3, upsample=False, prologue=False, silu=False, residual=False),      # thin: 64-pixel blocks
    dict(B=2, H=19, W=23, Cin=8, Cout=128, k=3, upsample=False, prologue=False, silu=False, residual=False),      # thin: 32-pixel blocks
    dict(B=2, H=5, W=13, Cin=8, Cout=128, k=3, upsample=False, prologue=False, silu=False, residual=False),       # thin: 16-pixel blocks
    dict(B=1, H=12, W=10, Cin=512, Cout=96, k=1, upsample=False, prologue=True, silu=False, residual=False),
    dict(B=2, H=21, W=30, Cin=64, Cout=32, k=1, upsample=False, prologue=False, silu=False, residual=True),
    dict(B=1, H=1, W=2, Cin=64, Cout=32, k=3, upsample=2, prologue=False, silu=False, residual=False),
    dict(B=2, H=8, W=11, Cin=128, Cout=64, k=3, upsample=2, prologue=False, silu=False, residual=False),
    dict(B=1, H=35, W=26, Cin=32, Cout=32, k=3, upsample=2, prologue=True, silu=True, residual=False),
    dict(B=2, H=19, W=23, Cin=128, Cout=3, k=3, upsample=False, prologue=True, silu=True, residual=False, out_nchw=True),
    dict(B=2, H=135, W=290, Cin=36, Cout=3, k=3, upsample=False, prologue=True, silu=True, residual=False, out_nchw=True),   # 32-pixel tiles
    dict(B=1, H=592, W=128, Cin=64, Cout=4, k=3, upsample=False, prologue=True, silu=True, residual=False, out_nchw=True),   # and a cluster
    dict(B=1, H=5, W=3, Cin=20, Cout=3, k=3, upsample=False, prologue=False, silu=False, residual=False, out_nchw=True),
]


@pytest.mark.parametrize("case", CASES)
def test_conv_f32_matches_oracle(env, case):                        # noqa: F811
    _, _, vd, _ = env
    got, want = _conv_case(env, seed=61, in_bf16=False, out_bf16=False, impl=vd.VD_IMPL_SIMT, bf16_ops=False, **case)
    assert got.shape == want.shape
    # rounding of K fp32 sums in sequence: 2^-24 / sqrt(3) * sqrt(K / 2) of the result at K = 4608, less when K is divided
    assert rel_l2(got, want) <= 2e-6
