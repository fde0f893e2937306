"""GroupNorm statistics of small samples (the cluster kernel) against the oracle's two-pass statistics: fewer pixels than
CTAs, pixel counts that no thread layout divides, every group width the kernel has, both sides of the size at which the
other kernel takes over, and a per-channel offset."""
import numpy as np
import pytest

from tests import util
from tests.test_gpu_ops import _gn_case, _rng, env                  # noqa: F401  (env is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,W,C,G,bf16", [
    (1, 1, 2, 512, 32, False), (2, 3, 3, 256, 32, True), (1, 19, 27, 128, 32, False), (3, 16, 16, 512, 32, True),
    (1, 77, 76, 512, 32, False), (1, 77, 77, 512, 32, False),       # 2 995 712 and 3 035 648 elements
])
def test_gn_stats_of_small_samples(env, B, H, W, C, G, bf16):       # noqa: F811
    sc, sh, wsc, wsh = _gn_case(env, 27, B, H, W, C, G, bf16)
    np.testing.assert_allclose(sc, wsc, rtol=2e-5)                  # fp32 sums of 1e5 terms about a reference value
    np.testing.assert_allclose(sh, wsh, rtol=2e-5, atol=2e-5)


def test_gn_stats_of_a_small_sample_with_an_offset_and_in_a_batch(env):       # noqa: F811
    torch, ref, vd, synth = env
    r = _rng(33)
    B, H, W, C, G = 3, 11, 7, 256, 32
    x = (r.standard_normal((B, C, H, W)) * 1.3 + 40.0).astype(np.float32)
    off = r.uniform(-2.0, 2.0, C).astype(np.float32)
    gamma, beta = r.uniform(0.9, 1.1, C).astype(np.float32), r.uniform(-0.1, 0.1, C).astype(np.float32)
    want, _, _ = ref.groupnorm(x + off[None, :, None, None], gamma, beta, G, 1e-6, return_stats=True)
    xd, dev = util.nchw_to_dev_nhwc(x, torch.float32), lambda a: torch.from_numpy(a).cuda()
    sc, sh = vd.op_gn_stats(xd, dev(gamma), dev(beta), G, 1e-6, offset=dev(off))
    one = vd.op_gn_stats(xd[2:3].contiguous(), dev(gamma), dev(beta), G, 1e-6, offset=dev(off))
    torch.cuda.synchronize()
    assert torch.equal(sc[2:3], one[0]) and torch.equal(sh[2:3], one[1])
    got = x * sc.cpu().numpy()[:, :, None, None] + sh.cpu().numpy()[:, :, None, None]
    assert util.rel_l2(got, want) <= 2e-5       # scale x ~ 40: 2^-24 x 40 per element before the shift takes it off


@pytest.mark.parametrize("P", [1, 3, 7])
@pytest.mark.parametrize("C,G,bf16", [(128, 32, True), (256, 32, False), (512, 32, True)])
def test_gn_stats_of_fewer_pixels_than_ctas(env, P, C, G, bf16):    # noqa: F811
    """CTAs of the cluster without a pixel send their (zero) sums at once: nothing to read hides the wait for the first CTA."""
    sc, sh, wsc, wsh = _gn_case(env, 41, 3, 1, P, C, G, bf16)
    np.testing.assert_allclose(sc, wsc, rtol=2e-5)
    np.testing.assert_allclose(sh, wsh, rtol=2e-5, atol=2e-5)
