"""GroupNorm statistics of single frames and of several at once are two kernels (handles of max_batch 1 and of more).  Both, against 64
bits: each storage type, wide and narrow layers, an offset per channel, a mean far from zero, groups without variance; the same
bits every time, alone and in a batch.  (Samples of up to 3 million elements in 16-channel columns are a third kernel's.)"""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vd():
    from paper_2602_00608_b200 import binding
    return binding


def want_of(x, gamma, beta, G, eps, off):
    B, H, W, C = x.shape
    t = (x.double() + (off.double() if off is not None else 0.0)).view(B, H * W, G, C // G)
    mean, var = t.mean(dim=(1, 3)), t.var(dim=(1, 3), unbiased=False)
    scale = gamma.double() * (var + eps).rsqrt().repeat_interleave(C // G, dim=1)
    return scale, beta.double() - mean.repeat_interleave(C // G, dim=1) * scale + (off.double() * scale if off is not None else 0.0)


@pytest.mark.parametrize("single", [False, True])
@pytest.mark.parametrize("B,H,W,C,G,bf16,offset,mean", [
    (1, 77, 77, 512, 32, False, False, 0.5), (1, 77, 77, 512, 32, True, True, 0.5), (2, 251, 203, 64, 8, False, True, 0.5),
    (1, 240, 360, 256, 32, False, False, 0.5), (1, 200, 131, 128, 32, True, True, 0.5), (3, 45, 61, 1000, 250, False, False, 0.5),
    (1, 70, 71, 20, 5, False, True, 0.5), (2, 70, 71, 24, 3, True, True, 0.5), (1, 70, 71, 20, 5, True, False, 0.5), (1, 160, 151, 128, 32, False, False, 300.0),
])
def test_gn_stats_of_either_kernel(vd, single, B, H, W, C, G, bf16, offset, mean):
    import torch
    g = torch.Generator(device="cuda").manual_seed(C + H)
    rnd = lambda *s: torch.randn(*s, device="cuda", generator=g)
    x = (rnd(B, H, W, C) + mean).to(torch.bfloat16 if bf16 else torch.float32)
    gamma, beta, off = 1 + 0.1 * rnd(C), 0.1 * rnd(C), rnd(C) if offset else None
    got = vd.op_gn_stats(x, gamma, beta, G, 1e-6, offset=off, single=single)
    want = want_of(x, gamma, beta, G, 1e-6, off)
    # fp32 sums of up to 1e6 terms about a reference value, in blocks; the mean itself is rounded to 2^-24 of it
    assert torch.allclose(got[0].double(), want[0], rtol=2e-5, atol=0)
    assert torch.allclose(got[1].double(), want[1], rtol=2e-5, atol=2e-5 + 2.0 ** -23 * mean)
    for part in (x, x[B - 1:].contiguous()):
        again = vd.op_gn_stats(part, gamma, beta, G, 1e-6, offset=off, single=single)
        assert torch.equal(got[0][-part.shape[0]:], again[0]) and torch.equal(got[1][-part.shape[0]:], again[1])


@pytest.mark.parametrize("single", [False, True])
def test_groups_without_variance(vd, single):
    import torch
    g = torch.Generator(device="cuda").manual_seed(3)
    const = torch.rand(2, 8, device="cuda", generator=g).mul_(10).sub_(5).repeat_interleave(16, dim=1)
    x = const[:, None, None, :].expand(2, 160, 151, 128).contiguous()
    gamma, beta = torch.linspace(0.9, 1.1, 128, device="cuda"), torch.linspace(-0.1, 0.1, 128, device="cuda")
    sc, sh = vd.op_gn_stats(x, gamma, beta, 8, 0.25, single=single)
    assert torch.allclose(sc, (gamma * 2).expand(2, 128), rtol=1e-6, atol=0)         # 1 / sqrt(0.25)
    assert torch.allclose(sh, beta - const * 2 * gamma, rtol=1e-5, atol=1e-6)
