"""The single-precision convolution on the tensor cores, at the sizes where it can go wrong: tiles cut by the image edge, one to
eight CTAs that share K, more taps than accumulators, the four parities of the upsampling form.

Small whole numbers are exact in one bf16 number and their sums in fp32, so the result is that of a 64-bit convolution bit for bit;
numbers with 24 significant bits, alone in their sums, show that the operands keep all of them."""
import pytest

from tests.test_gpu_conv_split import exact_conv, ints, vd            # noqa: F401  (vd is a fixture)

pytestmark = pytest.mark.gpu

# B, H, W, Cin, Cout, up
SHAPES = [
    (1, 1, 1, 32, 32, 0), (2, 17, 9, 64, 96, 0), (1, 16, 8, 256, 32, 0), (1, 8, 8, 512, 512, 0), (3, 33, 50, 32, 32, 0), (1, 30, 21, 96, 64, 0),
    (1, 24, 24, 512, 512, 0), (1, 61, 57, 128, 128, 0), (2, 33, 30, 96, 192, 0),
    (1, 3, 2, 64, 32, 2), (2, 17, 9, 128, 64, 2), (1, 8, 8, 512, 512, 2), (2, 33, 19, 32, 32, 2),
]


@pytest.mark.parametrize("shape", SHAPES)
def test_whole_numbers_are_exact(vd, shape):                          # noqa: F811
    import torch
    B, H, W, Cin, Cout, up = shape
    g = torch.Generator(device="cuda").manual_seed(H * 1000 + W * 10 + Cin)
    x, w, bias = ints(g, -4, 4, B, H, W, Cin), ints(g, -2, 2, Cout, Cin, 3, 3), ints(g, -8, 8, Cout)
    scale, shift = 2.0 ** ints(g, -1, 1, B, Cin), ints(g, -1, 1, B, Cin)
    want = exact_conv(x.double() * scale[:, None, None, :].double() + shift[:, None, None, :].double(), w, 3, up) + bias.double()
    res = None if up else ints(g, -64, 64, *want.shape)
    got = vd.op_conv2d(x, w, bias, scale, shift, res, upsample=up, impl=vd.VD_IMPL_TC_F32)
    assert torch.equal(got, (want if res is None else want + res.double()).float())


@pytest.mark.parametrize("shape", [(2, 17, 9, 64, 96, 0), (1, 8, 8, 512, 512, 0), (3, 33, 50, 32, 32, 0), (1, 64, 64, 128, 128, 0), (1, 8, 8, 512, 512, 2)])
def test_operands_keep_24_bits(vd, shape):                            # noqa: F811
    """A tap's sum has two truncating steps (2^-23 at most of a sum that grows to its size), a product lacks 2^-24 of itself at most,
    the parts' sum rounds by 2^-24, and at most 26 sums and partials are added with rounding (2^-24 / sqrt(3) each, on a sum that
    grows: sqrt(26 / 2)): two chunks of nine taps in a CTA, eight CTAs."""
    import torch
    B, H, W, Cin, Cout, up = shape
    g = torch.Generator(device="cuda").manual_seed(7)
    rnd = lambda *s: torch.randn(*s, device="cuda", generator=g)
    x, w = rnd(B, H, W, Cin), rnd(Cout, Cin, 3, 3) / (9 * Cin) ** 0.5
    want = exact_conv(x, w, 3, up)
    got = vd.op_conv2d(x, w, upsample=up, impl=vd.VD_IMPL_TC_F32).double()
    bound = 2 * 2.0 ** -23 / 2 + 2 * 2.0 ** -24 + 2.0 ** -24 / 3 ** 0.5 * (26 / 2) ** 0.5
    if up:
        bound += 2.0 ** -24                                           # the sums of up to four weights are rounded once
    assert float((got - want).norm() / want.norm()) <= bound


def wide(g, lo, hi, *shape):
    """Numbers of 24 significant bits, the last one set, of either sign and of sizes 2^lo to 2^hi."""
    import torch
    m = 2 * torch.randint(2 ** 22, 2 ** 23, shape, device="cuda", generator=g) + 1
    e = torch.randint(lo, hi + 1, shape, device="cuda", generator=g)
    sign = 2 * torch.randint(0, 2, shape, device="cuda", generator=g) - 1
    return torch.ldexp((sign * m).double(), (e - 23).double()).float()


@pytest.mark.parametrize("shape", [(1, 19, 21, 32, 32, 0), (1, 8, 8, 512, 512, 0), (1, 11, 5, 64, 32, 2)])
@pytest.mark.parametrize("whole", ["activations", "weights"])
def test_no_bit_of_an_operand_is_lost(vd, shape, whole):              # noqa: F811
    """One tap of one input channel per output channel, times a power of two: the other operand comes back as it was,
    sizes from 2^-110 to 2^100."""
    import torch
    B, H, W, Cin, Cout, up = shape
    g = torch.Generator(device="cuda").manual_seed(11)
    one = 2.0 ** torch.randint(-3, 4, (Cout,), device="cuda", generator=g).float()
    src = torch.randint(0, Cin, (Cout,), device="cuda", generator=g)
    if whole == "activations":
        x, taps = wide(g, -110, 100, B, H, W, Cin), one
    else:
        x, taps = torch.ones(B, H, W, Cin, device="cuda"), wide(g, -110, 100, Cout)
    w = torch.zeros(Cout, Cin, 3, 3, device="cuda")
    w[torch.arange(Cout, device="cuda"), src, 1, 1] = taps
    got = vd.op_conv2d(x, w, upsample=up, impl=vd.VD_IMPL_TC_F32)
    want = x[..., src].double() * taps.double()
    if up:
        want = want.repeat_interleave(2, dim=1).repeat_interleave(2, dim=2)
    assert torch.equal(got.double(), want)


@pytest.mark.parametrize("terms", [1, 2, 4])
def test_sums_of_few_products(vd, terms):                             # noqa: F811
    """Products of 24 by 24 bits, a few per sum: each lacks at most 2^-24 of itself (the parts that are not multiplied); of the partial
    sums, all but the smallest are exact but for truncations of 2^-23 of what they come to (the six of 2^-8 of a product, and where
    products of other sizes meet); the sum of the parts and its addition to the running sum round by 2^-24 each."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(12)
    x = wide(g, -3, 3, 1, 64, 64, 32)
    w = torch.zeros(32, 32, 9, device="cuda")
    for o in range(32):
        at = torch.randperm(288, device="cuda", generator=g)[:terms]
        w[o].view(-1)[at] = wide(g, -1, 1, terms)
    w = w.view(32, 32, 3, 3)
    got = vd.op_conv2d(x, w, impl=vd.VD_IMPL_TC_F32).double()
    err, size = (got - exact_conv(x, w, 3, 0)).abs(), exact_conv(x.abs(), w.abs(), 3, 0)
    bound = 2.0 ** -24 * (1 + 2 + (2 * terms if terms > 1 else 6 * 2.0 ** -7))
    assert float((err / size.clamp(min=1e-30)).max()) <= bound


@pytest.mark.parametrize("up", [0, 2])
@pytest.mark.parametrize("where", ["activations", "weights"])
def test_infinities_and_the_largest_numbers(vd, where, up):           # noqa: F811
    """Infinities, NaN and numbers that round to infinity in bf16 go through a layer as they do in 64 bits: with weights (or
    activations) of one, two and three parts, and with zero."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(13)
    rnd = lambda *s: torch.randn(*s, device="cuda", generator=g)
    x, w = rnd(1, 21, 20, 64), rnd(64, 64, 3, 3) / 40
    inf = float("inf")
    large = [inf, -inf, float("nan"), 3.4028234e38, -3.4028234e38, 3.3962e38, 3.3961e38, -3.39e38, 2.0 ** 127]
    if where == "activations":
        w[:, 5] = torch.tensor([0.5, -0.25, 1 / 3, -0.0078, 0.75390625, 0.0, 2.0 ** -20, 0.1], device="cuda")[torch.arange(64) % 8][:, None, None]
        if up:
            w *= 0.25                                                 # (sums of four weights stay below one)
        for i, v in enumerate(large):
            x[0, 2 + 7 * (i // 3), 2 + 7 * (i % 3), 5] = v
    else:
        x /= 8 * x.abs().max()
        x[0, ::3, ::2, 7], x[0, 1::3, ::2, 7], x[0, 2::3, 1::2, 7] = 0.5, 1 / 3, 0.0
        for i, v in enumerate(large):
            w[3 * i, 7, 1, 1] = v
    got, want = vd.op_conv2d(x, w, upsample=up, impl=vd.VD_IMPL_TC_F32), exact_conv(x, w, 3, up).float()
    assert int(torch.isinf(want).sum()) >= 9 and int(torch.isnan(want).sum()) >= 1 and float(want[torch.isfinite(want)].abs().max()) > 1e37
    assert torch.equal(torch.isnan(got), torch.isnan(want)) and torch.equal(torch.isinf(got), torch.isinf(want))
    fin = torch.isfinite(want)
    assert torch.equal(got[~fin].nan_to_num(nan=0.0), want[~fin].nan_to_num(nan=0.0))
    assert torch.allclose(got[fin], want[fin], rtol=1e-6, atol=2e-6)  # 4 * 2^-24 of a sum's largest term; of the others, sums of 576 of size 0.025


@pytest.mark.parametrize("B,H,W,Cin,Cout,cpg", [(2, 17, 9, 64, 128, 4), (1, 16, 16, 512, 512, 16), (1, 33, 50, 32, 64, 8)])
def test_records_of_the_output_and_of_the_input(vd, B, H, W, Cin, Cout, cpg):      # noqa: F811
    import torch
    g = torch.Generator(device="cuda").manual_seed(9)
    rnd = lambda *s: torch.randn(*s, device="cuda", generator=g)
    x, w, gamma, beta = rnd(B, H, W, Cin), rnd(Cout, Cin, 3, 3) / (9 * Cin) ** 0.5, 1 + 0.1 * rnd(Cout), 0.1 * rnd(Cout)
    y, rec = vd.op_conv2d(x, w, impl=vd.VD_IMPL_TC_F32, groups=Cout // cpg)
    want = vd.op_gn_stats(y, gamma, beta, Cout // cpg, 1e-6)
    got = vd.op_merge_records(rec, H * W, gamma, beta, 1e-6)
    for a, b in zip(got, want):
        assert torch.allclose(a, b, rtol=2e-5, atol=2e-5)             # fp32 sums of some 1e3 to 1e5 values, in two orders
    if rec.shape[2] <= 128:                                           # and merged by the next layer
        w2 = rnd(32, Cout, 3, 3) / (9 * Cout) ** 0.5
        a = vd.op_conv2d(y, w2, scale=want[0], shift=want[1], silu=True, impl=vd.VD_IMPL_TC_F32)
        b = vd.op_conv2d(y, w2, silu=True, impl=vd.VD_IMPL_TC_F32, in_records=(rec, gamma, beta, 1e-6))
        assert float((a - b).norm() / a.norm()) <= 1e-5
