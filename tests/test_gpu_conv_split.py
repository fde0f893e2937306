"""The convolutions that divide K among a cluster, and statistics as records, one operator at a time.

Small whole numbers, whose sums are exact in fp32 whatever their order, give the result of a 64-bit convolution bit for bit: for
every size of a cluster, K that the cluster does not divide evenly, tiles cut by the image edge, odd numbers of tiles on CTA
pairs, the fused shortcut, the four parities of the upsampling form and the frame head.  Records are checked against the
statistics pass over the stored tensor, on the producing and on the consuming side: one record lost of the largest number here
(128) moves a scale by 4e-3."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vd():
    from paper_2602_00608_b200 import binding
    return binding


def ints(g, lo, hi, *shape):
    import torch
    return torch.randint(lo, hi + 1, shape, device="cuda", generator=g).float()


def exact_conv(x, w, k, up):
    """x NHWC, 64 bits."""
    import torch.nn.functional as F
    t = x.double().permute(0, 3, 1, 2)
    if up:
        t = F.interpolate(t, scale_factor=2, mode="nearest")
    return F.conv2d(t, w.double(), padding=k // 2).permute(0, 2, 3, 1)


# B, H, W, Cin, Cout, k, up, CTAs of a cluster (None: CTA pairs)
SHAPES = [
    (2, 20, 20, 64, 128, 3, 0, 1),          # one chunk of 64 channels: nothing to divide
    (1, 16, 8, 128, 128, 3, 0, 2),          # one tile, filled
    (2, 17, 9, 256, 256, 3, 0, 4),          # one pixel more in each direction
    (1, 8, 8, 512, 512, 3, 0, 8),
    (1, 1, 1, 512, 128, 3, 0, 8),
    (1, 30, 21, 192, 128, 3, 0, 2),         # three chunks, two CTAs
    (1, 9, 33, 448, 256, 3, 0, 4),          # seven chunks, four CTAs
    (1, 40, 40, 256, 512, 3, 0, 2),         # limited by the CTAs that fit the chip
    (3, 5, 7, 512, 1536, 1, 0, 4),
    (1, 8, 8, 512, 512, 1, 0, 8),
    (1, 5, 7, 512, 512, 3, 2, 8),           # upsampling: eight blocks x four parities
    (2, 17, 9, 128, 128, 3, 2, 2),
    (1, 3, 2, 64, 256, 3, 2, 1),
    (1, 33, 19, 128, 3, 3, 0, 2),           # frame head
    (2, 8, 8, 512, 16, 3, 0, 8),
    (1, 37, 53, 512, 512, 3, 0, None),      # 21 tiles
    (2, 40, 24, 448, 512, 3, 0, None),      # 9 tiles a frame, seven chunks in two parts
    (1, 32, 40, 512, 512, 3, 0, None),      # ten pairs of tiles and blocks, the fewest
    (1, 64, 64, 512, 256, 3, 0, None),
]


def route_of(vd, B, H, W, Cin, Cout, k, up, in_bf16, out_bf16, nchw):
    d = vd.conv_desc(B, H, W, Cin, Cout, k, up, False, int(in_bf16), int(out_bf16), nchw, True, vd.VD_IMPL_TC_SPLIT)
    return vd.conv_route(d)


@pytest.mark.parametrize("in_bf16", [False, True])
@pytest.mark.parametrize("shape", SHAPES)
def test_divided_layers_are_exact(vd, shape, in_bf16):
    import torch
    B, H, W, Cin, Cout, k, up, _ = shape
    head = Cout % 128 != 0
    in_bf16 = in_bf16 and not head and not up                # (those read the fp32 residual stream)
    g = torch.Generator(device="cuda").manual_seed(H * 1000 + W * 10 + Cin)
    x = ints(g, -4, 4, B, H, W, Cin).to(torch.bfloat16 if in_bf16 else torch.float32)
    w = ints(g, -2, 2, Cout, Cin, k, k).to(torch.bfloat16)
    bias = ints(g, -8, 8, Cout)
    scale, shift = 2.0 ** ints(g, -1, 1, B, Cin), ints(g, -1, 1, B, Cin)
    want = exact_conv(x.double() * scale[:, None, None, :].double() + shift[:, None, None, :].double(), w, k, up) + bias.double()
    for out_bf16 in (False, True):
        res = None if out_bf16 or head or up else ints(g, -64, 64, *want.shape)
        route = route_of(vd, B, H, W, Cin, Cout, k, up, in_bf16, out_bf16, head)
        assert route == (vd.VD_ROUTE_SPLIT_PAIRS if shape[-1] is None else vd.VD_ROUTE_SPLIT)
        got = vd.op_conv2d(x, w, bias, scale, shift, res, upsample=up, out_nchw=head, out_dtype=int(out_bf16), bf16_operands=True,
                           impl=vd.VD_IMPL_TC_SPLIT)
        ref = want if res is None else want + res.double()
        ref = (ref.permute(0, 3, 1, 2) if head else ref).float()
        assert torch.equal(got, ref.to(torch.bfloat16) if out_bf16 else ref)


@pytest.mark.parametrize("impl", ["VD_IMPL_TC_SPLIT", "VD_IMPL_TC"])
@pytest.mark.parametrize("B,H,W,Cin,Cin2,Cout", [(1, 9, 13, 256, 512, 256), (2, 16, 8, 128, 96, 128), (1, 21, 30, 128, 32, 128), (1, 8, 8, 512, 256, 512)])
def test_fused_shortcut_is_exact(vd, impl, B, H, W, Cin, Cin2, Cout):
    import torch
    g = torch.Generator(device="cuda").manual_seed(Cin + Cin2 + H)
    x, w = ints(g, -4, 4, B, H, W, Cin).to(torch.bfloat16), ints(g, -2, 2, Cout, Cin, 3, 3).to(torch.bfloat16)
    x2, w2 = ints(g, -16, 16, B, H, W, Cin2), ints(g, -16, 16, Cout, Cin2)
    bias, bias2 = ints(g, -8, 8, Cout), ints(g, -8, 8, Cout)
    got = vd.op_conv2d(x, w, bias, out_dtype=vd.VD_F32, bf16_operands=True, impl=getattr(vd, impl), shortcut=(x2, w2, bias2))
    want = exact_conv(x, w, 3, 0) + exact_conv(x2, w2[:, :, None, None], 1, 0) + (bias + bias2).double()
    assert torch.equal(got, want.float())


@pytest.mark.parametrize("in_bf16", [False, True])
@pytest.mark.parametrize("B,H,W,Cin,Cout,k", [(2, 17, 9, 256, 256, 3), (1, 37, 53, 512, 512, 3), (1, 12, 20, 512, 512, 1)])
def test_silu_prologue_is_that_of_the_undivided_kernel(vd, B, H, W, Cin, Cout, k, in_bf16):
    import torch
    g = torch.Generator(device="cuda").manual_seed(5)
    rnd = lambda *s: torch.randn(*s, device="cuda", generator=g)
    x, w = rnd(B, H, W, Cin).to(torch.bfloat16 if in_bf16 else torch.float32), (rnd(Cout, Cin, k, k) / Cin ** 0.5).to(torch.bfloat16)
    kw = dict(scale=rnd(B, Cin), shift=rnd(B, Cin), silu=True, out_dtype=vd.VD_F32, bf16_operands=True)
    got, want = (vd.op_conv2d(x, w, impl=i, **kw).double() for i in (vd.VD_IMPL_TC_SPLIT, vd.VD_IMPL_TC))
    # The same operands; the sums differ in order.  The tensor core adds 16 products at a time to an fp32 accumulator and drops
    # what does not fit, up to 2^-23 of it: 288 times for K = 4608, on sums that grow to their size (half of it on average).
    assert float((got - want).norm() / want.norm()) <= 288 * 2.0 ** -23 / 2


def layer(vd, g, impl, B, H, W, Cin, Cout, k, up, in_bf16, out_bf16, x2=False):
    import torch
    rnd = lambda *s: torch.randn(*s, device="cuda", generator=g)
    bf = impl != vd.VD_IMPL_SIMT
    ramp = torch.linspace(-1, 2, H * W, device="cuda").view(1, H, W, 1)            # records differ from one another
    x = (rnd(B, H, W, Cin) + ramp).to(torch.bfloat16 if in_bf16 else torch.float32)
    w = (rnd(Cout, Cin, k, k) / (Cin * k * k) ** 0.5 + 0.5 / (Cin * k * k)).to(torch.bfloat16 if bf else torch.float32)
    kw = dict(upsample=up, out_dtype=int(out_bf16), bf16_operands=bf, impl=impl)
    if x2:
        kw["shortcut"] = (rnd(B, H, W, 64), rnd(Cout, 64) / 8, None)
    if impl != vd.VD_IMPL_TC:                                # (records of conv_tc.cu are those of layers without a bias)
        kw["bias"] = 3 * rnd(Cout)
    return x, w, kw


# impl, B, H, W, Cin, Cout, k, up, in_bf16, out_bf16, fused shortcut
PRODUCERS = [
    ("SIMT", 2, 19, 23, 4, 128, 3, 0, False, False, False),          # first convolution: 64, 32 and 16 pixels per block
    ("SIMT", 1, 19, 23, 8, 256, 3, 0, False, False, False),
    ("SIMT", 2, 5, 13, 4, 512, 3, 0, False, False, False),
    ("SIMT", 2, 17, 9, 36, 128, 3, 0, False, False, False),          # fp32: cluster, and none
    ("SIMT", 1, 8, 8, 512, 64, 3, 0, False, False, False),
    ("SIMT", 1, 40, 50, 32, 32, 3, 0, False, False, False),
    ("SIMT", 1, 12, 10, 64, 64, 1, 0, False, False, False),
    ("SIMT", 2, 9, 21, 64, 32, 3, 2, False, False, False),
    ("TC_SPLIT", 2, 17, 9, 256, 256, 3, 0, False, True, False),
    ("TC_SPLIT", 1, 8, 8, 512, 512, 3, 0, True, False, False),
    ("TC_SPLIT", 1, 20, 20, 64, 128, 3, 0, True, False, False),
    ("TC_SPLIT", 1, 5, 7, 512, 512, 3, 2, False, False, False),
    ("TC_SPLIT", 2, 21, 30, 128, 128, 3, 0, True, False, True),
    ("TC_SPLIT", 1, 12, 20, 512, 512, 1, 0, True, False, False),
    ("TC_SPLIT", 1, 37, 53, 512, 512, 3, 0, False, True, False),     # CTA pairs
    ("TC_SPLIT", 2, 40, 24, 448, 512, 3, 0, True, False, False),
    ("TC", 1, 33, 50, 64, 256, 3, 0, False, True, False),            # the record builds of conv_tc.cu
    ("TC", 2, 70, 61, 128, 512, 3, 0, False, True, False),
    ("TC", 1, 33, 50, 128, 128, 3, 0, True, False, True),
    ("TC", 2, 49, 40, 128, 256, 3, 0, True, False, True),
]


@pytest.mark.parametrize("cpg", [4, 8, 16])
@pytest.mark.parametrize("case", PRODUCERS)
def test_records_hold_the_statistics_of_the_output(vd, case, cpg):
    import torch
    impl, B, H, W, Cin, Cout, k, up, in_bf16, out_bf16, x2 = case
    g = torch.Generator(device="cuda").manual_seed(H + W + Cin)
    impl = getattr(vd, "VD_IMPL_" + impl)
    x, w, kw = layer(vd, g, impl, B, H, W, Cin, Cout, k, up, in_bf16, out_bf16, x2)
    pending = torch.randn(Cout, device="cuda", generator=g) if impl == vd.VD_IMPL_TC else None
    y, records = vd.op_conv2d(x, w, groups=Cout // cpg, pending=pending, **kw)
    assert torch.equal(y, vd.op_conv2d(x, w, **kw))          # leaving records changes nothing
    gamma, beta = (torch.rand(Cout, device="cuda", generator=g) + a for a in (0.5, -0.5))
    got = vd.op_merge_records(records, y.shape[1] * y.shape[2], gamma, beta, 1e-6, offset=pending)
    want = vd.op_gn_stats(y, gamma, beta, Cout // cpg, 1e-6, offset=pending)
    assert float(records[..., 0].sum(2).sub(y.shape[1] * y.shape[2] * cpg).abs().max()) == 0
    # two orders of fp32 sums about different reference values, as between the statistics kernels and the oracle
    torch.testing.assert_close(got[0], want[0], rtol=2e-5, atol=0)
    torch.testing.assert_close(got[1], want[1], rtol=2e-5, atol=2e-5 * float(want[1].abs().max()))


@pytest.mark.parametrize("slots", [1, 9, 16, 17, 40, 65, 128])
@pytest.mark.parametrize("route,shape", [
    ("F32", (2, 12, 10, 64, 32, 3)), ("F32", (8, 40, 50, 512, 32, 1)), ("SPLIT", (2, 17, 9, 256, 256, 3)),
    ("SPLIT", (1, 20, 20, 64, 128, 3)), ("SPLIT", (1, 12, 20, 512, 512, 1)), ("SPLIT_PAIRS", (1, 37, 53, 512, 512, 3)),
])
@pytest.mark.parametrize("cpg", [4, 16])
def test_layers_merge_the_records_of_their_input(vd, route, shape, slots, cpg):
    """Records of `slots` shares of the pixels, some of them empty, against scale and shift from the statistics pass."""
    import torch
    B, H, W, Cin, Cout, k = shape
    g = torch.Generator(device="cuda").manual_seed(slots)
    f32 = route == "F32"
    impl = vd.VD_IMPL_SIMT if f32 else vd.VD_IMPL_TC_SPLIT
    x, w, kw = layer(vd, g, impl, B, H, W, Cin, Cout, k, 0, False, False)
    d = vd.conv_desc(B, H, W, Cin, Cout, k, 0, True, vd.VD_F32, vd.VD_F32, False, not f32, impl)
    assert vd.conv_route(d) == getattr(vd, "VD_ROUTE_" + route)
    G = Cin // cpg
    t = x.double().view(B, H * W, G, cpg)
    records = torch.zeros(B, G, slots, 4, device="cuda")
    bounds = [H * W * i // slots for i in range(slots + 1)] if slots % 2 else [H * W * (i // 2) // (slots // 2) for i in range(slots + 1)]
    for i in range(slots):
        part = t[:, bounds[i]:bounds[i + 1]].transpose(1, 2).reshape(B, G, -1)
        if part.shape[2]:
            mean = part.mean(2)
            records[:, :, i, 0] = part.shape[2]
            records[:, :, i, 1] = mean
            records[:, :, i, 2] = (part - mean[:, :, None]).square().sum(2)
    if slots > 1 and slots % 2 == 0:                         # the first record of a layer is never empty
        records = records.flip(2)
    gamma, beta = (torch.rand(Cin, device="cuda", generator=g) + a for a in (0.5, -0.5))
    scale, shift = vd.op_gn_stats(x, gamma, beta, G, 1e-6)
    got = vd.op_conv2d(x, w, silu=True, in_records=(records, gamma, beta, 1e-6), **kw).double()
    want = vd.op_conv2d(x, w, scale=scale, shift=shift, silu=True, **kw).double()
    # scale and shift agree to about 1e-6: fp32 operands follow, bf16 ones change their rounding once in 4000 values
    # (2^-8 * sqrt(1 / 4000) = 6e-5 of the operand)
    assert float((got - want).norm() / want.norm()) <= (1e-5 if f32 else 2e-4)
