"""Which kernel a single fp32 convolution takes, on the host: the kernels that read and write 16 bytes at a time must not be
given tensors that lie elsewhere (a misaligned access ends the CUDA context); those stay on the direct kernel."""
import ctypes

import pytest

from paper_2602_00608_b200 import binding as vd


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2602_00608_b200 import build
    build.build()


def desc(cin, cout, k=3, upsample=0, nchw=False, impl=vd.VD_IMPL_SIMT, h=12, w=10, b=1):
    return vd.conv_desc(b, h, w, cin, cout, k, upsample, False, vd.VD_F32, vd.VD_F32, nchw, False, impl)


LAYERS = {                     # descriptor, its kernel, the tensors that this kernel takes in 16-byte pieces
    "f32": (desc(64, 32), vd.VD_ROUTE_F32, {"x", "w", "bias", "residual", "y"}),
    "1x1": (desc(36, 96, 1), vd.VD_ROUTE_F32, {"x", "w", "bias", "residual", "y"}),
    "head": (desc(64, 3, nchw=True), vd.VD_ROUTE_F32, {"x"}),
    "thin": (desc(4, 256), vd.VD_ROUTE_THIN, {"x", "w", "bias", "y"}),
    "thin8": (desc(8, 128), vd.VD_ROUTE_THIN, {"x", "w", "bias", "y"}),
}


@pytest.mark.parametrize("impl", [vd.VD_IMPL_SIMT, vd.VD_IMPL_AUTO])
@pytest.mark.parametrize("name", LAYERS)
def test_misaligned_tensors_take_the_direct_kernel(name, impl):
    d, kernel, vector = LAYERS[name]
    d.impl = impl
    aligned = {"x": 1 << 20, "w": 2 << 20, "bias": 3 << 20, "y": 5 << 20}
    if "residual" in vector:
        aligned["residual"] = 4 << 20
    assert vd.conv_route(d, **aligned) == kernel
    for t in aligned:
        for off in (4, 8, 12):
            want = vd.VD_ROUTE_DIRECT if t in vector else kernel
            assert vd.conv_route(d, **{**aligned, t: aligned[t] + off}) == want, (t, off)


def test_phase_collapsed_layers_of_misaligned_tensors_are_refused():
    d = desc(32, 32, upsample=2)
    assert vd.conv_route(d) == vd.VD_ROUTE_F32
    for t in ("x", "w", "y", "bias"):
        with pytest.raises(vd.VdError) as e:
            vd.conv_route(d, **{t: 1028})
        assert e.value.status == vd.VD_ERR_UNSUPPORTED and "aligned" in str(e.value)


def test_phase_collapsed_layers_beyond_the_kernel_are_refused():
    """No other FFMA kernel reads weights packed as sixteen 2x2 taps: what the kernel cannot plan must not be accepted."""
    assert vd.conv_route(desc(4096, 32, upsample=2)) == vd.VD_ROUTE_F32
    for d in (desc(4100, 32, upsample=2), desc(64, 32, upsample=2, h=32768, w=32768), desc(4, 32, upsample=2, h=65536, w=32768)):
        with pytest.raises(vd.VdError) as e:
            vd.conv_route(d)
        assert e.value.status == vd.VD_ERR_UNSUPPORTED
        n = ctypes.c_size_t()
        assert vd.lib().vd_conv_packed_weight_bytes(ctypes.byref(d), ctypes.byref(n)) == vd.VD_ERR_UNSUPPORTED


def test_layers_beyond_the_kernels_indices_take_the_direct_kernel():
    assert vd.conv_route(desc(4096, 64)) == vd.VD_ROUTE_F32 and vd.conv_route(desc(4100, 64)) == vd.VD_ROUTE_DIRECT
    # 2^32 - 1 pieces of four channels and 2^31 - 1 pixels of a frame are the last ones
    assert vd.conv_route(desc(64, 32, h=16384, w=16383)) == vd.VD_ROUTE_F32
    assert vd.conv_route(desc(64, 32, h=16384, w=16384)) == vd.VD_ROUTE_DIRECT
    assert vd.conv_route(desc(4, 32, h=65536, w=32767)) == vd.VD_ROUTE_F32
    assert vd.conv_route(desc(4, 32, h=65536, w=32768)) == vd.VD_ROUTE_DIRECT


@pytest.mark.gpu
@pytest.mark.parametrize("cin,cout,k,nchw,moved", [
    (36, 64, 3, False, "x"), (36, 64, 3, False, "bias"), (36, 64, 3, False, "residual"), (64, 96, 1, False, "x"),
    (64, 96, 1, False, "bias"), (32, 3, 3, True, "x"), (32, 3, 3, True, "bias"), (4, 128, 3, False, "x"), (4, 128, 3, False, "bias")])
def test_views_into_larger_buffers_give_the_same_result(cin, cout, k, nchw, moved):
    import torch
    g = torch.Generator(device="cuda").manual_seed(7)
    B, H, W = 2, 9, 13

    def tensor(name, *shape):
        flat = torch.randn(int(torch.tensor(shape).prod()) + 1, device="cuda", generator=g)
        return flat[1:].view(shape) if name == moved else flat[:-1].view(shape).clone()
    x, bias, w = tensor("x", B, H, W, cin), tensor("bias", cout), torch.randn(cout, cin, k, k, device="cuda", generator=g)
    res = tensor("residual", B, H, W, cout) if moved == "residual" else None
    got = vd.op_conv2d(x, w, bias, residual=res, out_nchw=nchw, impl=vd.VD_IMPL_SIMT)
    want = torch.nn.functional.conv2d(x.permute(0, 3, 1, 2).double(), w.double(), bias.double(), padding=k // 2)
    if not nchw:
        want = want.permute(0, 2, 3, 1)
    if res is not None:
        want = want + res.double()
    # fp32 sums of at most 324 products in sequence: 2^-24 / sqrt(3) * sqrt(324 / 2)
    assert float((got.double() - want).norm() / want.norm()) <= 1e-6


def test_the_single_precision_tensor_core_kernel_is_named():
    for upsample in (0, 2):
        assert vd.conv_route(desc(128, 64, upsample=upsample, impl=vd.VD_IMPL_TC_F32)) == vd.VD_ROUTE_F32_TC
        assert vd.conv_route(desc(128, 64, upsample=upsample, impl=vd.VD_IMPL_AUTO)) == vd.VD_ROUTE_F32
    for d in (desc(128, 64, k=1), desc(20, 64), desc(128, 48), desc(128, 64, upsample=1)):
        d.impl = vd.VD_IMPL_TC_F32
        with pytest.raises(vd.VdError):
            vd.conv_route(d)
    d = desc(128, 64, impl=vd.VD_IMPL_TC_F32)
    with pytest.raises(vd.VdError):
        vd.conv_route(d, w=264)                              # (a bulk copy starts on a 16-byte boundary)
