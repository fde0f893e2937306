"""VD_FLAG_FORCE_SIMT plans every layer on the FFMA kernels, in either storage type: the cross-check path of the tensor-core ones."""
import pytest

from tests.util import F32_REL_L2, rel_l2


@pytest.fixture(scope="module")
def vd():
    from paper_2602_00608_b200 import binding, build
    build.build()
    return binding


def test_the_fp32_plan_packs_plain_weights(vd):
    """Weights of the tensor-core layers take 6 bytes instead of 4, which the workspace shows (52 million of them, sixteen taps
    counted in the upsampling layers)."""
    size = [vd.query_workspace(vd.make_config("sdvae", "f32", 8, 8, 1, 32, 1e-6, f)) for f in (0, vd.VD_FLAG_FORCE_SIMT)]
    assert size[0] - size[1] > 2 * 40e6


@pytest.mark.gpu
def test_fp32_decodes_with_and_without_the_tensor_cores(vd):
    import torch
    from oracle import ref
    from paper_2602_00608_b200 import synth
    wl = synth.WORKLOADS[2]
    wts = synth.workload_weights(wl)
    z = synth.workload_latents(wl, batch=1, h=8, w=7)
    want = ref.decode(wl.arch, wts, z, wl.groups, wl.eps)
    frames, impl = [], []
    for flags in (0, vd.VD_FLAG_FORCE_SIMT):
        dec = vd.Decoder(wl.arch, "f32", 8, 7, 1, wl.groups, wl.eps, wts, flags)
        frames.append(dec.decode(torch.from_numpy(z).cuda()).double().cpu().numpy())
        torch.cuda.synchronize()
        dec.check_status()
        impl.append({s["name"] for s in dec.steps() if s["impl"]})
        assert rel_l2(frames[-1], want) <= F32_REL_L2
    assert not impl[1] and {"mid.res0.conv1", "up0.upconv", "up3.res2.conv2"} <= impl[0] and not {"conv_in", "mid.attn.o", "conv_out"} & impl[0]
    assert 0 < rel_l2(frames[0], frames[1]) <= 1e-5      # fp32 sums of up to 4608 products in another order, 34 layers deep
