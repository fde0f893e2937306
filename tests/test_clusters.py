"""Plans without thread-block clusters (what vd_create falls back to on a device that cannot hold them): the workspace that
vd_query_workspace names, which asks no device, holds either plan, and such a decoder gives the same frames up to rounding."""
import pytest

from tests.util import BF16_MAX_ABS, BF16_REL_L2


@pytest.fixture(scope="module")
def vd():
    from paper_2602_00608_b200 import binding, build
    build.build()
    return binding


@pytest.mark.parametrize("arch,dtype,groups", [("tiny", "f32", 8), ("tiny", "bf16", 8), ("sdvae", "f32", 32), ("sdvae", "bf16", 32), ("sdvae", "bf16", 16)])
@pytest.mark.parametrize("h,w,b", [(1, 1, 1), (8, 8, 1), (32, 32, 4), (37, 53, 1), (60, 90, 8)])
def test_the_workspace_holds_the_plan_without_clusters(vd, arch, dtype, groups, h, w, b):
    size = [vd.query_workspace(vd.make_config(arch, dtype, h, w, b, groups, 1e-6, f)) for f in (0, vd.VD_FLAG_NO_CLUSTERS)]
    assert 0 < size[1] <= size[0] <= 1.1 * size[1]


@pytest.mark.gpu
@pytest.mark.parametrize("index,h,w,b", [(1, 8, 8, 1), (1, 11, 7, 3), (2, 8, 8, 2), (2, 24, 16, 1)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_decodes_without_clusters(vd, index, h, w, b, dtype):
    import torch
    from paper_2602_00608_b200 import synth
    if (index, dtype) == (2, "f32"):
        h, w = 5, 7                                          # (the FFMA kernels take their time)
    wl = synth.WORKLOADS[index]
    wts = synth.workload_weights(wl)
    z = torch.from_numpy(synth.workload_latents(wl, batch=b, h=h, w=w)).to("cuda:0", torch.bfloat16 if dtype == "bf16" else torch.float32)
    frames, clusters = [], []
    for flag in (0, vd.VD_FLAG_NO_CLUSTERS):
        dec = vd.Decoder(wl.arch, dtype, h, w, b, wl.groups, wl.eps, wts, vd.VD_FLAG_CANARY | flag)
        frames.append(dec.decode(z).double())
        torch.cuda.synchronize()
        dec.check_status()
        assert dec.check_canaries() > 0
        clusters.append(max(s["cluster"] for s in dec.steps()))
    assert clusters[0] > 1 and clusters[1] == 1
    d = frames[1] - frames[0]
    # two paths that each meet the layout's bound against the exact result differ by at most twice the bound
    if dtype == "bf16":
        assert float(d.norm() / frames[0].norm()) <= 2 * BF16_REL_L2 and float(d.abs().max()) <= 2 * BF16_MAX_ABS
    else:
        assert float(d.norm() / frames[0].norm()) <= 1e-5    # fp32 sums of up to 4608 products in another order, 34 layers deep
