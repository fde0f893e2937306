"""Decodes whose layers are divided along K among clusters of CTAs, at the sizes where that can go wrong: a tile filled
exactly and one pixel more, one row of tiles, several frames, an odd number of tiles on pairs of CTAs (40x20: 25 tiles at 80x40),
frame sizes at which some levels are divided and others are not.
Against the FFMA kernels on every pixel, with canaries behind every workspace region, and bitwise the same for a frame decoded
by itself and in a batch."""
import pytest

from tests.util import BF16_MAX_ABS, BF16_REL_L2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h,w,b", [(16, 8, 1), (17, 9, 1), (3, 40, 2), (24, 16, 1), (40, 20, 1)])
def test_small_decodes_match_the_ffma_kernels(h, w, b):
    import torch
    from paper_2602_00608_b200 import binding as vd, synth
    wl = synth.WORKLOADS[2]
    wts = synth.workload_weights(wl)
    z = torch.from_numpy(synth.workload_latents(wl, batch=b, h=h, w=w)).to("cuda:0", torch.bfloat16)
    dec = vd.Decoder(wl.arch, wl.dtype, h, w, b, wl.groups, wl.eps, wts, vd.VD_FLAG_CANARY)
    got = dec.decode(z)
    again = dec.decode(z)
    last = dec.decode(z[b - 1:b].contiguous())
    ffma = vd.Decoder(wl.arch, wl.dtype, h, w, b, wl.groups, wl.eps, wts, vd.VD_FLAG_FORCE_SIMT)
    want = ffma.decode(z)
    torch.cuda.synchronize()
    dec.check_status()
    assert dec.check_canaries() > 0
    assert torch.equal(got, again) and torch.equal(got[b - 1:b], last)
    # two paths that each meet the bound against the exact result differ by at most twice the bound
    d = got.float() - want.float()
    assert float(d.norm() / want.float().norm()) <= 2 * BF16_REL_L2 and float(d.abs().max()) <= 2 * BF16_MAX_ABS


@pytest.mark.parametrize("h,w", [(8, 8), (60, 90)])
def test_statistics_steps_count_what_they_read(h, w):
    """A pass reads the tensor; where the layer before has left records the step reads those, or is no launch and reads nothing."""
    from paper_2602_00608_b200 import binding as vd, synth
    wl = synth.WORKLOADS[2]
    dec = vd.Decoder(wl.arch, wl.dtype, h, w, 1, wl.groups, wl.eps, synth.workload_weights(wl))
    seen = set()
    for s in dec.steps():
        if s["kind"] != vd.VD_STEP_GN_STATS:
            continue
        values = s["out_h"] * s["out_w"] * s["c_in"]
        if s["launches"] == 0:
            assert s["bytes_per_frame"] == 0
            seen.add("merged by the next layer")
        elif s["bytes_per_frame"] in (2 * values, 4 * values):
            seen.add("pass")
        else:
            assert s["bytes_per_frame"] % (16 * wl.groups) == 0 and 0 < s["bytes_per_frame"] < values
            seen.add("merged")
    # 8x8: every layer leaves few records and merges them; 60x90: no level is divided along K, some leave records
    assert seen == ({"merged by the next layer"} if h == 8 else {"merged", "pass"})
