"""The tensor-core attention at the edges of its tiles: 128 queries per CTA pair, 256 keys per tile in blocks of 64, one to four
pairs that share the keys, the single-tile kernel of up to 128 tokens; and the rescaling of the output where a pair walks
several tiles."""
import math

import numpy as np
import pytest

from tests.test_gpu_ops import _attn_case, _rng, env, rel_l2         # noqa: F401  (env is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T", [(1, 1), (3, 63), (2, 65), (1, 127), (2, 129), (1, 256), (1, 257), (2, 511), (1, 513), (1, 769), (1, 1025), (2, 1961),
                                 (1, 1537), (1, 1600), (1, 1791), (1, 2049), (1, 2112), (1, 2200)])        # four pairs, then three (see below)
def test_attention_at_the_edges_of_tiles(env, B, T):                  # noqa: F811
    _, _, vd, _ = env
    got, want = _attn_case(env, 61, B, T, 512, True, vd.VD_IMPL_TC)
    assert rel_l2(got, want) <= 6e-3              # bf16 probabilities and bf16 output: two roundings of 2^-9 relative


@pytest.mark.parametrize("h,w,pairs", [(24, 24, 1), (32, 32, 2), (29, 53, 4), (40, 40, 4), (9, 199, 4), (44, 48, 3), (40, 55, 3), (50, 60, 2), (60, 90, 1)])
def test_pairs_that_share_the_keys(env, h, w, pairs):                 # noqa: F811
    """The sizes above and below are those at which a 148-SM device takes one to four pairs."""
    torch, _, vd, synth = env
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the choice is that of a 148-SM device")
    wl = synth.WORKLOADS[2]
    dec = vd.Decoder(wl.arch, "bf16", h, w, 1, wl.groups, wl.eps, synth.workload_weights(wl))
    assert [s["cluster"] for s in dec.steps() if s["name"] == "mid.attn.core"] == [2 * pairs if pairs > 1 else 1]


@pytest.mark.parametrize("T", [1791, 2200, 3000])                     # four pairs (1, 2, 2, 2 tiles), three (3 each), two (6 each)
def test_attention_rescales_within_a_share_of_the_keys(env, T):       # noqa: F811
    """Key tiles whose scores keep growing by more than the rescaling threshold, within a pair's share and from one to the next."""
    torch, ref, vd, synth = env
    C = 512
    r = _rng(62)
    q = r.standard_normal((1, T, C)).astype(np.float32)
    k = r.standard_normal((1, T, C)).astype(np.float32) * 0.05
    up = np.sign(q.mean(axis=1, keepdims=True))
    k = k + (np.arange(T) // 256).astype(np.float32)[None, :, None] * 0.6 * up
    q = q + 0.5 * up
    v = r.standard_normal((1, T, C)).astype(np.float32)
    qkv = synth.round_to_bf16(np.concatenate([q, k, v], axis=2))
    scale = 1.0 / math.sqrt(C)
    qq, kk, vv = (qkv[0, :, i * C:(i + 1) * C].astype(np.float64) for i in range(3))
    rows = np.r_[0:64, 1000:1064, T - 64:T]
    s = qq[rows] @ kk.T * scale
    tile_max = np.stack([s[:, i:i + 256].max(axis=1) for i in range(0, T, 256)], axis=1)
    assert np.median(np.diff(tile_max, axis=1)) * 1.4427 > 8.0        # really beyond the threshold
    p = np.exp(s - s.max(axis=1, keepdims=True))
    want = (p / p.sum(axis=1, keepdims=True)) @ vv
    got = vd.op_attention(torch.from_numpy(qkv).cuda().bfloat16(), C, scale, vd.VD_IMPL_TC)
    torch.cuda.synchronize()
    assert rel_l2(got[0].float().cpu().numpy()[rows], want) <= 6e-3
