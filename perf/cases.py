"""The work that users of the frame decoder have it do, as a list of sized cases.

A case is one call of `Decoder` on latents of one size: the device entry points (`decode`, `decode_extrapolated`) and
the host transport (`decode_host_stream`), the two layouts, and the two storage types.  Sizes are those of the
workload table (`synth.WORKLOADS`) and of the benchmark, plus ragged ones; `draw` spreads over the same ranges.

A case's fields: arch, dtype; h, w (latent size; frames are 8h x 8w); batch (frames per decode); frames (frames per
call; more than `batch` only for the host transport); api; packed (frames leave as display-packed uint8); latents (the
input distribution).
"""
import math

import torch

from paper_2602_00608_b200 import binding, synth

GROUPS = {"tiny": 8, "sdvae": 32}
EPS = 1e-6
LAMBDA = 0.5          # extrapolation step of the action-hit branch


def _case(name, arch, dtype, h, w, batch, frames, api, packed, latents):
    c = {"arch": arch, "dtype": dtype, "h": h, "w": w, "batch": batch, "frames": frames, "api": api, "packed": packed,
         "latents": latents}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call there is: one 64x64 frame of the small layout; latency of a chain of small kernels
        _case("tiny-f32-64x64", "tiny", "f32", 8, 8, 1, 1, "decode", False, "normal"),
        # sixteen 256x256 frames of the small layout streamed through pinned host memory, packed for display
        _case("tiny-f32-256x256-host16", "tiny", "f32", 32, 32, 4, 16, "host_stream", True, "ar1"),
        # the full-width layout in single precision, as it is run to check the bf16 decoder
        _case("sdvae-f32-64x64", "sdvae", "f32", 8, 8, 1, 1, "decode", False, "normal"),
        # the full-width layout on the smallest frame: every layer is a fraction of the GPU
        _case("sdvae-bf16-64x64", "sdvae", "bf16", 8, 8, 1, 1, "decode", False, "normal"),
        # one 256x256 frame of a platformer whose latent is extrapolated from the last two (player input as predicted)
        _case("sdvae-bf16-256x256-extrapolated", "sdvae", "bf16", 32, 32, 1, 1, "extrapolated", False, "normal"),
        # four consecutive 256x256 frames in one decode
        _case("sdvae-bf16-256x256-stream4", "sdvae", "bf16", 32, 32, 4, 4, "decode", False, "ar1"),
        # a size that no tile divides: 424x296
        _case("sdvae-bf16-424x296", "sdvae", "bf16", 37, 53, 1, 1, "decode", False, "normal"),
        # the headline: one 720x480 frame
        _case("sdvae-bf16-720x480", "sdvae", "bf16", 60, 90, 1, 1, "decode", False, "normal_scaled"),
        # the same frame by frame through pinned host memory: what a game session's frame queue sees
        _case("sdvae-bf16-720x480-host8", "sdvae", "bf16", 60, 90, 1, 8, "host_stream", False, "ar1"),
        # throughput: eight 720x480 frames per decode
        _case("sdvae-bf16-720x480-stream8", "sdvae", "bf16", 60, 90, 8, 8, "decode", False, "ar1"),
        # two 1280x720 frames: the longest attention (14400 tokens)
        _case("sdvae-bf16-1280x720-b2", "sdvae", "bf16", 90, 160, 2, 2, "decode", False, "normal"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    most = max(work(c)["flops"] for c in listed())
    while True:
        kind = rng.choice(("tiny", "sdvae-f32", "sdvae", "sdvae", "sdvae", "sdvae"))
        if kind == "tiny":
            h, w, batch = _log_int(rng, 8, 48), _log_int(rng, 8, 48), rng.randint(1, 4)
            api = rng.choice(("decode", "host_stream"))
            packed = api == "host_stream" and rng.random() < 0.5
            arch, dtype = "tiny", "f32"
        elif kind == "sdvae-f32":
            h, w, batch, api, packed, arch, dtype = rng.randint(5, 12), rng.randint(5, 12), 1, "decode", False, "sdvae", "f32"
        else:
            h, w, batch = _log_int(rng, 8, 96), _log_int(rng, 8, 160), _log_int(rng, 1, 8)
            api, packed, arch, dtype = rng.choice(("decode", "decode", "extrapolated", "host_stream")), False, "sdvae", "bf16"
        frames = batch * rng.randint(1, 4) if api == "host_stream" else batch
        c = _case("", arch, dtype, h, w, batch, frames, api, packed, "ar1" if frames > 1 else rng.choice(("normal", "normal_scaled")))
        if h * w <= 14400 and work(c)["flops"] <= (0.02 * most if dtype == "f32" else most):
            return c


def _weights(arch, seed):
    """Random-initialised parameters: Kaiming-uniform weights, small biases, normalisation scales around 1."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    out = {}
    for name, shape, kind in synth.manifest(arch):
        u = torch.rand(shape, generator=g, device="cuda") * 2 - 1
        if kind == "weight":
            out[name] = u * math.sqrt(3.0 / math.prod(shape[1:]))
        elif kind == "gn_gamma":
            out[name] = 1 + 0.1 * u
        else:
            out[name] = 0.01 * u
    return out


def _latents(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed + 7919)
    z = torch.randn((case["frames"], 4, case["h"], case["w"]), generator=g, device="cuda")
    if case["latents"] == "normal_scaled":
        z = z / 0.18215
    elif case["latents"] == "ar1":                       # consecutive frames resemble one another
        for t in range(1, case["frames"]):
            z[t] = 0.95 * z[t - 1] + math.sqrt(1 - 0.95 * 0.95) * z[t]
    return z


def prepare(case, seed):
    flags = binding.VD_FLAG_OUT_U8 if case["packed"] else 0
    dec = binding.Decoder(case["arch"], case["dtype"], case["h"], case["w"], case["batch"], GROUPS[case["arch"]], EPS,
                          _weights(case["arch"], seed), flags)
    z = _latents(case, seed).to(dec.dtype)
    s = {"case": case, "decoder": dec, "latents": z}
    frames = (case["frames"],) + dec.out_shape
    if case["api"] == "host_stream":
        s["latents"] = z.cpu().pin_memory()
        s["frames"] = torch.empty(frames, dtype=dec.out_dtype).pin_memory()
    else:
        s["frames"] = torch.empty(frames, dtype=dec.out_dtype, device="cuda")
    if case["api"] == "extrapolated":
        g = torch.Generator(device="cuda").manual_seed(seed + 104729)
        s["motion"] = (0.3 * torch.randn(z.shape, generator=g, device="cuda")).to(dec.dtype)
    return s


def run(state):
    dec = state["decoder"]
    api = state["case"]["api"]
    if api == "host_stream":
        return dec.decode_host_stream(state["latents"], state["frames"], state["case"]["batch"])
    if api == "extrapolated":
        return dec.decode_extrapolated(state["latents"], state["motion"], LAMBDA, state["frames"])
    return dec.decode(state["latents"], state["frames"])


def work(case):
    """Parameters, latents and frames once each; multiply-adds of every convolution (the ones on a nearest-2x upsampled
    tensor as the four 2x2 convolutions of its source that they are) and of the attention."""
    p0 = case["h"] * case["w"]
    flops, params = 0.0, 0
    level = 1                                            # pixels per latent pixel
    for name, shape, kind in synth.manifest(case["arch"]):
        params += math.prod(shape)
        if kind != "weight":
            continue
        if name.endswith("upconv.weight"):
            flops += 2.0 * shape[0] * shape[1] * 16 * p0 * level
            level *= 4
        else:
            flops += 2.0 * math.prod(shape) * p0 * level
    if case["arch"] == "sdvae":
        flops += 4.0 * p0 * p0 * 512
    size = 4 if case["dtype"] == "f32" else 2
    latent, frame = 4 * p0 * size, 3 * 64 * p0 * (1 if case["packed"] else size)
    moved = latent * (4 if case["api"] == "extrapolated" else 1) + frame
    return {"bytes": params * size + case["frames"] * moved, "flops": case["frames"] * flops}


def tolerance(case):
    """Measured.  fp32: this path against the same decoder in 64 bits is off by up to 3.0e-6 (2-norm) and 1.5e-5
    (largest).  bf16: two paths of the library that sum in other orders (tensor-core and FFMA kernels, 9-tap and
    phase-collapsed upsampling, statistics by pass and by epilogue) are 7.3e-3 and 4.1e-2 apart, each 4.5e-3 to 5.8e-3
    from 64 bits; the layout's own parity bar is 1e-2.  Packed frames in fp32: an error of 6e-7 crosses a rounding
    boundary of the 1/127.5 steps for about one value in ten thousand."""
    if case["packed"]:
        return {"differ": 5e-4}
    return {"rel": 1.2e-5, "max": 6e-5} if case["dtype"] == "f32" else {"rel": 1e-2, "max": 0.12}
