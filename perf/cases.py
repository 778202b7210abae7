"""What the performance of this library is measured on: its own configurations, through the entry points
that a program calls, from one image to bulk batches, in both directions.

A case is one call (or a few calls in flight) on one flow:

  config   key of iodf_synth.CONFIGS: "0" the tiny flow, "1" the ImageNet32-shaped and "2" the
           ImageNet64-shaped pruned flow, "4s" its unpruned width-512 variant, "R32" / "R64" the paper's
           residual coupling network on the two geometries
  call     encode      uint8 images on the device -> latents and prior parameters
           decode      latents on the device -> uint8 images
           compress    host images -> host byte stream (flow, entropy coder, copies)
           decompress  host byte stream -> host images
           patches     one large image on the device, encoded as rows x cols patches
  batch    images per call
  lanes    calls in flight, each on a stream and a handle of its own (handles made with the throughput
           plan); 1: one call on the current stream, default plan

Every path is integer arithmetic, so two correct implementations give the same values.
"""
import functools
import math

import numpy as np
import torch

import iodf_synth as S
import paper_2206_08869_b200 as G

# int8 operations of the largest listed case: no drawn case costs more
MOST_OPS = 1023 * 2 * 456.6e6
MAX_BATCH = 2048


def _case(name, config, call, batch, lanes=1, rows=0, cols=0):
    return {"name": name, "config": config, "call": call, "batch": batch, "lanes": lanes, "rows": rows, "cols": cols}


def listed():
    return [
        # a small flow on a small batch: one launch, nothing but latency
        _case("tiny encode b16", "0", "encode", 16),
        # a single picture, as an interactive user has it
        _case("im64 encode b1", "2", "encode", 1),
        # the default batch of the benchmark, one call at a time
        _case("im64 encode b128", "2", "encode", 128),
        # the same with four batches in flight, as a service with a queue runs it
        _case("im64 encode b128 x4", "2", "encode", 128, lanes=4),
        # the decoder of the ImageNet32-shaped flow at its configuration's batch
        _case("im32 decode b256", "1", "decode", 256),
        # bulk decoding of an archive; the batch does not divide into whole waves of CTAs
        _case("im64 decode b1023", "2", "decode", 1023),
        # a picture of 704 x 1216 pixels as 209 patches
        _case("im64 patches 11x19", "2", "patches", 209, rows=11, cols=19),
        # the unpruned width-512 network: hidden layers too wide to keep the weights on chip
        _case("wide512 encode b64", "4s", "encode", 64),
        # the paper's own network, encoder and decoder
        _case("res32 encode b64", "R32", "encode", 64),
        _case("res64 decode b32", "R64", "decode", 32),
        # whole compressor and decompressor between host buffers
        _case("im64 compress b128", "2", "compress", 128),
        _case("im64 decompress b128", "2", "decompress", 128),
    ]


def draw(rng):
    config = rng.choice(["0", "1", "1", "2", "2", "2", "2", "4s", "4s", "R32", "R32", "R64"])
    call = rng.choice(["encode", "encode", "encode", "decode", "decode", "compress", "decompress", "patches"])
    if config == "0" and call not in ("encode", "decode"):
        call = rng.choice(["encode", "decode"])        # the tiny flow has no prior head: nothing to code with
    lanes = rng.choice([1, 1, 2, 3, 4]) if call in ("encode", "decode") else 1
    most = max(1, min(MAX_BATCH, int(MOST_OPS / (2.0 * _numbers(config)["macs"]))) // lanes)
    batch = max(1, min(most, int(round(math.exp(rng.uniform(0.0, math.log(most)))))))
    rows = cols = 0
    if call == "patches":
        rows = max(1, min(batch, int(round(math.sqrt(batch) * math.exp(rng.uniform(-0.5, 0.5))))))
        cols = max(1, batch // rows)
        batch = rows * cols
    c = _case("", config, call, batch, lanes, rows, cols)
    del c["name"]
    return c


# ---- flows, handles and images -------------------------------------------------------------------------
def _key(config):
    return int(config) if config.isdigit() else config


@functools.lru_cache(maxsize=None)
def _model(config):
    """The flow's description: weights, requantisation constants, permutations."""
    return S.config_model(_key(config))


@functools.lru_cache(maxsize=None)
def _numbers(config):
    """Sizes of a flow: multiply-accumulates per image, those of the prior heads, bytes of its weights, latents."""
    m = _model(config)
    head = weights = 0
    for lv in m["levels"]:
        for cp in lv["couplings"]:
            weights += sum(ly["w"].size + 12 * ly["c_out"] for ly in cp["layers"])
        if lv["prior"] is not None:
            ly = lv["prior"]["layer"]
            head += lv["h"] * lv["w"] * ly["w"].size
            weights += ly["w"].size + 12 * ly["c_out"]
    d, d_fact, _ = S.latent_sizes(m)
    return {"macs": S.model_macs(m), "head_macs": head, "weight_bytes": weights, "d": d, "d_fact": d_fact}


@functools.lru_cache(maxsize=8)
def _handle(config, max_batch, plan, lane):
    """A program makes a handle once and keeps it; lanes have handles of their own."""
    return G.iodf_create(_model(config), max_batch=max_batch, device=0, plan=plan)


@functools.lru_cache(maxsize=8)
def _codec(config, max_batch):
    return G.iodf_codec_create(_handle(config, max_batch, G.IODF_PLAN_LATENCY, 0), S.logistic_codec())


def _images(config, batch, seed, height=0, width=0):
    """Smooth fields with pixel noise (mean 120, deviation 60, noise 8), uint8 [batch, 3, h, w] on the device."""
    cfg = S.CONFIGS[_key(config)]
    h, w = height or cfg["hw"], width or cfg["hw"]
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    f = torch.randn((batch, 3, h, w), generator=gen, device="cuda")
    r = int(math.ceil(3.0 * cfg["sigma"]))
    taps = np.exp(-0.5 * (np.arange(-r, r + 1) / cfg["sigma"]) ** 2)
    taps /= taps.sum()
    for axis in (-1, -2):
        out = torch.zeros_like(f)
        for k in range(-r, r + 1):
            out.add_(torch.roll(f, k, dims=axis), alpha=float(taps[k + r]))
        f = out
    f -= f.mean(dim=(1, 2, 3), keepdim=True)
    f /= f.square().mean(dim=(1, 2, 3), keepdim=True).sqrt().clamp_min(1e-12)
    f = f * 60.0 + 120.0 + 8.0 * torch.randn(f.shape, generator=gen, device="cuda")
    return torch.floor(f + 0.5).clamp_(0, 255).to(torch.uint8)


def prepare(case, seed):
    config, call, batch, lanes = case["config"], case["call"], case["batch"], case["lanes"]
    if call in ("encode", "decode") and lanes > 1:
        state = {"call": call, "lanes": []}
        for k in range(lanes):
            m = _handle(config, batch, G.IODF_PLAN_THROUGHPUT, k)
            x = _images(config, batch, seed * 64 + k)
            z, prior = G.iodf_forward(m, x)
            lane = {"model": m, "stream": _stream(k), "x": x, "z": z, "prior": prior}
            if call == "encode":
                lane["z"] = torch.zeros_like(z)
                lane["prior"] = torch.zeros_like(prior) if prior is not None else None
            else:
                lane["x"] = torch.zeros_like(x)
            state["lanes"].append(lane)
        return state
    m = _handle(config, batch, G.IODF_PLAN_LATENCY, 0)
    if call == "patches":
        side = S.CONFIGS[_key(config)]["hw"]
        image = _images(config, 1, seed, case["rows"] * side, case["cols"] * side)[0].contiguous()
        return {"call": call, "model": m, "image": image}
    x = _images(config, batch, seed)
    if call == "encode":
        return {"call": call, "model": m, "x": x}
    if call == "decode":
        return {"call": call, "model": m, "z": G.iodf_forward(m, x)[0]}
    codec = _codec(config, batch)
    host = x.cpu().pin_memory()
    packed = torch.zeros(G.iodf_rans_packed_capacity(codec, batch), dtype=torch.uint8).pin_memory()
    if call == "compress":
        return {"call": call, "model": m, "codec": codec, "host": host, "packed": packed}
    _, nbytes = G.iodf_compress_host(m, codec, host, packed)
    return {"call": call, "model": m, "codec": codec, "batch": batch, "host": torch.zeros_like(host).pin_memory(),
            "packed": packed[:nbytes].clone().pin_memory(), "bytes": nbytes}


@functools.lru_cache(maxsize=None)
def _stream(k):
    return torch.cuda.Stream()


def run(state):
    call = state["call"]
    if "lanes" in state:
        here = torch.cuda.current_stream()
        for lane in state["lanes"]:
            lane["stream"].wait_stream(here)
            if call == "encode":
                G.iodf_forward(lane["model"], lane["x"], lane["z"], lane["prior"], stream=lane["stream"])
            else:
                G.iodf_inverse(lane["model"], lane["z"], lane["x"], stream=lane["stream"])
        for lane in state["lanes"]:
            here.wait_stream(lane["stream"])
        return [(lane["z"], lane["prior"]) if call == "encode" else lane["x"] for lane in state["lanes"]]
    if call == "encode":
        return G.iodf_forward(state["model"], state["x"])
    if call == "decode":
        return G.iodf_inverse(state["model"], state["z"])
    if call == "patches":
        return G.iodf_forward_patches(state["model"], state["image"])
    if call == "compress":
        out, nbytes = G.iodf_compress_host(state["model"], state["codec"], state["host"], state["packed"])
        return {"stream": out, "bytes": nbytes}            # the buffer's bytes past the stream stay as they were: zero
    x = G.iodf_decompress_host(state["model"], state["codec"], state["packed"], state["bytes"], state["batch"], state["host"])
    torch.cuda.current_stream().synchronize()          # the host images are valid from here on
    return x


def work(case):
    n = _numbers(case["config"])
    d, prior, coded = n["d"], 8 * n["d_fact"], 15 * n["d"] // 8       # about 15 bits per coded element of these flows
    per_image = {"encode": d + 4 * d + prior, "patches": d + 4 * d + prior, "decode": 4 * d + d,
                 "compress": d + coded, "decompress": coded + d}[case["call"]]
    macs = n["macs"] - (n["head_macs"] if case["call"] == "decode" else 0)
    images = case["batch"] * case["lanes"]
    return {"bytes": images * per_image + case["lanes"] * n["weight_bytes"], "flops": 2.0 * macs * images}


def tolerance(case):
    return "exact"
