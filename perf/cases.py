"""The work that a user has this library do, as cases that can be timed: whole UNet steps and VAE decoders, single
layers through each entry point, and the filter transform of a model load.

A case is one of three kinds:
  net     the 3x3 convolutions of one UNet step or one VAE decoder, in order, in one call of the multi-layer entry
  layer   one convolution through the entry that `entry` names (conv: fp16; ex: fp16 with residual and SiLU; f32: fp32
          tensors; f32_scaled: fp32 of any magnitude; q8: 8-bit filters; stride2: the downsampling convolution)
  filter  the transform of one weight tensor, as a model load does it for every layer
Sizes are those of `paper_2412_05781_b200.workloads` (SD v1.5, v2.1 and SDXL UNets, their VAE decoders), and of the same
networks on other image sizes.  The algorithm of a layer is the one sdwino_choose_algorithm names, as in the README.
"""
import math

import torch

from paper_2412_05781_b200 import binding as sd
from paper_2412_05781_b200 import workloads


def listed():
    return [
        # one small layer, the single-layer workload: the latency of a call
        {"name": "layer_320_at32", "kind": "layer", "entry": "conv", "N": 1, "C": 320, "K": 320, "H": 32, "W": 32},
        # one denoising step at 512x512 with classifier-free guidance (batch 2)
        {"name": "sd15_unet_step", "kind": "net", "net": "unet", "N": 2, "H": 64, "W": 64},
        # one denoising step at 768x768 for a batch of two images with guidance
        {"name": "sd21_unet_step_n4", "kind": "net", "net": "unet", "N": 4, "H": 96, "W": 96},
        # the image decoder after the last step, 512x512
        {"name": "vae_decoder_512", "kind": "net", "net": "vae", "N": 1, "H": 64, "W": 64},
        # the largest configuration: UNet step and VAE decoder at 1024x1024
        {"name": "sdxl_1024", "kind": "net", "net": "sdxl", "N": 2, "H": 128, "W": 128},
        # a UNet layer of an image whose latent is 100x74 (800x592): widths that no vector divides
        {"name": "ragged_640_at50x37", "kind": "layer", "entry": "conv", "N": 2, "C": 640, "K": 640, "H": 50, "W": 37},
        # the deepest level of the UNet, where a layer is its weights: latency of the weight stream
        {"name": "weights_1280_at16", "kind": "layer", "entry": "conv", "N": 2, "C": 1280, "K": 1280, "H": 16, "W": 16},
        # the second convolution of a decoder ResNet block with what follows it
        {"name": "residual_silu_512_at128", "kind": "layer", "entry": "ex", "N": 1, "C": 512, "K": 512, "H": 128, "W": 128},
        # a model kept in fp32
        {"name": "f32_640to320_at64", "kind": "layer", "entry": "f32", "N": 2, "C": 640, "K": 320, "H": 64, "W": 64},
        # a model kept with quantised weights
        {"name": "q8_1280_at32", "kind": "layer", "entry": "q8", "N": 2, "C": 1280, "K": 1280, "H": 32, "W": 32},
        # the downsampling convolution between two UNet levels
        {"name": "stride2_320_at64", "kind": "layer", "entry": "stride2", "N": 2, "C": 320, "K": 320, "H": 64, "W": 64},
        # model load: one of the UNet's larger weight tensors
        {"name": "filters_1280x1280", "kind": "filter", "C": 1280, "K": 1280, "tile": 2},
    ]


# channel pairs of the UNet by level (full latent, 1/2, 1/4, 1/8) and of the VAE decoder by scale over the latent
_UNET = [[(4, 320), (320, 320), (640, 320), (960, 320), (320, 4)],
         [(320, 640), (640, 640), (960, 640), (1280, 640), (1920, 640)],
         [(640, 1280), (1280, 1280), (1920, 1280), (2560, 1280)],
         [(1280, 1280), (2560, 1280)]]
_VAE = [(1, [(4, 512), (512, 512)]), (2, [(512, 512)]), (4, [(512, 512), (512, 256), (256, 256)]),
        (8, [(256, 256), (256, 128), (128, 128), (128, 3)])]
_MOST_FLOPS = 1.0e12      # direct-convolution flops of a drawn layer: below the largest layer of the listed cases


def _latent(rng, lo, hi):
    """A latent of an image between about 8 lo and 8 hi on a side, any aspect ratio from 1:2 to 2:1, any size."""
    side = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    ratio = math.exp(rng.uniform(math.log(0.5), math.log(2.0)) / 2)
    return max(8, round(side * ratio)), max(8, round(side / ratio))


def draw(rng):
    kind = rng.choice(["unet_layer"] * 5 + ["vae_layer"] * 2 + ["net"] * 2 + ["filter"])
    if kind == "net":
        net = rng.choice(["unet", "vae"])
        if net == "unet":
            h, w = _latent(rng, 32, 96)
            return {"kind": "net", "net": "unet", "N": rng.choice([1, 2, 4]), "H": h, "W": w}
        h, w = _latent(rng, 24, 72)
        return {"kind": "net", "net": "vae", "N": 1, "H": h, "W": w}
    if kind == "filter":
        C, K = rng.choice([p for level in _UNET for p in level] + [(512, 512), (256, 256), (128, 128)])
        return {"kind": "filter", "C": C, "K": K, "tile": rng.choice([2, 4])}
    while True:
        if kind == "unet_layer":
            h, w = _latent(rng, 32, 160)
            level = rng.randrange(4)
            C, K = rng.choice(_UNET[level])
            case = {"kind": "layer", "entry": "conv", "N": rng.choice([1, 2, 2, 4, 8]), "C": C, "K": K,
                    "H": -(-h >> level), "W": -(-w >> level)}
        else:
            h, w = _latent(rng, 24, 128)
            scale, pairs = rng.choice(_VAE)
            C, K = rng.choice(pairs)
            case = {"kind": "layer", "entry": "conv", "N": 1, "C": C, "K": K, "H": h * scale, "W": w * scale}
        if min(C, K) > 8:
            case["entry"] = rng.choice(["conv"] * 5 + ["ex", "f32", "f32_scaled", "q8"])
            if C == K and kind == "unet_layer" and rng.random() < 0.15:
                case["entry"] = "stride2"
        if 18.0 * case["N"] * C * K * case["H"] * case["W"] <= _MOST_FLOPS:
            return case


def _layers(case):
    if case["kind"] != "net":
        return [workloads.ConvLayer(C=case["C"], K=case["K"], H=case["H"], W=case["W"], N=case["N"])]
    h, w, n = case["H"], case["W"], case["N"]
    if case["net"] == "sdxl":
        return workloads.sdxl_1024()
    if case["net"] == "unet":      # the layer list of sd15_unet on a latent of h x w
        return [workloads.ConvLayer(C=L.C, K=L.K, H=-(-h * L.H // 64), W=-(-w * L.W // 64), N=n) for L in workloads.sd15_unet(n)]
    return [workloads.ConvLayer(C=L.C, K=L.K, H=h * L.H // 64, W=w * L.W // 64, N=n) for L in workloads.sd_vae_decoder_512()]


def _tile(case, L):
    if case["kind"] == "layer" and case["entry"] == "stride2":
        return 1
    if case["kind"] == "layer" and case["entry"] in ("f32", "f32_scaled", "q8"):    # Winograd only
        return sd.sdwino_choose_tile(L.N, L.C, L.H, L.W, L.K)
    return sd.sdwino_choose_algorithm(L.N, L.C, L.H, L.W, L.K)


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape, std=1.0, dtype=torch.float16):
        return (torch.randn(*shape, generator=g, device="cuda", dtype=torch.float32) * std).to(dtype)

    if case["kind"] == "filter":
        C, K = case["C"], case["K"]
        return {"kind": "filter", "tile": case["tile"], "w": normal(K, C, 3, 3, std=(9 * C) ** -0.5)}
    entry = case.get("entry", "conv")
    dtype = torch.float32 if entry.startswith("f32") else torch.float16
    rows, need = [], 0
    for L in _layers(case):
        tile = _tile(case, L)
        # activations after a normalisation, weights that keep the variance; fp32 activations of any magnitude for the
        # range-safe entry
        x = normal(L.N, L.C, L.H, L.W, std=3.0e4 if entry == "f32_scaled" else 1.0, dtype=dtype)
        w = normal(L.K, L.C, 3, 3, std=(9 * L.C) ** -0.5, dtype=dtype)
        b = normal(L.K, std=0.02, dtype=dtype)
        wT = sd.sdwino_filter_transform_f32(w, tile) if dtype == torch.float32 else sd.sdwino_filter_transform(w, tile)
        if entry == "q8":
            wT = sd.sdwino_filter_quantize(wT, L.K, L.C, tile)
        step = 2 if entry == "stride2" else 1
        y = torch.empty(L.N, L.K, -(-L.H // step), -(-L.W // step), dtype=dtype, device="cuda")
        res = normal(*y.shape) if entry == "ex" else None
        need = max(need, sd.sdwino_workspace_bytes_direct(L.N, L.C, L.H, L.W, L.K, 2) if entry == "stride2"
                   else sd.sdwino_workspace_bytes(L.N, L.C, L.H, L.W, L.K, tile))
        rows.append({"x": x, "wT": wT, "b": b, "y": y, "K": L.K, "tile": tile, "res": res})
    state = {"kind": case["kind"], "entry": entry, "rows": rows, "ws": sd.alloc_workspace(need)}
    if case["kind"] == "net":
        state["seq"] = sd.make_sequence([(r["x"], r["wT"], r["b"], r["y"], r["K"], r["tile"]) for r in rows])
    return state


def run(state):
    if state["kind"] == "filter":
        wT = sd.sdwino_filter_transform(state["w"], state["tile"])
        # what is written of the buffer: the four words of the header (it is 1 KB long) and the filters
        return {"header": wT[:16].view(torch.int32), "filters": wT[1024:].view(torch.float16)}
    ws = state["ws"]
    if state["kind"] == "net":
        sd.sdwino_conv3x3_sequence(state["seq"], ws)
        return [r["y"] for r in state["rows"]]
    r, entry = state["rows"][0], state["entry"]
    if entry == "conv":
        return sd.sdwino_conv3x3(r["x"], r["wT"], r["b"], r["K"], r["tile"], y=r["y"], workspace=ws)
    if entry == "ex":
        return sd.sdwino_conv3x3_ex(r["x"], r["wT"], r["b"], r["res"], r["K"], r["tile"], sd.ACT_SILU, ws, y=r["y"])
    if entry in ("f32", "f32_scaled"):
        return sd.sdwino_conv3x3_f32(r["x"], r["wT"], r["b"], r["K"], r["tile"], ws, y=r["y"], scaled=entry == "f32_scaled")
    if entry == "q8":
        return sd.sdwino_conv3x3_q8(r["x"], r["wT"], r["b"], r["K"], r["tile"], ws, y=r["y"])
    return sd.sdwino_conv3x3_direct(r["x"], r["wT"], r["b"], r["K"], 2, ws, y=r["y"])


def work(case):
    """Each tensor once (weights as nine values each, one byte each where they are 8-bit), and the multiplications that
    the cheapest of the supported algorithms needs: 36 per 16 outputs for stride 1, nine per output for stride 2."""
    if case["kind"] == "filter":
        return {"bytes": 18 * case["C"] * case["K"] + sd.sdwino_filter_bytes(case["K"], case["C"], case["tile"]), "flops": 0}
    entry = case.get("entry", "conv")
    size = 4 if entry.startswith("f32") else 2
    total, flops = 0, 0
    for L in _layers(case):
        pixels = L.N * L.H * L.W
        outs = L.N * -(-L.H // 2) * -(-L.W // 2) if entry == "stride2" else pixels
        total += size * (pixels * L.C + outs * L.K + L.K) + (1 if entry == "q8" else 2) * 9 * L.C * L.K
        total += 2 * outs * L.K if entry == "ex" else 0
        flops += (18.0 if entry == "stride2" else 4.5) * outs * L.C * L.K
    return {"bytes": total, "flops": flops}


def tolerance(case):
    """About four times the distance from the convolution in fp64 (relative 2-norm; largest difference): 1.9e-3 and 2.4e-2
    with F(4x4), whose matrices amplify the fp16 rounding of the transformed tensors, 6.4e-4 and 4.3e-3 with F(2x2), 2.9e-4
    and 1.3e-3 for the direct form.  Quantised filters are part of their operator.  A transformed filter is one rounding of
    an fp32 value: implementations differ where that value lies next to a tie."""
    if case["kind"] == "filter":
        return {"rel": 1e-4, "max": 2e-3}
    if case.get("entry") == "stride2":
        return {"rel": 1.2e-3, "max": 6e-3}
    wide = max(sd.sdwino_choose_tile(L.N, L.C, L.H, L.W, L.K) for L in _layers(case)) == 4
    return {"rel": 8e-3, "max": 0.1} if wide else {"rel": 2.5e-3, "max": 1.7e-2}
