"""The work whose speed is followed from one version of this framework to the next.

A case is what a program that serves or converts a W4A4 network has the framework do, called through the Python
binding the way such a program calls it:

  layer    one linear layer: quantize the activations, run the layer on the codes (`quantize_act`, then `w4a4_linear`,
           or `w4a4_linear_pow2` for the power-of-two steps)
  encoder  the 32 linear layers of the 4-stage encoder in execution order
  map      a channel-major feature map quantized in place, then a 1x1 convolution (`quantize_act_nchw`, `w4a4_linear`)
  host     a layer on host buffers, copies included (`quant_linear_host`)
  weights  conversion of one weight matrix (`quantize_weight`)

`kept` says whether the program keeps its output buffers and the workspace from call to call (a serving loop) or
leaves them to the binding (the form of the package's docstring).  Activations are the heavy-tailed token mixture of
`synth_inputs.py`, drawn on the GPU; weights are N(0, 0.02) and quantized beforehand, as they are static.
"""
import math

import torch

import synth_inputs
from paper_2604_16855_b200 import tdq

DTYPES = {"fp32": torch.float32, "bf16": torch.bfloat16, "fp16": torch.float16}
MAX_MACS = 16384 * 4096 * 4096     # the largest listed layer
MAX_CELLS = 16384 * 4096           # its activations, and its outputs


def layer(name, rows, cin, cout, x="bf16", y="fp32", g=32, steps="exact", zr=0.2, p=1.0, bias=True, kept=True):
    return {"name": name, "op": "layer", "rows": rows, "cin": cin, "cout": cout, "x": x, "y": y, "g": g, "steps": steps,
            "zr": zr, "p": p, "bias": bias, "kept": kept}


def listed():
    return [
        # the smallest workload of the benchmark (its first configuration), in the form the package's docstring shows:
        # latency, launches and host work
        layer("single_layer_fp32", 256, 64, 64, x="fp32", bias=False, kept=False),
        # stage-1 MLP of the encoder on one 384 x 384 image (second configuration): many tokens, two groups each
        layer("stage1_fc1", 9216, 64, 256, bias=False),
        # stage-3 attention qkv at batch 16 (third configuration) with a 16-bit output, as the attention that follows takes it
        layer("stage3_qkv_bf16", 16 * 576, 320, 960, y="bf16"),
        # ViT-B MLP at batch 32 (fourth configuration, the one the benchmark's headline is quoted on)
        layer("vitb_fc1", 32 * 577, 768, 3072, bias=False),
        # the same layer of a program that trades accuracy for speed with power-of-two steps
        layer("vitb_fc1_pow2", 32 * 577, 768, 3072, y="bf16", steps="pow2"),
        # wider token groups (the group-size ablation), half precision out
        layer("vitb_fc1_g128_fp16", 8 * 577, 768, 3072, y="fp16", g=128),
        # overlapping patch embedding: 7 x 7 x 3 = 147 channels, padded to the group; odd numbers of rows and outputs
        layer("patch_embed_147", 9217, 147, 63, x="fp32", kept=False),
        # one step per token over a long contraction: the compute-bound end, the largest layer
        layer("token_steps_4096", 16384, 4096, 4096, y="bf16", g=4096),
        # every linear layer of the encoder at batch 8 (fifth configuration)
        {"name": "encoder_b8", "op": "encoder", "batch": 8},
        # a convolutional feature map quantized along its channels, then a 1x1 convolution
        {"name": "feature_map_1x1", "op": "map", "batch": 16, "cin": 320, "height": 24, "width": 24, "cout": 320, "x": "bf16",
         "y": "bf16", "zr": 0.2, "bias": True, "kept": True},
        # the third configuration for a caller whose data is on the host
        {"name": "stage3_qkv_host", "op": "host", "rows": 16 * 576, "cin": 320, "cout": 960, "x": "bf16", "y": "fp32"},
        # conversion of a large weight matrix
        {"name": "weights_4096", "op": "weights", "cin": 4096, "cout": 4096, "x": "fp32", "g": 32},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["layer", "encoder", "map", "host", "weights"], [12, 1, 3, 2, 2])[0]
    x = rng.choice(["bf16", "bf16", "fp32"])
    y = rng.choice(["fp32", "bf16", "bf16", "fp16"])
    if kind == "encoder":
        return {"op": "encoder", "batch": rng.randint(1, 8)}
    if kind == "weights":
        return {"op": "weights", "cin": _log(rng, 32, 4096), "cout": _log(rng, 32, 4096), "x": x, "g": rng.choice([32, 32, 128])}
    if kind == "host":
        return {"op": "host", "rows": _log(rng, 128, 9216), "cin": 32 * _log(rng, 1, 24), "cout": 8 * _log(rng, 4, 128), "x": x, "y": y}
    if kind == "map":
        return {"op": "map", "batch": rng.randint(1, 16), "cin": 32 * _log(rng, 1, 24), "height": rng.randint(6, 60),
                "width": rng.randint(6, 60), "cout": _log(rng, 32, 1024), "x": x, "y": y,
                "zr": rng.choice([0.1, 0.2, 0.2, 0.3]), "bias": rng.random() < 0.5, "kept": rng.random() < 0.7}
    while True:
        rows, cin, cout = _log(rng, 64, 65536), _log(rng, 32, 4096), _log(rng, 32, 4096)
        if rng.random() < 0.6:       # most layers of a network have channel counts of this kind
            cin = max(32, cin // 32 * 32)
        if rng.random() < 0.6:
            cout = max(32, cout // 8 * 8)
        if rows * cin * cout <= MAX_MACS and rows * max(cin, cout) <= MAX_CELLS:
            break
    g = rng.choice([32, 32, 32, 32, 64, 128, -1])
    g = (cin + 31) // 32 * 32 if g < 0 else g      # -1: one step per token
    c = layer("", rows, cin, cout, x, y, g, steps=rng.choice(["exact"] * 5 + ["pow2"]), zr=rng.choice([0.1, 0.2, 0.2, 0.2, 0.3]),
              p=rng.choice([1.0, 1.0, 1.0, 1.0, 0.9]), bias=rng.random() < 0.5, kept=rng.random() < 0.7)
    del c["name"]
    return c


class _Inputs:
    """Seeded inputs made on the GPU: the distributions of synth_inputs.py."""

    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(1000003 * int(seed) + 17)

    def normal(self, *shape):
        return torch.randn(*shape, generator=self.gen, device="cuda")

    def tokens(self, rows, cin, dtype):
        """Most tokens N(0, s^2) with ln s ~ N(0, 0.5), every tenth one a background token 20 t_3, 1 % thin structured
        low-amplitude ones, 2 % outlier tokens x50."""
        u = torch.rand(rows, generator=self.gen, device="cuda")
        x = self.normal(rows, cin)
        gain = torch.exp(0.5 * self.normal(rows))
        gain = torch.where(u > 0.98, 50.0 * gain, gain)
        x *= gain[:, None]
        bg = torch.nonzero(u < 0.10).flatten()
        if bg.numel():
            t = self.normal(4, bg.numel(), cin)
            x[bg] = 20.0 * t[3] / torch.sqrt((t[:3] ** 2).mean(0))
        bd = torch.nonzero((u >= 0.10) & (u < 0.11)).flatten()
        if bd.numel():
            f = torch.randint(1, 4, (bd.numel(), 1), generator=self.gen, device="cuda")
            c = torch.arange(cin, device="cuda")
            x[bd] = 0.05 * (torch.cos(2 * math.pi * f * c / cin + self.normal(bd.numel(), 1)) + 0.1 * self.normal(bd.numel(), cin))
        return x.to(dtype)


def prepare(case, seed):
    inp = _Inputs(seed)
    op = case["op"]
    if op == "encoder":
        s = {"op": op, "layers": []}
        need = 0
        for _, m, i, o in synth_inputs.sweep_shapes(case["batch"]):
            wc, ws = tdq.quantize_weight(0.02 * inp.normal(o, i))
            s["layers"].append(dict(x=inp.tokens(m, i, torch.bfloat16), wc=wc, ws=ws,
                                    codes=torch.empty((m, i // 2), dtype=torch.uint8, device="cuda"),
                                    scale=torch.empty((m, i // 32), dtype=torch.float32, device="cuda"),
                                    y=torch.empty((m, o), dtype=torch.float32, device="cuda")))
            need = max(need, tdq.linear_workspace(m, i, o, 32, "cuda").numel())
        s["workspace"] = torch.zeros((need,), dtype=torch.uint8, device="cuda")
        return s
    cin, cout = case["cin"], case["cout"]
    if op == "weights":
        return {"op": op, "w": (0.02 * inp.normal(cout, cin)).to(DTYPES[case["x"]]), "g": case["g"]}
    g = case.get("g", 32)
    flags = tdq.ENABLE_C1 | tdq.ENABLE_C2 | (tdq.POW2_STEP if case.get("steps") == "pow2" else 0)
    s = {"op": op, "g": g, "pow2": case.get("steps") == "pow2", "out_dtype": DTYPES[case["y"]], "bias": None,
         "params": tdq.act_params(g=g, zr=case.get("zr", 0.2), p=case.get("p", 1.0), flags=flags), "codes": None,
         "scale": None, "y": None, "workspace": None}
    s["wc"], s["ws"] = tdq.quantize_weight(0.02 * inp.normal(cout, cin), pad_to=g)
    if case.get("bias"):
        s["bias"] = 0.1 * inp.normal(cout)
    if op == "map":
        b, h, w = case["batch"], case["height"], case["width"]
        rows = b * h * w
        s["x"] = inp.tokens(rows, cin, DTYPES[case["x"]]).view(b, h, w, cin).permute(0, 3, 1, 2).contiguous()
    else:
        rows = case["rows"]
        s["x"] = inp.tokens(rows, cin, DTYPES[case["x"]])
    if op == "host":
        s["x"] = s["x"].cpu().pin_memory()
        s["y"] = torch.empty((rows, cout), dtype=s["out_dtype"]).pin_memory()
    elif case["kept"]:
        k = (cin + g - 1) // g
        s["codes"] = torch.empty((rows, k * g // 2), dtype=torch.uint8, device="cuda")
        s["scale"] = torch.empty((rows, k), dtype=torch.float32, device="cuda")
        s["y"] = torch.empty((rows, cout), dtype=s["out_dtype"], device="cuda")
        s["workspace"] = tdq.linear_workspace(rows, k * g, cout, g, "cuda")
    return s


def run(s):
    op = s["op"]
    if op == "encoder":
        out = []
        for l in s["layers"]:
            tdq.quantize_act(l["x"], codes=l["codes"], scale=l["scale"])
            out.append(tdq.w4a4_linear(l["codes"], l["scale"], l["wc"], l["ws"], y=l["y"], workspace=s["workspace"]))
        return out
    if op == "weights":
        return tdq.quantize_weight(s["w"], s["g"])
    if op == "host":
        y, s["buffers"] = tdq.quant_linear_host(s["x"], s["wc"], s["ws"], params=s["params"], out_dtype=s["out_dtype"], y_host=s["y"])
        return y
    quantize = tdq.quantize_act_nchw if op == "map" else tdq.quantize_act
    linear = tdq.w4a4_linear_pow2 if s["pow2"] else tdq.w4a4_linear
    codes, scale = quantize(s["x"], s["params"], codes=s["codes"], scale=s["scale"])
    y = linear(codes, scale, s["wc"], s["ws"], s["bias"], g=s["g"], out_dtype=s["out_dtype"], y=s["y"], workspace=s["workspace"])
    return codes, scale, y


def _layer_work(rows, cin, cout, x, y, g, bias):
    """Activations, packed weight codes and channel constants in; codes, steps and outputs out."""
    k = (cin + g - 1) // g
    xb, yb = (4 if t == "fp32" else 2 for t in (x, y))
    return {"bytes": rows * cin * xb + cout * k * g // 2 + 4 * cout * (2 if bias else 1) + rows * (k * g // 2 + 4 * k) + rows * cout * yb,
            "flops": 2 * rows * k * g * cout}


def work(case):
    op = case["op"]
    if op == "encoder":
        ws = [_layer_work(m, i, o, "bf16", "fp32", 32, False) for _, m, i, o in synth_inputs.sweep_shapes(case["batch"])]
        return {"bytes": sum(w["bytes"] for w in ws), "flops": sum(w["flops"] for w in ws)}
    cin, cout = case["cin"], case["cout"]
    if op == "weights":
        return {"bytes": cout * (cin * (4 if case["x"] == "fp32" else 2) + (cin + case["g"] - 1) // case["g"] * case["g"] // 2 + 4), "flops": 0}
    rows = case["batch"] * case["height"] * case["width"] if op == "map" else case["rows"]
    return _layer_work(rows, cin, cout, case["x"], case["y"], case.get("g", 32), case.get("bias", False))


def tolerance(case):
    """Codes are whole numbers and stay the same; outputs are binary32 sums, rounded once more for 16-bit types."""
    if case["op"] == "weights":
        return "exact"
    return {"rel": {"fp32": 1e-5, "bf16": 4e-3, "fp16": 5e-4}[case.get("y", "fp32")]}
