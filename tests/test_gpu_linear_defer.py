"""The kernel of the linear layer that does a tile's epilogue during the next tile (g = 32, 64, 128, several tiles per SM), at the
edges of its dispatch: every number of groups modulo four, fewer groups than the pieces of an epilogue, both plans for the
steps, ragged rows and columns, blocks with one tile more than others, each output type, nothing written past the last column."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


SHAPES = [(10113, 320, 1024, 32), (5249, 352, 1920, 32), (10240, 384, 1016, 32), (9999, 416, 1024, 32),
          (9345, 768, 776, 32), (75777, 320, 128, 32), (9473, 1504, 760, 32), (10000, 1536, 768, 32),
          (2305, 576, 1280, 64), (5000, 1088, 640, 64), (2500, 4096, 1024, 64), (9600, 512, 760, 64),
          (9600, 512, 1016, 128), (2305, 640, 1272, 128), (2400, 768, 2048, 128), (2305, 4096, 1280, 128)]


@pytest.mark.parametrize("M,C,O,g", SHAPES)
def test_shapes(M, C, O, g):
    from paper_2604_16855_b200 import tdq
    rng = np.random.default_rng(M + C + O)
    gen = torch.Generator("cuda").manual_seed(M)
    x = torch.randn((M, C), device="cuda", generator=gen) * torch.exp(0.5 * torch.randn((M, 1), device="cuda", generator=gen))
    xc, xs = tdq.quantize_act(x, tdq.act_params(g=g))
    wc, ws = tdq.quantize_weight(torch.from_numpy(si.weights(rng, O, C)).cuda(), pad_to=g)
    bias = torch.from_numpy(rng.standard_normal(O).astype(np.float32)).cuda()
    wsp = tdq.linear_workspace(M, C, O, g, "cuda")
    out = {}
    for dt in (torch.float32, torch.bfloat16, torch.float16):
        buf = torch.full((M, O + 8), 3.0, dtype=dt, device="cuda")
        out[dt] = tdq.w4a4_linear(xc, xs, wc, ws, bias, g=g, y=buf[:, :O], workspace=wsp)
        assert tdq.workspace_status(wsp) == (tdq.OK, 0)
        assert bool((buf[:, O:] == 3.0).all())
    y = out[torch.float32]
    assert torch.equal(out[torch.bfloat16], y.to(torch.bfloat16)) and torch.equal(out[torch.float16], y.to(torch.float16))
    # the kernels for a y that tensor stores cannot write compute the same bits
    odd = torch.empty((M, O + 1), device="cuda")[:, 1:]
    assert torch.equal(tdq.w4a4_linear(xc, xs, wc, ws, bias, g=g, y=odd, workspace=wsp), y)
    assert torch.equal(tdq.w4a4_linear(xc, xs, wc, ws, g=g, workspace=wsp) + bias, tdq.w4a4_linear(xc, xs, wc, ws, g=g, y=odd, workspace=wsp) + bias)
    rows = np.unique(np.concatenate([np.arange(3), rng.integers(0, M, 60), np.arange(M - 130, M)]))
    want = oracle.w4a4_linear(xc.cpu().numpy()[rows], xs.cpu().numpy()[rows], wc.cpu().numpy(), ws.cpu().numpy(), bias=bias.cpu().numpy(), g=g)
    # K products, K sums, the scaling and the bias, each rounded once (2^-24 of a partial sum)
    t = want["t_abs"] + np.abs(bias.cpu().numpy())[None, :]
    err = np.abs(y.cpu().numpy()[rows].astype(np.float64) - want["y_d"])
    assert (err <= np.maximum(1e-5 * np.abs(want["y_d"]), (C // g + 3) * 2.0 ** -24 * t)).all()


WHICH = """
import sys
import torch
from torch.profiler import ProfilerActivity, profile
from paper_2604_16855_b200 import tdq
shapes = %s
calls = []
for M, C, O, g in shapes:
    codes, wcodes = [torch.zeros((n, C // 2), dtype=torch.uint8, device="cuda") for n in (M, O)]
    calls.append((codes, torch.ones((M, C // g), device="cuda"), wcodes, torch.ones((O,), device="cuda"), g, torch.empty((M, O), device="cuda")))
torch.cuda.synchronize()
with profile(activities=[ProfilerActivity.CUDA]) as p:
    for codes, scale, wcodes, wscale, g, y in calls:
        tdq.w4a4_linear(codes, scale, wcodes, wscale, g=g, y=y)
    torch.cuda.synchronize()
names = [e.name for e in sorted((e for e in p.events() if "w4a4" in e.name), key=lambda e: e.time_range.start)]
assert len(names) == len(shapes), names
for n in names:
    print("KERNEL", n)
"""


def test_these_shapes_run_it():
    """The shapes above take this kernel; the same ones with a row block less than its rule asks for do not."""
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    def bound(C, O, g):                                       # the most row blocks that another kernel takes
        tiles_n = -(-O // 128)
        per_sm = (3 if C >= 768 else 4) if g == 32 else 3 if C <= 512 else 1
        return per_sm * sm // tiles_n * 128
    few = [(bound(C, O, g), C, O, g) for C, O, g in ((320, 1024, 32), (768, 768, 32), (512, 1024, 64), (512, 1024, 128), (768, 1280, 64))]
    r = subprocess.run([sys.executable, "-c", WHICH % (SHAPES + few)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    names = [line for line in r.stdout.splitlines() if line.startswith("KERNEL")]
    assert all("w4a4_defer_kernel" in n for n in names[:len(SHAPES)]), names
    assert not any("w4a4_defer_kernel" in n for n in names[len(SHAPES):]), names
