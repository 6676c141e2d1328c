"""The row-major quantizer at g = 32 at the edges of its 64-group blocks and 32-group warps: dense rows and rows with a pitch, both
input types, every block boundary, against the oracle; nothing written past the last group."""
import json
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


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("pad", [0, 8])
@pytest.mark.parametrize("M,K", [(1, 1), (1, 3), (31, 1), (32, 1), (33, 1), (1, 63), (64, 1), (13, 5), (9, 7), (19, 5), (96, 1), (1, 127), (64, 2), (43, 3), (5, 64)])
def test_block_edges(M, K, pad, dtype):
    from paper_2604_16855_b200 import tdq
    rng = np.random.default_rng(100 * M + K)
    x = si.token_mixture(rng, 1, M, 32 * K, sigma_log_std=0.5, bg_frac=0.1, bg_nu=3.0, bg_amp=20.0).reshape(M, 32 * K)
    store = torch.zeros((M, 32 * K + pad), dtype=dtype, device="cuda")
    store[:, :32 * K] = torch.from_numpy(x).to(dtype)
    xt = store[:, :32 * K]
    want = oracle.quantize_act(xt.float().cpu().numpy())
    codes = torch.full((M + 1, 16 * K), 77, dtype=torch.uint8, device="cuda")
    scale = torch.full((M + 1, K), -1.0, device="cuda")
    tdq.quantize_act(xt, codes=codes[:M], scale=scale[:M])
    assert np.array_equal(codes[:M].cpu().numpy(), want["codes"]) and np.array_equal(scale[:M].cpu().numpy(), want["scale"])
    assert bool((codes[M] == 77).all()) and bool((scale[M] == -1.0).all())


def _rows_with_rare_ones(M, C, seed):
    """Rows among which some have a large mean (the deviation in binary64), some huge numbers (IEEE division) and some nothing but zeros."""
    gen = torch.Generator("cuda").manual_seed(seed)
    x = torch.randn((M, C), device="cuda", generator=gen) * torch.exp(0.5 * torch.randn((M, 1), device="cuda", generator=gen))
    x[5::50] += 30.0
    x[7::50] *= 1e32
    x[9::50] = 0.0
    return x


def _check_long(xt, p, **oracle_args):
    """Codes and steps of a long input: nothing written past them, the same bits as block by block of rows (too short for the instances
    of long inputs), and the oracle's on some rows."""
    from paper_2604_16855_b200 import tdq
    M, C = xt.shape
    codes = torch.full((M + 1, C // 2), 77, dtype=torch.uint8, device="cuda")
    scale = torch.full((M + 1, C // 32), -1.0, device="cuda")
    offset = torch.full((M + 1, C // 32), -1.0, device="cuda")
    tdq.quantize_act(xt, p, codes=codes[:M], scale=scale[:M], offset=offset[:M])
    assert bool((codes[M] == 77).all()) and bool((scale[M] == -1.0).all())
    assert bool((offset[:M] == 0.0).all()) and bool((offset[M] == -1.0).all())
    for r in range(0, M, 1000):
        c, s = tdq.quantize_act(xt[r:r + 1000], p)
        assert torch.equal(c, codes[r:min(r + 1000, M)]) and torch.equal(s, scale[r:min(r + 1000, M)])
    some = list(range(0, M, 61)) + [5, 7, 9, M - 1]
    want = oracle.quantize_act(xt[some].float().cpu().numpy(), **oracle_args)
    assert np.array_equal(codes[some].cpu().numpy(), want["codes"]) and np.array_equal(scale[some].cpu().numpy(), want["scale"])


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("zr", [0.1, 0.2, 0.3, 0.4, 0.5, 1.0])
@pytest.mark.parametrize("M,K,pad,long", [(7301, 32, 0, False), (3701, 63, 8, False), (12001, 32, 0, True), (6101, 63, 8, True)])
def test_long_inputs(M, K, pad, long, zr, dtype):
    """bf16 inputs of 40 and more blocks per SM have an instance of their own for each of these zero-bin ranks, whose rare paths are
    calls; both sides of that line."""
    from paper_2604_16855_b200 import tdq
    assert ((M * K + 63) // 64 >= 40 * torch.cuda.get_device_properties(0).multi_processor_count) == long and M * K % 64
    store = torch.zeros((M, 32 * K + pad), dtype=dtype, device="cuda")
    store[:, :32 * K] = _rows_with_rare_ones(M, 32 * K, M + K).to(dtype)
    _check_long(store[:, :32 * K], tdq.act_params(zr=zr), zr=zr)


@pytest.mark.parametrize("flags", [0, oracle.ENABLE_C1, oracle.ENABLE_C2, oracle.ENABLE_C1 | oracle.ENABLE_C2 | oracle.POW2_STEP])
def test_long_inputs_by_setting(flags):
    """The same with the bounds off, with one of them, and with power-of-two steps."""
    from paper_2604_16855_b200 import tdq
    _check_long(_rows_with_rare_ones(12001, 1024, 11).to(torch.bfloat16), tdq.act_params(flags=flags), flags=flags)


RESIDENCY = """
import json, os, sys, tempfile
import torch
from torch.profiler import ProfilerActivity, profile
from paper_2604_16855_b200 import tdq
dtype = getattr(torch, sys.argv[1])
rows, maps = {                         # blocks per SM: maps by blocks of their own for each image, and across the images
    "few": ((18944, 128), [(2, 64, 24, 24), (70, 64, 9, 9)]),                # 8, 0.2, 1.2
    "short": ((9216, 320), [(16, 320, 24, 24), (64, 512, 9, 9)]),            # 9.7, 9.7, 8.8
    "below": ((15000, 768), [(16, 512, 35, 40)]),                            # 38, 38
    "long": ((18464, 768), [(16, 512, 60, 60)])}[sys.argv[2]]                # 47, 99
x = torch.randn(rows, device="cuda").to(dtype)
maps = [torch.randn(m, device="cuda").to(dtype) for m in maps]
with profile(activities=[ProfilerActivity.CUDA]) as prof:
    for zr, p in [(0.1, 1.0), (0.2, 1.0), (1.0, 1.0)] + [(0.35, 1.0), (0.2, 0.9), (0.3, 0.5)] * (sys.argv[2] in ("few", "short")):
        tdq.quantize_act(x, tdq.act_params(zr=zr, p=p))
    for zr in (0.1, 0.2, 1.0):
        for m in maps:
            tdq.quantize_act_nchw(m, tdq.act_params(zr=zr))
    torch.cuda.synchronize()
with tempfile.TemporaryDirectory() as d:
    prof.export_chrome_trace(os.path.join(d, "t.json"))
    for e in json.load(open(os.path.join(d, "t.json")))["traceEvents"]:
        if e.get("cat") == "kernel" and "act_g32" in e["name"]:
            print(json.dumps([e["name"], e["args"]["registers per thread"], e["args"]["block"][0]]))
"""


@pytest.mark.parametrize("dtype", ["bfloat16", "float32"])
@pytest.mark.parametrize("length,launches", [("few", 6 + 3 * 2), ("short", 6 + 3 * 2), ("below", 3 + 3), ("long", 3 + 3)])
def test_resident_blocks(length, launches, dtype):
    """Inputs of up to eight blocks per SM may take the registers of eight (bf16 rows have no use for them); those of more run ten at once;
    bf16 inputs of 40 and more have instances of which still more fit, long fp32 inputs have not (more blocks per SM take the room in which
    the layer behind starts)."""
    assert torch.cuda.get_device_properties(0).multi_processor_count == 148    # what the sizes are made for
    r = subprocess.run([sys.executable, "-c", RESIDENCY, dtype, length], cwd=ROOT, capture_output=True, text=True, timeout=300)   # the profiler stays out of this process
    assert r.returncode == 0, r.stderr
    kernels = [json.loads(line) for line in r.stdout.splitlines()]
    assert len(kernels) == launches and {n.split("<")[0].split("::")[-1] for n, _, _ in kernels} == {"act_g32_kernel", "act_g32_nchw_kernel"}
    for name, registers, threads in kernels:
        warp = -(-registers * 32 // 256) * 256            # a warp's registers come in pieces of 256, each scheduler has 16384
        blocks = 4 * (16384 // warp) * 32 // threads
        if length == "few" and (dtype == "float32" or "nchw" in name):
            assert blocks == 8, (name, registers)
        elif (length, dtype) == ("long", "bfloat16"):
            assert blocks >= 14, (name, registers)
        else:
            assert 10 <= blocks <= 12, (name, registers)
