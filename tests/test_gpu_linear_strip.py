"""The one-launch kernel of the linear layer that keeps a row block's operands for a run of column tiles (g = 32, a few tiles per
SM), at the edges of its dispatch: every number of groups modulo four, one to six chunks, row blocks that end inside a block's
run and reuse another's place, ragged rows and columns, an empty second half, each output type, nothing written past the
last column, codes at the ends of their range, and the same bits under capture."""
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


def _check(xc, xs, wc, ws, O):
    from paper_2604_16855_b200 import tdq
    M, K = xs.shape
    bias = torch.randn((O,), device="cuda", generator=torch.Generator("cuda").manual_seed(O))
    wsp = tdq.linear_workspace(M, K * 32, O, 32, "cuda")
    # a y that tensor stores cannot write goes to another kernel, which computes the same bits
    odd = torch.empty((M, O + 1), device="cuda")[:, 1:]
    ref = tdq.w4a4_linear(xc, xs, wc, ws, bias, y=odd, workspace=wsp)
    for dt in (torch.float32, torch.bfloat16, torch.float16):
        buf = torch.full((M, O + 8), 3.0, dtype=dt, device="cuda")
        n0 = tdq.kernel_launch_count()
        y = tdq.w4a4_linear(xc, xs, wc, ws, bias, y=buf[:, :O], workspace=wsp)
        assert tdq.kernel_launch_count() - n0 == 1            # this kernel: the others expand the operands first at these sizes
        assert tdq.workspace_status(wsp) == (tdq.OK, 0)
        assert torch.equal(y, ref.to(dt))
        assert bool((buf[:, O:] == 3.0).all())
    rows = np.unique(np.concatenate([np.arange(min(M, 3)), np.random.default_rng(M).integers(0, M, 40), np.arange(max(M - 70, 0), M)]))
    want = oracle.w4a4_linear(xc.cpu().numpy()[rows], xs.cpu().numpy()[rows], wc.cpu().numpy(), ws.cpu().numpy(), bias=bias.cpu().numpy(), g=32)
    # K products, K sums, the scaling and the bias, each rounded once (2^-24 of a partial sum)
    t = want["t_abs"] + np.abs(bias.cpu().numpy())[None, :]
    err = np.abs(ref.cpu().numpy()[rows].astype(np.float64) - want["y_d"])
    assert (err <= np.maximum(1e-5 * np.abs(want["y_d"]), (K + 3) * 2.0 ** -24 * t)).all()
    return ref


# one to four groups (one chunk, six row blocks held), up to two and three chunks (three and two held), and one held beyond; tiles
# per SM from less than one to twelve; 72 and 136 outputs: an empty second half in the last or the only column tile
@pytest.mark.parametrize("M,O", [(20001, 200), (6000, 1032), (40000, 72), (18500, 136)])
@pytest.mark.parametrize("K", [1, 2, 3, 4, 5, 6, 7, 8, 9])
def test_short(M, O, K):
    _run(M, O, K)


@pytest.mark.parametrize("M,O,K", [(2305, 1000, 10), (1153, 1280, 11), (1152, 1536, 12), (9216, 264, 13), (8000, 520, 14), (2305, 1536, 15), (4609, 1288, 16),
                                   (18433, 128, 10), (18432, 72, 17), (30000, 104, 19), (36000, 128, 24), (20000, 128, 22)])
def test_long(M, O, K):
    _run(M, O, K)


def _run(M, O, K):
    from paper_2604_16855_b200 import tdq
    rng = np.random.default_rng(M + O + K)
    gen = torch.Generator("cuda").manual_seed(M)
    x = torch.randn((M, 32 * K), device="cuda", generator=gen) * torch.exp(0.5 * torch.randn((M, 1), device="cuda", generator=gen))
    xc, xs = tdq.quantize_act(x)
    wc, ws = tdq.quantize_weight(torch.from_numpy(si.weights(rng, O, 32 * K)).cuda())
    _check(xc, xs, wc, ws, O)


@pytest.mark.parametrize("x,w", [(0x88, 0x88), (0x88, 0x77), (0x77, 0x88), (0x77, 0x77), (0x00, 0x88), (0x88, 0x00), (0x8F, 0x71), (None, None)])
def test_extreme_codes(x, w):
    """Codes from -8 to 7, also those no quantizer makes."""
    M, O, K = 12000, 264, 6
    rng = np.random.default_rng(5)
    xc = torch.from_numpy(np.full((M, K * 16), x, np.uint8) if x is not None else rng.integers(0, 256, (M, K * 16), dtype=np.uint8)).cuda()
    wc = torch.from_numpy(np.full((O, K * 16), w, np.uint8) if w is not None else rng.integers(0, 256, (O, K * 16), dtype=np.uint8)).cuda()
    xs = torch.from_numpy(rng.uniform(0.1, 2.0, (M, K)).astype(np.float32)).cuda()
    ws = torch.from_numpy(rng.uniform(0.1, 2.0, O).astype(np.float32)).cuda()
    _check(xc, xs, wc, ws, O)


def test_under_capture():
    """From ten groups on a captured call may take another kernel."""
    from paper_2604_16855_b200 import tdq
    M, C, O = 9216, 320, 320
    x = torch.randn((M, C), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    xc, xs = tdq.quantize_act(x)
    wc, ws = tdq.quantize_weight(torch.from_numpy(si.weights(np.random.default_rng(1), O, C)).cuda())
    wsp = tdq.linear_workspace(M, C, O, 32, "cuda")
    n0 = tdq.kernel_launch_count()
    want = tdq.w4a4_linear(xc, xs, wc, ws, workspace=wsp)
    assert tdq.kernel_launch_count() - n0 == 1
    y = torch.empty_like(want)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        tdq.w4a4_linear(xc, xs, wc, ws, y=y, workspace=wsp)
    graph.replay()
    assert tdq.workspace_status(wsp) == (tdq.OK, 0)
    assert torch.equal(y, want)


FIRST_USE = """
import sys
import torch
from paper_2604_16855_b200 import tdq
warm, M, C, O = [int(v) for v in sys.argv[1:]]
gen = torch.Generator("cuda").manual_seed(M)
xc, xs = tdq.quantize_act(torch.randn((M, C), device="cuda", generator=gen))
wc, ws = tdq.quantize_weight(torch.randn((O, C), device="cuda", generator=gen))
wsp = tdq.linear_workspace(M, C, O, 32, "cuda")
y = torch.empty((M, O), device="cuda")
counts = []
if warm:
    n = tdq.kernel_launch_count()
    tdq.w4a4_linear(xc, xs, wc, ws, y=y, workspace=wsp)
    counts.append(tdq.kernel_launch_count() - n)
    y.zero_()
torch.cuda.synchronize()
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph):
    n = tdq.kernel_launch_count()
    tdq.w4a4_linear(xc, xs, wc, ws, y=y, workspace=wsp)
    counts.append(tdq.kernel_launch_count() - n)
graph.replay()
assert tdq.workspace_status(wsp) == (tdq.OK, 0)
z = tdq.w4a4_linear(xc, xs, wc, ws, workspace=wsp)
assert torch.equal(y, z), "the replay's bits differ"
print("launches", counts)
"""


# launches of the eager and of the captured call: one where this kernel wins in a graph too; expansion and another kernel where it
# does not (many groups; a last round of tiles that is mostly empty; half of the last column tile empty; wide binary32 outputs)
@pytest.mark.parametrize("M,C,O,captured", [(9216, 320, 320, 2), (2304, 288, 1280, 2), (64000, 128, 192, 2), (9216, 256, 1280, 2), (18432, 192, 768, 1), (1152, 512, 2048, 1)])
@pytest.mark.parametrize("warm", [0, 1])
def test_first_use_in_a_capture(M, C, O, captured, warm):
    """A process whose first launch of the layer's kernels is inside a capture, and one that has only called the layer eagerly
    before: the captured call takes the kernel that is the faster one in a graph, and its replay gives the eager call's bits."""
    r = subprocess.run([sys.executable, "-c", FIRST_USE, str(warm), str(M), str(C), str(O)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    assert "launches %s" % ([1, captured] if warm else [captured]) in r.stdout
