"""The one-launch kernel of the linear layer for no more 128 x 64 tiles than SMs, at the edges of its tiles and of its dispatch:
every number of groups modulo its eight TMEM slots and its stages, groups that end inside a stage, ragged rows and columns,
each output type with and without tensor stores, codes at the ends of their range, nothing written past the last column."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si

pytestmark = pytest.mark.gpu


def _check(xc, xs, wc, ws, g, O):
    from paper_2604_16855_b200 import tdq
    M, K = xs.shape
    bias = torch.randn((O,), device="cuda", generator=torch.Generator("cuda").manual_seed(O))
    want = oracle.w4a4_linear(xc.cpu().numpy(), xs.cpu().numpy(), wc.cpu().numpy(), ws.cpu().numpy(), bias=bias.cpu().numpy(), g=g)
    wsp = tdq.linear_workspace(M, K * g, O, g, "cuda")
    n0 = tdq.kernel_launch_count()
    y = tdq.w4a4_linear(xc, xs, wc, ws, bias, g=g, workspace=wsp)
    assert tdq.kernel_launch_count() - n0 == (2 if g == 32 and K > 28 else 1)   # no expansion but beyond the rule's end
    assert tdq.workspace_status(wsp) == (tdq.OK, 0)
    # K products, K sums, the scaling and the bias, each rounded once (2^-24 of a partial sum)
    t = want["t_abs"] + np.abs(bias.cpu().numpy())[None, :]
    err = np.abs(y.cpu().numpy().astype(np.float64) - want["y_d"])
    assert (err <= np.maximum(1e-5 * np.abs(want["y_d"]), (K + 3) * 2.0 ** -24 * t)).all()
    # the group sums' kernel adds in the same order
    acc = torch.zeros((M, O, K), dtype=torch.int32, device="cuda")
    assert torch.equal(tdq.w4a4_linear(xc, xs, wc, ws, bias, g=g, workspace=wsp, acc_debug=acc), y)
    O8 = (O + 7) // 8 * 8
    for dt in (torch.float32, torch.bfloat16, torch.float16):
        for pitch, first in ((O8 + 8, 8), (O8 + 1, 0), (O8 + 2, 2), (O8 + 3, 1)):
            buf = torch.full((M, pitch), 3.0, dtype=dt, device="cuda")
            z = tdq.w4a4_linear(xc, xs, wc, ws, bias, g=g, y=buf[:, first:first + O], workspace=wsp)
            assert tdq.workspace_status(wsp) == (tdq.OK, 0)
            assert torch.equal(z, y.to(dt))
            assert bool((buf[:, :first] == 3.0).all()) and bool((buf[:, first + O:] == 3.0).all())


@pytest.mark.parametrize("M,O", [(1, 1), (127, 63), (129, 65), (300, 130), (1000, 516), (130, 4670)])
@pytest.mark.parametrize("g,K", [(32, k) for k in (1, 3, 4, 5, 6, 7, 8, 9, 11, 12, 13, 15, 16, 17, 24, 27, 28, 29)] + [(64, k) for k in (1, 2, 3, 7, 8, 9, 16)] +
                         [(96, 1), (96, 4), (96, 9), (128, 1), (128, 5), (128, 8), (128, 16), (160, 3), (256, 3), (320, 1), (512, 4), (1312, 1), (2048, 1)])
def test_shapes(M, O, g, K):
    from paper_2604_16855_b200 import tdq
    if M * O * K > 4_000_000:
        M = 140
    rng = np.random.default_rng(M + O + K * g)
    x = si.token_mixture(rng, 1, M, K * g, sigma_log_std=0.5, bg_frac=0.1, bg_nu=3.0, bg_amp=20.0).reshape(M, K * g)
    xc, xs = tdq.quantize_act(torch.from_numpy(x).cuda(), tdq.act_params(g=g))
    wc, ws = tdq.quantize_weight(torch.from_numpy(si.weights(rng, O, K * g)).cuda(), pad_to=g)
    _check(xc, xs, wc, ws, g, O)


@pytest.mark.parametrize("g,K", [(32, 9), (64, 5), (256, 4), (2048, 1)])
@pytest.mark.parametrize("x,w", [(0x88, 0x88), (0x88, 0x77), (0x77, 0x88), (0x77, 0x77), (0x00, 0x88), (0x88, 0x00), (0x8F, 0x71), (None, None)])
def test_extreme_codes(g, K, x, w):
    """Codes from -8 to 7, also those no quantizer makes."""
    M, O = 131, 70
    rng = np.random.default_rng(g)
    shape_x, shape_w = (M, K * g // 2), (O, K * g // 2)
    xc = torch.from_numpy(np.full(shape_x, x, np.uint8) if x is not None else rng.integers(0, 256, shape_x, dtype=np.uint8)).cuda()
    wc = torch.from_numpy(np.full(shape_w, w, np.uint8) if w is not None else rng.integers(0, 256, shape_w, dtype=np.uint8)).cuda()
    xs = torch.from_numpy(rng.uniform(0.1, 2.0, (M, K)).astype(np.float32)).cuda()
    ws = torch.from_numpy(rng.uniform(0.1, 2.0, O).astype(np.float32)).cuda()
    _check(xc, xs, wc, ws, g, O)


@pytest.mark.parametrize("g,K", [(32, 9), (64, 5), (96, 3), (128, 4), (160, 3), (256, 4), (768, 1)])
@pytest.mark.parametrize("step,channel", [(1e-8, 1e-30), (2e34, 1e-30), (1e-37, 1e37), (1e-30, 1.0), (0.0, 1.0), (float("inf"), 1.0), (1.0, float("inf")), (float("nan"), 1.0)])
def test_ends_of_the_range(g, K, step, channel):
    """Steps and channel scales at which a product or a sum nears the ends of binary32: the same bits, infinities and NaNs as the
    kernel that writes the group sums, which takes every layer."""
    from paper_2604_16855_b200 import tdq
    M, O = 131, 72
    rng = np.random.default_rng(g + K)
    xc = torch.from_numpy(rng.integers(0, 256, (M, K * g // 2), dtype=np.uint8)).cuda()
    wc = torch.from_numpy(rng.integers(0, 256, (O, K * g // 2), dtype=np.uint8)).cuda()
    xs = torch.from_numpy(rng.uniform(0.1, 2.0, (M, K)).astype(np.float32)).cuda() * step
    ws = torch.from_numpy(rng.uniform(0.1, 2.0, O).astype(np.float32)).cuda() * channel
    bias = torch.from_numpy(rng.standard_normal(O).astype(np.float32)).cuda()
    wsp = tdq.linear_workspace(M, K * g, O, g, "cuda")
    acc = torch.zeros((M, O, K), dtype=torch.int32, device="cuda")
    want = tdq.w4a4_linear(xc, xs, wc, ws, bias, g=g, workspace=wsp, acc_debug=acc)
    n0 = tdq.kernel_launch_count()
    got = tdq.w4a4_linear(xc, xs, wc, ws, bias, g=g, workspace=wsp)
    assert tdq.kernel_launch_count() - n0 == 1                # this kernel, not the expansion and another one
    assert torch.equal(torch.isnan(got), torch.isnan(want))
    assert torch.equal(torch.nan_to_num(got, nan=0.0, posinf=3e38, neginf=-3e38), torch.nan_to_num(want, nan=0.0, posinf=3e38, neginf=-3e38))
