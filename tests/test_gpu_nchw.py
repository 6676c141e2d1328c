"""The channel-major quantizer at the edges of its 64-position blocks, with channel rows on and off the 16-byte grid, against the
row-major kernel on the permuted tensor (itself pinned to the oracle): the same bits."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("H,W", [(1, 1), (1, 8), (3, 7), (1, 63), (8, 8), (1, 65), (9, 8), (12, 12), (1, 127), (16, 8), (11, 12), (17, 19), (24, 24)])
@pytest.mark.parametrize("B,C,first", [(1, 32, 0), (3, 96, 0), (2, 64, 1)])
def test_shapes(B, C, H, W, first, dtype):
    from paper_2604_16855_b200 import tdq
    gen = torch.Generator("cuda").manual_seed(B + C + H * W)
    store = torch.randn((first + B * C * H * W,), device="cuda", generator=gen).to(dtype)
    x = store[first:].view(B, C, H, W)          # first = 1: no row of x is on the 16-byte grid
    for zr in (0.1, 0.2, 0.3):
        p = tdq.act_params(zr=zr)
        codes, scale = tdq.quantize_act_nchw(x, p)
        want_codes, want_scale = tdq.quantize_act(x.permute(0, 2, 3, 1).reshape(-1, C).contiguous(), p)
        assert torch.equal(codes.view(want_codes.shape), want_codes) and torch.equal(scale.view(want_scale.shape), want_scale)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("B,C,H,W", [(16, 512, 12, 12), (70, 768, 9, 9), (700, 160, 1, 3), (1500, 32, 13, 5), (900, 32, 1, 1)])
def test_blocks_across_images(B, C, H, W, dtype):
    """Maps whose blocks of positions run on from one image to the next."""
    from paper_2604_16855_b200 import tdq
    x = torch.randn((B, C, H, W), device="cuda", generator=torch.Generator("cuda").manual_seed(B)).to(dtype)
    codes = torch.full((B * H * W + 1, C // 2), 77, dtype=torch.uint8, device="cuda")
    scale = torch.full((B * H * W + 1, C // 32), -1.0, device="cuda")
    tdq.quantize_act_nchw(x, codes=codes[:-1], scale=scale[:-1])
    want_codes, want_scale = tdq.quantize_act(x.permute(0, 2, 3, 1).reshape(-1, C).contiguous())
    assert torch.equal(codes[:-1], want_codes.view(-1, C // 2)) and torch.equal(scale[:-1], want_scale.view(-1, C // 32))
    assert bool((codes[-1] == 77).all()) and bool((scale[-1] == -1.0).all())


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("B,C,H,W,long", [(16, 512, 33, 35, False), (17, 768, 24, 24, False), (16, 512, 41, 37, True), (28, 768, 24, 24, True)])
def test_long_maps(B, C, H, W, long, dtype):
    """bf16 maps of 40 and more blocks per SM have an instance of their own, whose rare paths (a large mean, huge numbers) are calls; both
    sides of that line, against calls on one image at a time (short, so on the other instance) and, at some positions, the oracle."""
    from paper_2604_16855_b200 import tdq
    assert (B * (C // 32) * ((H * W + 63) // 64) >= 40 * torch.cuda.get_device_properties(0).multi_processor_count) == long
    x = torch.randn((B, C, H, W), device="cuda", generator=torch.Generator("cuda").manual_seed(C))
    x[:, :, 1::7] += 30.0
    x[:, :, 3::7] *= 1e32
    x = x.to(dtype)
    rows = x.permute(0, 2, 3, 1).reshape(-1, C)
    some = list(range(0, rows.shape[0], 199)) + [W, 3 * W, rows.shape[0] - 1]
    for zr in (0.1, 0.2, 0.3, 0.4, 0.5, 1.0):
        p = tdq.act_params(zr=zr)
        codes, scale = tdq.quantize_act_nchw(x, p)
        codes, scale = codes.view(B, H * W, C // 2), scale.view(B, H * W, C // 32)
        for b in range(B):
            c, s = tdq.quantize_act_nchw(x[b:b + 1], p)
            assert torch.equal(codes[b], c.view(codes[b].shape)) and torch.equal(scale[b], s.view(scale[b].shape))
        want = oracle.quantize_act(rows[some].float().cpu().numpy(), zr=zr)
        assert np.array_equal(codes.view(-1, C // 2)[some].cpu().numpy(), want["codes"])
        assert np.array_equal(scale.view(-1, C // 32)[some].cpu().numpy(), want["scale"])
