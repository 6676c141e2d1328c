"""The quantizer kernel for wide groups and unaligned rows at the edges of its instances: every width at which the lanes
per group or the chunks per lane change, remainders of a row, every load width, both ranks, ties and zeros."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from parity_utils import compare_quantizer, to_cuda

pytestmark = pytest.mark.gpu


def _rows(rng, M, C):
    x = si.token_mixture(rng, 1, M, C, sigma_log_std=0.5, bg_frac=0.1, bg_nu=3.0, bg_amp=20.0).reshape(M, C)
    x[1::7] += 3.0                                          # the dispersion bound is the minimum
    x[2::7] = np.maximum(x[2::7] - 0.8, 0.0)                # more zeros than the zero-bin rank
    x[3::7] = np.round(x[3::7] * 4.0) / 4.0                 # ties
    x[4] = 0.0
    x[5] = np.where(np.arange(C) % 3 == 0, 1e-9, -2e-9)     # below the floors
    x[6, ::5] = 3e4
    return x


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("g", [8, 24, 32, 40, 64, 72, 96, 104, 128, 136, 192, 200, 256, 264, 384, 392, 512, 520, 768, 776,
                               1024, 1032, 1536, 1544, 2048, 2056, 3072, 3080, 4096])
def test_widths_and_remainders(g, bf16):
    from paper_2604_16855_b200 import tdq
    rng = np.random.default_rng(g)
    for C, offset in ((2 * g, 0), (2 * g + 13, 0), (g + 6, 2), (max(g - 3, 5), 1)):   # offset: first channel of a wider matrix
        full = _rows(rng, 23, C + offset + 3)
        full = si.f32_to_bf16_bits(full) if bf16 else full
        x = np.ascontiguousarray(full[:, offset:offset + C])
        for kw in (dict(), dict(p=0.9, zr=0.5), dict(tau=0.4, zr=0.05, flags=7)):
            ref = oracle.quantize_act(x, g=g, **kw)
            params = tdq.act_params(g=g, tau=kw.get("tau", 1.0), zr=kw.get("zr", 0.2), p=kw.get("p", 1.0), flags=kw.get("flags", 3))
            codes, scale = tdq.quantize_act(to_cuda(full, bf16=bf16)[:, offset:offset + C], params)
            rep = compare_quantizer(si.bf16_bits_to_f32(x) if bf16 else x, g, ref, codes.cpu().numpy(), scale.cpu().numpy())
            assert rep["scale_max_rel"] <= 1e-6, (C, offset, kw, rep)


def test_many_groups():
    """More than one wave of blocks, a last warp that is only partly filled, offsets written."""
    from paper_2604_16855_b200 import tdq
    rng = np.random.default_rng(5)
    x = si.f32_to_bf16_bits(_rows(rng, 9001, 192))
    ref = oracle.quantize_act(x, g=64)
    off = torch.full((9001, 3), 7.0, device="cuda")
    codes, scale = tdq.quantize_act(to_cuda(x, bf16=True), tdq.act_params(g=64), offset=off)
    assert np.array_equal(codes.cpu().numpy(), ref["codes"]) and np.array_equal(scale.cpu().numpy(), ref["scale"])
    assert float(off.abs().max()) == 0.0


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("g", [8, 16, 24, 32])
def test_one_lane_per_group(g, bf16):
    """Groups that a single lane holds: a last warp with one group, cut chunks, every load width, codes that are only 4-byte
    aligned (which at g = 32 is what brings a group here)."""
    from paper_2604_16855_b200 import tdq
    rng = np.random.default_rng(100 + g)
    for M, C, pitch in ((97, g, g), (65, 5 * g, 5 * g + 8), (33, 3 * g - 3, 3 * g + 2), (129, 7 * g - 1, 7 * g + 1), (41, 2 * g + 4, 2 * g + 4)):
        full = _rows(rng, M, pitch)
        full = si.f32_to_bf16_bits(full) if bf16 else full
        x = np.ascontiguousarray(full[:, :C])
        K = (C + g - 1) // g
        buf = torch.full((M * K * g // 2 + 20,), 0x55, dtype=torch.uint8, device="cuda")
        for kw in (dict(), dict(p=0.8, zr=0.5), dict(tau=0.4, zr=1.0)):
            ref = oracle.quantize_act(x, g=g, **kw)
            params = tdq.act_params(g=g, tau=kw.get("tau", 1.0), zr=kw.get("zr", 0.2), p=kw.get("p", 1.0))
            codes, scale = tdq.quantize_act(to_cuda(full, bf16=bf16)[:, :C], params, codes=buf[4:-16].view(M, K * g // 2))
            rep = compare_quantizer(si.bf16_bits_to_f32(x) if bf16 else x, g, ref, codes.cpu().numpy(), scale.cpu().numpy())
            assert rep["scale_max_rel"] <= 1e-6, (M, C, kw, rep)
            assert bool((buf[:4] == 0x55).all()) and bool((buf[-16:] == 0x55).all())


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("g", [32, 64, 320, 768, 1024, 2048, 4096])
def test_dispersion_bound_beside_the_other_bounds(g, bf16):
    """The binary32 screen may only say that the dispersion bound is idle when it is: groups whose 7 tau sigma lies within a
    few 1e-6 to 2 % of the smaller of the other two bounds, on either side, with means up to where the screen gives up
    (mean^2 = 15 var) and past it."""
    from paper_2604_16855_b200 import tdq
    rng = np.random.default_rng(g)
    base = rng.standard_normal((8, g))
    base = base - base.mean(1, keepdims=True)
    base /= base.std(1, keepdims=True)
    x = (base + np.array([0.0, 0.3, 1.0, 2.0, 3.0, 3.8, 4.2, 30.0])[:, None]).astype(np.float32)
    full = si.f32_to_bf16_bits(x) if bf16 else x
    xf = si.bf16_bits_to_f32(full) if bf16 else x
    mags = np.sort(np.abs(xf), axis=1)
    other = np.minimum(mags[:, -1], np.float32(14.0) * mags[:, int(np.ceil(0.2 * g)) - 1]).astype(np.float64)
    ratio = other / (7.0 * xf.astype(np.float64).std(1))     # tau at which the two meet
    for row in range(8):
        for d in (-2e-2, -6e-3, -4e-3, -1e-3, -1e-4, -1e-5, -2e-6, 0.0, 2e-6, 1e-5, 1e-4, 1e-3, 4e-3, 6e-3, 2e-2):
            tau = float(np.float32(ratio[row] * (1.0 + d)))
            ref = oracle.quantize_act(full, g=g, tau=tau)
            codes, scale = tdq.quantize_act(to_cuda(full, bf16=bf16), tdq.act_params(g=g, tau=tau))
            compare_quantizer(xf, g, ref, codes.cpu().numpy(), scale.cpu().numpy())


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("g", [64, 96, 128, 1024, 2048, 4096])
def test_rank_search_edges(g, bf16):
    """Groups at the edges of the rank search: as many zeros as the zero-bin rank and one more or less, padding, few distinct
    values, magnitudes over the whole range, and a rank-k magnitude at, just above and just below a fourteenth of the base
    radius, above which the search may stop."""
    from paper_2604_16855_b200 import tdq
    rng = np.random.default_rng(200 + g)
    k = int(np.ceil(0.2 * g - 1e-6))
    rows = []
    for z in (k - 1, k, k + 1, g // 2, g - 1):
        x = rng.standard_normal(g)
        x[:z] = 0.0
        rows.append(x)
    rows.append(np.full(g, -0.3))
    rows.append(np.where(np.arange(g) % 3 == 0, 1.0, -14.0))
    rows.append(rng.choice([0.5, -1.0, 2.0, 6.0], g))
    rows.append(np.clip(rng.standard_normal(g) * 4.0, 0.0, 6.0))
    rows.append(10.0 ** rng.uniform(-30, 30, g))
    rows.append(10.0 ** rng.uniform(-44, -36, g))
    rows.append(1.0 + 1e-3 * np.arange(g))
    for top in (14.0, 13.9, 7.0 * 1.5, 1.234567e-3, 3e33):
        edge = np.float32(top) / np.float32(14.0)
        for ulps in (-66000, -65536, -2, -1, 0, 1, 2, 65536, 66000):
            v = (np.float32(edge).view(np.int32) + np.int32(ulps)).view(np.float32)
            x = rng.uniform(1.5, 13.0, g) * float(v)
            x[:k - 1] = rng.uniform(0.1, 0.9, k - 1) * float(v)
            x[k - 1] = v
            x[-1] = top
            rows.append(x)
    x = np.stack([rng.permutation(r) for r in rows]).astype(np.float32)
    x *= rng.choice([-1.0, 1.0], x.shape).astype(np.float32)
    for C in (g, g - g // 4 - 3):                            # the second: a quarter of the group is padding
        full = si.f32_to_bf16_bits(x[:, :C]) if bf16 else np.ascontiguousarray(x[:, :C])
        for kw in (dict(), dict(p=0.9), dict(zr=0.5, p=0.3)):
            ref = oracle.quantize_act(full, g=g, **kw)
            codes, scale = tdq.quantize_act(to_cuda(full, bf16=bf16), tdq.act_params(g=g, zr=kw.get("zr", 0.2), p=kw.get("p", 1.0)))
            compare_quantizer(si.bf16_bits_to_f32(full) if bf16 else full, g, ref, codes.cpu().numpy(), scale.cpu().numpy())


@pytest.mark.parametrize("M,C,g", [(5462, 1536, 1536), (6100, 1030, 1152), (4097, 2048, 2048), (3500, 2056, 2056), (2731, 3072, 3072), (2049, 4090, 4096), (1400, 6144, 3072)])
def test_eight_chunks_a_lane(M, C, g):
    """Long groups of bf16 in tensors of 8 M channels and more; rows off the 16-byte grid as well."""
    from paper_2604_16855_b200 import tdq
    rng = np.random.default_rng(M)
    some = _rows(rng, 97, C)
    pick = np.sort(rng.choice(M, 97, replace=False))
    for pad in (0, 1, 8):
        gen = torch.Generator("cuda").manual_seed(M)
        x = torch.randn((M, C + pad), device="cuda", generator=gen).to(torch.bfloat16)
        bits = si.f32_to_bf16_bits(some)
        x[torch.from_numpy(pick).cuda(), :C] = to_cuda(bits, bf16=True)
        for kw in (dict(), dict(p=0.9, zr=0.5), dict(tau=0.4, flags=7)):
            ref = oracle.quantize_act(bits, g=g, **kw)
            codes, scale = tdq.quantize_act(x[:, :C], tdq.act_params(g=g, tau=kw.get("tau", 1.0), zr=kw.get("zr", 0.2), p=kw.get("p", 1.0), flags=kw.get("flags", 3)))
            compare_quantizer(si.bf16_bits_to_f32(bits), g, ref, codes.cpu().numpy()[pick], scale.cpu().numpy()[pick])


@pytest.mark.parametrize("g", [32, 128, 256, 2048, 4096])
def test_dispersion_screen_on_bf16_sums(g):
    """Groups whose bf16 partial sums round one way (a dominant first term, equal terms, terms about a mean) with 7 tau sigma just
    above and below the maximum, where only the exact deviation may decide."""
    from paper_2604_16855_b200 import tdq
    rng = np.random.default_rng(300 + g)
    rows = []
    for first, rest in ((1.0, 0.06298828125), (1.0, 0.0629), (3.0, 0.19), (1.0, 0.3)):
        x = np.full(g, rest)
        x[::32] = first                                   # the first two terms of every sum of sixteen pairs
        x[1::32] = -first
        rows.append(x)
    for mean, spread in ((1.0, 1.0), (1.004, 0.97), (0.73, 0.69), (0.0, 1.0)):
        rows.append(mean + spread * np.where(np.arange(g) // 2 % 2 == 0, 1.0, -1.0))
        rows.append(mean + spread * rng.standard_normal(g))
    x = np.stack(rows).astype(np.float32)
    bits = si.f32_to_bf16_bits(x)
    v = si.bf16_bits_to_f32(bits).astype(np.float64)
    edge = np.abs(v).max(1) / (7.0 * v.std(1))             # tau at which the two bounds meet
    fill = 7 * 32 * 32 // g + 1                           # whole blocks of the kernels take part
    for e in edge:
        for off in (-0.05, -1e-3, -1e-6, 1e-6, 1e-3, 0.02, 0.04, 0.08, 0.2):
            tau = float(np.float32(e * (1.0 + off)))
            ref = oracle.quantize_act(np.tile(bits, (fill, 1)), g=g, tau=tau, flags=1)
            codes, scale = tdq.quantize_act(to_cuda(np.tile(bits, (fill, 1)), bf16=True), tdq.act_params(g=g, tau=tau, flags=1))
            compare_quantizer(si.bf16_bits_to_f32(np.tile(bits, (fill, 1))), g, ref, codes.cpu().numpy(), scale.cpu().numpy())
