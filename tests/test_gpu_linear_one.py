"""The cluster kernel of the linear layer (groups wider than 32, power-of-two steps) at the edges of its 256 x 256 tiles: odd
numbers of 128-row and 128-column blocks, ragged edges, more tiles than clusters, short and long contractions, every type."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from parity_utils import to_cuda

pytestmark = pytest.mark.gpu


def _check(M, C, O, g, pow2):
    from paper_2604_16855_b200 import tdq
    rng = np.random.default_rng(M + C + O)
    rows = np.unique(np.concatenate([np.arange(min(M, 130)), np.arange(max(M - 3, 0), M), rng.integers(0, M, 20)]))
    x = torch.randn((M, C), device="cuda", generator=torch.Generator("cuda").manual_seed(M)) * 2.0
    w = torch.from_numpy(si.weights(rng, O, C)).cuda()
    bias = torch.from_numpy(rng.standard_normal(O).astype(np.float32)).cuda()
    xc, xs = tdq.quantize_act(x, tdq.act_params(g=g, flags=7 if pow2 else 3))
    wc, ws = tdq.quantize_weight(w, pad_to=g)
    want = oracle.w4a4_linear(xc.cpu().numpy()[rows], xs.cpu().numpy()[rows], wc.cpu().numpy(), ws.cpu().numpy(),
                              bias=bias.cpu().numpy(), g=g)
    wsp = tdq.linear_workspace(M, C, O, g, "cuda")
    fn = tdq.w4a4_linear_pow2 if pow2 else tdq.w4a4_linear
    ref = None
    for dt in (torch.float32, torch.bfloat16, torch.float16):
        buf = torch.full((M, O + 8), 3.0, dtype=dt, device="cuda")
        y = fn(xc, xs, wc, ws, bias, g=g, y=buf[:, :O], workspace=wsp)
        assert tdq.workspace_status(wsp) == (tdq.OK, 0)
        assert bool((buf[:, O:] == 3.0).all())
        if dt == torch.float32:
            ref = y.clone()
            terms = C if pow2 else C // g                    # rounded additions per output
            err = np.abs(ref.cpu().numpy()[rows].astype(np.float64) - want["y_d"])
            t = want["t_abs"] + np.abs(bias.cpu().numpy())[None, :]
            assert (err <= np.maximum(1e-5 * np.abs(want["y_d"]), (terms + 2) * 2.0 ** -24 * t)).all()
        else:
            assert torch.equal(y, ref.to(dt))


@pytest.mark.parametrize("M,C,O", [(9473, 32, 8), (9600, 64, 264), (9300, 96, 264), (1025, 160, 2100), (9473, 224, 256), (2700, 256, 1032),
                                   (129, 384, 9480), (20000, 768, 1096), (4100, 4096, 2056), (40000, 128, 512), (3000, 1056, 776),
                                   (300, 512, 256)])
def test_one_group(M, C, O):
    _check(M, C, O, C, False)
    _check(M, C, O, 32, True)


@pytest.mark.parametrize("M,C,O,g", [(9473, 128, 8, 64), (1025, 320, 2100, 64), (20000, 768, 1096, 64), (20000, 768, 1096, 128),
                                     (9300, 288, 264, 96), (2700, 768, 1032, 256), (129, 640, 9480, 128), (4100, 4096, 2056, 128),
                                     (4100, 4096, 1032, 1024), (3000, 480, 1032, 160)])
def test_several_groups(M, C, O, g):
    _check(M, C, O, g, False)


@pytest.mark.parametrize("C,g,pow2", [(32, 32, True), (64, 64, False), (96, 96, False), (96, 32, True), (256, 256, False), (64, 32, False)])
def test_one_row_of_any_pitch(C, g, pow2):
    """A y of one row may come with a pitch (2^40 bytes and more) that no tensor map holds: the same numbers, by a kernel that
    writes without one.  (The contractions of fewer than 128 channels went to the cluster kernel with an empty map.)"""
    from paper_2604_16855_b200 import tdq
    O = 16384
    rng = np.random.default_rng(C)
    x = torch.from_numpy(rng.standard_normal((1, C)).astype(np.float32)).cuda()
    xc, xs = tdq.quantize_act(x, tdq.act_params(g=g, flags=7 if pow2 else 3))
    wc, ws = tdq.quantize_weight(torch.from_numpy(si.weights(rng, O, C)).cuda(), pad_to=g)
    fn = tdq.w4a4_linear_pow2 if pow2 else tdq.w4a4_linear
    wsp = tdq.linear_workspace(1, C, O, g, "cuda")
    terms = C if pow2 else C // g                            # rounded additions per output
    want = oracle.w4a4_linear(xc.cpu().numpy(), xs.cpu().numpy(), wc.cpu().numpy(), ws.cpu().numpy(), g=g)
    for dt in (torch.float32, torch.bfloat16):
        for pitch in (O, 1 << 40, 1 << 61):
            buf = torch.full((O + 8,), 3.0, dtype=dt, device="cuda")
            y = fn(xc, xs, wc, ws, g=g, y=buf[:O].as_strided((1, O), (pitch, 1)), workspace=wsp)
            assert y.stride(0) == pitch and tdq.workspace_status(wsp) == (tdq.OK, 0)
            assert bool((buf[O:] == 3.0).all())
            err = np.abs(buf[:O].float().cpu().numpy()[None].astype(np.float64) - want["y_d"])
            half_ulp = 0.0 if dt == torch.float32 else 2.0 ** -8 * np.abs(want["y_d"])
            assert (err <= np.maximum(1e-5 * np.abs(want["y_d"]), (terms + 2) * 2.0 ** -24 * want["t_abs"]) + half_ulp).all()
