"""The two-blocks-per-SM kernel of the linear layer (g = 32, 64, 128) at the edges of its tiles and of its dispatch: every number of
groups modulo a ring stage, ragged rows and columns, more tiles than blocks, each output type with and without tensor stores,
group sums, and nothing written past the last column."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from parity_utils import to_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,C,O", [(1, 32, 1), (127, 32, 64), (128, 64, 65), (129, 96, 63), (300, 128, 130), (257, 160, 4), (130, 192, 200),
                                   (200, 224, 64), (140, 256, 127), (20000, 64, 129), (6000, 288, 1028), (130, 1536, 72), (130, 1568, 72),
                                   (40, 2048, 260), (3000, 2048, 1000), (12000, 768, 60), (9000, 512, 384), (30000, 384, 64), (140, 384, 65), (260, 416, 65), (50001, 192, 63)])
@pytest.mark.parametrize("g", [32, 64, 128])
def test_shapes(M, C, O, g):
    from paper_2604_16855_b200 import tdq
    rng = np.random.default_rng(M + C + O)
    if g > 32:
        C = C // 32 * g if C <= 256 else C // g * g         # one to eight groups, and long contractions
    x = si.token_mixture(rng, 1, M, C, sigma_log_std=0.5, bg_frac=0.1, bg_nu=3.0, bg_amp=20.0).reshape(M, C)
    xa, wq = oracle.quantize_act(x, g=g), oracle.quantize_weight(si.weights(rng, O, C), pad_to=g)
    xc, xs, wc, ws = (to_cuda(v) for v in (xa["codes"], xa["scale"], wq["codes"], wq["scale"]))
    bias = torch.from_numpy(rng.standard_normal(O).astype(np.float32)).cuda()
    O4 = (O + 7) // 8 * 8
    ref = tdq.w4a4_linear(xc, xs, wc, ws, bias, g=g)
    for dt in (torch.float32, torch.bfloat16, torch.float16):
        for pitch, first in ((O4, 0), (O4 + 8, 8), (O4 + 1, 0), (O4 + 2, 2), (O4 + 3, 1)):    # aligned, even and odd
            buf = torch.full((M, pitch), 3.0, dtype=dt, device="cuda")
            ws_ = tdq.linear_workspace(M, C, O, g, "cuda")
            y = tdq.w4a4_linear(xc, xs, wc, ws, bias, g=g, y=buf[:, first:first + O], workspace=ws_)
            assert tdq.workspace_status(ws_)[0] == tdq.OK
            assert torch.equal(y, ref.to(dt))
            assert bool((buf[:, :first] == 3.0).all()) and bool((buf[:, first + O:] == 3.0).all())
    rows = np.unique(np.concatenate([np.arange(min(M, 3)), [M // 2, M - 1]]))
    want = oracle.w4a4_linear(xa["codes"][rows], xa["scale"][rows], wq["codes"], wq["scale"], bias=bias.cpu().numpy(), g=g, want_acc=True)
    K = C // g
    err = np.abs(ref.cpu().numpy()[rows].astype(np.float64) - want["y_d"])
    assert (err <= np.maximum(1e-5 * np.abs(want["y_d"]), (K + 2) * 2.0 ** -24 * want["t_abs"])).all()
    if M <= 300:
        acc = torch.zeros((M, O, K), dtype=torch.int32, device="cuda")
        tdq.w4a4_linear(xc, xs, wc, ws, g=g, y=torch.empty((M, O4), device="cuda")[:, :O], acc_debug=acc)
        assert np.array_equal(acc.cpu().numpy()[rows], want["acc"])
