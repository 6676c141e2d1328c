"""The register-resident weight quantizer at the edges of its instances, and the rows that stay with the other kernel."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from parity_utils import to_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("I,pad_to", [(8, 8), (33, 32), (255, 32), (256, 32), (257, 8), (512, 32), (520, 8), (1024, 32), (1031, 32), (2048, 128),
                                      (2049, 32), (4096, 32), (4100, 8), (8192, 32), (8193, 32), (30, 6)])
def test_rows(I, pad_to, bf16):
    from paper_2604_16855_b200 import tdq
    rng = np.random.default_rng(I)
    w = si.weights(rng, 37, I)
    w[3] = 0.0
    w[4] *= 1e-9                                        # below the step floor
    w[5] = np.round(w[5] * 200.0) / 28.0                # quotients on half-integers
    w[5, 0] = 7.0 / 4.0
    if bf16:
        w = si.bf16_bits_to_f32(si.f32_to_bf16_bits(w))
    wc, ws = tdq.quantize_weight(to_cuda(si.f32_to_bf16_bits(w), bf16=True) if bf16 else to_cuda(w), pad_to=pad_to)
    ref = oracle.quantize_weight(w, pad_to=pad_to)
    assert np.array_equal(wc.cpu().numpy(), ref["codes"]) and np.array_equal(ws.cpu().numpy(), ref["scale"])
