"""The quantizer against the oracle, bit for bit, at the edges of its launches: every group size that has a kernel of its own
(32, 64, 128, 256), groups held in a CTA's registers or read twice by a warp (neither a power of two nor a multiple of the team), matrices that end
inside a warp's share, and weights whose quotients by the scale are often exact half-integers."""
import numpy as np
import pytest
import torch

import oracle
import paper_2602_02711_b200 as dmr
from paper_2602_02711_b200 import inputs, QFormat
from helpers import to_dev_bf16

pytestmark = pytest.mark.gpu


def small_integers(N, K, seed):
    """Small integers times a power of two per block of 32: scales are short numbers, so half-integer quotients are common."""
    g = np.random.default_rng(seed)
    x = g.integers(-60, 61, size=(N, K)).astype(np.float64)
    return inputs.f64_to_bf16_bits(x * np.exp2(g.integers(-100, 100, size=(N, K // 32)).repeat(32, axis=1).astype(np.float64)))


@pytest.mark.parametrize("bits", [3, 4, 8])
@pytest.mark.parametrize("N,K,group", [
    (1, 32, 32), (3, 96, 32), (65, 1056, 32),
    (1, 64, 64), (33, 1344, 64),
    (1, 128, 128), (17, 384, 128), (131, 1152, 128),
    (1, 256, 256), (9, 768, 256),
    (5, 480, 96), (7, 1920, 384), (3, 1024, 1024),
    (2, 1056, 1056), (3, 4096, 2048), (2, 8192, 8192), (2, 8224, 8224), (5, 27648, 27648), (1, 32768, 32768), (2, 32800, 32800),
])
def test_quantize_matches_oracle(N, K, group, bits):
    for W in (inputs.weights(N, K, seed=N + K), small_integers(N, K, seed=N + K)):
        q = dmr.dmr_quantize(to_dev_bf16(W), QFormat(bits, 0 if group == K else group))
        qw, sc, zp = oracle.quantize(W, bits=bits, group=0 if group == K else group)
        assert np.array_equal(q.scales.cpu().view(torch.int16).numpy().view(np.uint16), sc)
        assert np.array_equal(q.zeros.cpu().numpy(), zp)
        assert np.array_equal(q.qweight.cpu().numpy().view(np.uint32), qw)
