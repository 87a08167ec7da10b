"""Batches of more than 128 rows (the SM-pair kernel) against the oracle at the edges of its tiles: row counts around 128, 256 and
multiples of 16, feature counts below, at and beyond one 256-feature tile, one k block and an odd number of them, a split along k,
3-bit rows that are and are not whole boxes (from 33 rows on); and routed rows bit for bit against the unrouted calls."""
import numpy as np
import pytest
import torch

import oracle
import paper_2602_02711_b200 as dmr
from paper_2602_02711_b200 import inputs, QFormat, OUT_BF16, OUT_F32
from paper_2602_02711_b200.binding import OP_LOWBIT
from helpers import to_dev_bf16, rel_err

pytestmark = pytest.mark.gpu

TOL_DENSE = 5e-5  # exact bf16 products, fp32 sums of up to 4096 terms
# One rounding of every dequantized weight to fp16: a relative error of at most 2^-11, evenly spread, so of 2^-11 / sqrt(3) in the root
# mean square.  The errors of an output's terms are independent, so that is the bound of the relative 2-norm error of all outputs.
TOL_LOW = 2.0 ** -11 / 3 ** 0.5

SHAPES = [(129, 256, 64), (144, 100, 192), (256, 257, 128), (257, 512, 320), (300, 640, 2048), (401, 384, 256), (520, 250, 128)]


@pytest.mark.parametrize("M,N,K", SHAPES)
def test_dense(M, N, K):
    W, X = inputs.weights(N, K, seed=M), inputs.activations(M, K, seed=M)
    want = oracle.dense_linear(X, W)
    Y = dmr.dmr_dense_linear(to_dev_bf16(X), to_dev_bf16(W), OUT_F32)
    assert rel_err(Y.cpu().numpy().astype(np.float64), want) <= TOL_DENSE
    assert torch.equal(dmr.dmr_dense_linear(to_dev_bf16(X), to_dev_bf16(W), OUT_BF16), Y.to(torch.bfloat16))


@pytest.mark.parametrize("bits,group", [(4, 64), (8, 0), (3, 64)])
@pytest.mark.parametrize("M,N,K", SHAPES)
def test_low_bit(M, N, K, bits, group):
    assert dmr.dmr_describe_dispatch(OP_LOWBIT, M, N, K, QFormat(bits, group))["kernel"] == "pair"
    W, X = inputs.weights(N, K, seed=K), inputs.activations(M, K, seed=N, outlier_frac=0.01)
    q = dmr.dmr_quantize(to_dev_bf16(W), QFormat(bits, group))
    want = oracle.lowbit_linear(X, *oracle.quantize(W, bits=bits, group=group), bits=bits, group=group)
    Y = dmr.dmr_lowbit_linear(to_dev_bf16(X), q, OUT_F32)
    assert np.linalg.norm(Y.cpu().numpy() - want) <= TOL_LOW * np.linalg.norm(want)
    assert torch.equal(dmr.dmr_lowbit_linear(to_dev_bf16(X), q, OUT_BF16), Y.to(torch.bfloat16))


# rows of an odd number of k blocks: one tile, both feature tiles ragged, a split along k whose parts are odd, several tiles per pair, groups of one
# to all k blocks, the fewest rows
@pytest.mark.parametrize("M,N,K,group", [(129, 256, 64, 64), (33, 100, 192, 64), (64, 300, 2880, 320), (65, 257, 2880, 0), (300, 640, 4544, 64), (1100, 2600, 960, 192)])
def test_3_bit_rows_that_are_not_whole_boxes(M, N, K, group):
    assert dmr.dmr_describe_dispatch(OP_LOWBIT, M, N, K, QFormat(3, group))["kernel"] == "pair"
    W, X = inputs.weights(N, K, seed=K), inputs.activations(M, K, seed=N, outlier_frac=0.01)
    q = dmr.dmr_quantize(to_dev_bf16(W), QFormat(3, group))
    want = oracle.lowbit_linear(X, *oracle.quantize(W, bits=3, group=group), bits=3, group=group)
    Y = dmr.dmr_lowbit_linear(to_dev_bf16(X), q, OUT_F32)
    assert np.linalg.norm(Y.cpu().numpy() - want) <= TOL_LOW * np.linalg.norm(want)
    assert torch.equal(dmr.dmr_lowbit_linear(to_dev_bf16(X), q, OUT_BF16), Y.to(torch.bfloat16))


@pytest.mark.parametrize("bits,group,K", [(4, 128, 1024), (8, 0, 1024), (3, 128, 1024), (3, 64, 960)])
@pytest.mark.parametrize("M,high", [(200, 60), (300, 0), (300, 300), (513, 1)])
def test_routed_rows_equal_unrouted_ones(M, high, bits, group, K):
    N = 700
    W, X = to_dev_bf16(inputs.weights(N, K, seed=1)), to_dev_bf16(inputs.activations(M, K, seed=2))
    q = dmr.dmr_quantize(W, QFormat(bits, group))
    mask = np.zeros(M, dtype=np.uint8)
    mask[np.random.default_rng(M).permutation(M)[:high]] = 1
    md = torch.from_numpy(mask).cuda()
    Y = dmr.dmr_routed_linear(X, md, W, q, OUT_F32)
    want = torch.where(md[:, None] != 0, dmr.dmr_dense_linear(X, W, OUT_F32), dmr.dmr_lowbit_linear(X, q, OUT_F32))
    assert torch.equal(Y, want)
