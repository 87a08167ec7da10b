"""Batches of up to 64 rows (and of up to 128 on narrow layers with 4- and 8-bit codes) against the oracle at the edges of the kernel that
multiplies exact integers: row counts around its three row tiles, feature counts below, at and beyond one 128-feature tile and not multiples
of four, half a unit of inputs, one unit, and more units than CTAs, groups of half a unit, one, several and the whole row; routed rows bit
for bit against the unrouted calls; and repeated calls of several layers on one stream."""
import numpy as np
import pytest
import torch

import oracle
import paper_2602_02711_b200 as dmr
from paper_2602_02711_b200 import inputs, QFormat, OUT_BF16, OUT_F32
from paper_2602_02711_b200.binding import OP_DENSE, OP_LOWBIT, OP_ROUTED
from helpers import to_dev_bf16, rel_err

pytestmark = pytest.mark.gpu

TOL = 5e-5  # exact products (integers times bf16, scaled in fp32), fp32 sums of up to 5120 terms

SHAPES = [(1, 128, 128), (3, 100, 64), (16, 129, 192), (17, 257, 384), (32, 130, 576), (33, 640, 512), (63, 1024, 2048), (64, 2304, 1088)]


@pytest.mark.parametrize("M,N,K", SHAPES)
def test_dense(M, N, K):
    W, X = inputs.weights(N, K, seed=M), inputs.activations(M, K, seed=M)
    Y = dmr.dmr_dense_linear(to_dev_bf16(X), to_dev_bf16(W), OUT_F32)
    assert rel_err(Y.cpu().numpy().astype(np.float64), oracle.dense_linear(X, W)) <= TOL
    assert torch.equal(dmr.dmr_dense_linear(to_dev_bf16(X), to_dev_bf16(W), OUT_BF16), Y.to(torch.bfloat16))


@pytest.mark.parametrize("bits", [3, 4, 8])
@pytest.mark.parametrize("M,N,K,group", [s + (g,) for s in SHAPES for g in (64, 0)] + [(20, 700, 1024, 128), (64, 129, 1536, 256), (33, 128, 768, 384),
                                                                                        (65, 1024, 512, 128), (128, 1920, 384, 64), (100, 250, 576, 192),
                                                                                        (33, 1024, 960, 320), (64, 100, 960, 192), (128, 1920, 2880, 576)])
def test_low_bit(M, N, K, bits, group):
    if bits == 3 and (M > 64 or K % 128 != 0):
        pytest.skip("the SM-pair kernel (test_gpu_pair.py), or up to 32 rows the one for any shape (test_gpu_w3.py)")
    W, X = inputs.weights(N, K, seed=K), inputs.activations(M, K, seed=N, outlier_frac=0.01)
    assert M <= 16 or dmr.dmr_describe_dispatch(OP_LOWBIT, M, N, K, QFormat(bits, group))["kernel"] == "small"
    q = dmr.dmr_quantize(to_dev_bf16(W), QFormat(bits, group))
    want = oracle.lowbit_linear(X, *oracle.quantize(W, bits=bits, group=group), bits=bits, group=group)
    Y = dmr.dmr_lowbit_linear(to_dev_bf16(X), q, OUT_F32)
    assert rel_err(Y.cpu().numpy().astype(np.float64), want) <= TOL
    assert torch.equal(dmr.dmr_lowbit_linear(to_dev_bf16(X), q, OUT_BF16), Y.to(torch.bfloat16))


@pytest.mark.parametrize("bits,group,K", [(4, 128, 1024), (4, 64, 1024), (8, 0, 1024), (3, 128, 1024), (4, 320, 960)])
@pytest.mark.parametrize("M,high,N", [(2, 1, 700), (16, 5, 128), (17, 0, 700), (40, 40, 130), (64, 63, 700), (64, 20, 2304), (100, 30, 700)])
def test_routed_rows_equal_unrouted_ones(M, high, N, bits, group, K):
    W, X = to_dev_bf16(inputs.weights(N, K, seed=1)), to_dev_bf16(inputs.activations(M, K, seed=2))
    q = dmr.dmr_quantize(W, QFormat(bits, group))
    mask = np.zeros(M, dtype=np.uint8)
    mask[np.random.default_rng(M).permutation(M)[:high]] = 1
    md = torch.from_numpy(mask).cuda()
    ws = dmr.new_workspace(OP_ROUTED, M, N, K, q.fmt)
    Y = dmr.dmr_routed_linear(X, md, W, q, OUT_F32, workspace=ws)
    want = torch.where(md[:, None] != 0, dmr.dmr_dense_linear(X, W, OUT_F32), dmr.dmr_lowbit_linear(X, q, OUT_F32))
    assert torch.equal(Y, want)
    assert int(ws[:4].view(torch.int32).item()) == 0


@pytest.mark.parametrize("M,N,K", [(65, 257, 320), (100, 2000, 512), (128, 1930, 1024)])
def test_rows_between_the_small_and_the_large_batches(M, N, K):
    W, X = inputs.weights(N, K, seed=M), inputs.activations(M, K, seed=M)
    Y = dmr.dmr_dense_linear(to_dev_bf16(X), to_dev_bf16(W), OUT_F32)
    assert rel_err(Y.cpu().numpy().astype(np.float64), oracle.dense_linear(X, W)) <= TOL
    for bits in (3, 4, 8) if N > 1920 else ():
        q = dmr.dmr_quantize(to_dev_bf16(W), QFormat(bits, 128))
        want = oracle.lowbit_linear(X, *oracle.quantize(W, bits=bits, group=128), bits=bits, group=128)
        Y = dmr.dmr_lowbit_linear(to_dev_bf16(X), q, OUT_F32)
        # weights rounded to fp16: 2^-11 / sqrt(3) in the root mean square, independent errors
        assert np.linalg.norm(Y.cpu().numpy() - want) <= 2.0 ** -11 / 3 ** 0.5 * np.linalg.norm(want)


@pytest.mark.parametrize("bits,M", [(0, 5), (0, 64), (4, 30), (8, 13), (8, 128)])
def test_calls_one_after_the_other(bits, M):
    """Each launch starts before the one ahead of it has ended: outputs, partial sums and counters must not meet."""
    layers = []
    for N, K in [(1024, 5120), (5120, 1024), (1024, 5120)]:
        W, X = to_dev_bf16(inputs.weights(N, K, seed=N)), to_dev_bf16(inputs.activations(M, K, seed=K))
        q = dmr.dmr_quantize(W, QFormat(bits, 0)) if bits else None
        ws = dmr.new_workspace(OP_LOWBIT if bits else OP_DENSE, M, N, K, QFormat(bits or 4, 0))
        layers.append(lambda X=X, W=W, q=q, ws=ws: dmr.dmr_lowbit_linear(X, q, OUT_F32, workspace=ws) if q else dmr.dmr_dense_linear(X, W, OUT_F32, workspace=ws))
    first = []
    for f in layers:
        first.append(f())
        torch.cuda.synchronize()
    for _ in range(20):
        again = [f() for f in layers for _ in range(2)]
        assert all(torch.equal(y, first[i // 2]) for i, y in enumerate(again))


def test_one_workspace_for_calls_of_all_kernels():
    """Zeroed once, a workspace serves calls of any sizes in any order: one kernel's partial sums and gathered rows must not lie on the
    counters that another one expects to be zero."""
    def case(op, M, N, K, bits=0, group=0):
        W, X = to_dev_bf16(inputs.weights(N, K, seed=N)), to_dev_bf16(inputs.activations(M, K, seed=K))
        q = dmr.dmr_quantize(W, QFormat(bits, group)) if bits else None
        mask = torch.from_numpy(inputs.precision_mask(M, 0.4, seed=M)).cuda()
        call = {OP_DENSE: lambda **k: dmr.dmr_dense_linear(X, W, OUT_F32, **k), OP_LOWBIT: lambda **k: dmr.dmr_lowbit_linear(X, q, OUT_F32, **k),
                OP_ROUTED: lambda **k: dmr.dmr_routed_linear(X, mask, W, q, OUT_F32, **k)}[op]
        return call, dmr.dmr_workspace_bytes(op, M, N, K, QFormat(bits or 4, group))

    cases = [case(OP_DENSE, 64, 4096, 4096),            # partial sums of 148 shares
             case(OP_DENSE, 16, 2304, 8200),            # streaming kernel, feature groups shared by CTAs
             case(OP_LOWBIT, 300, 4096, 11008, 4, 128),  # prepared activations, split along k
             case(OP_LOWBIT, 8, 4096, 8256, 8, 192),    # streaming kernel
             case(OP_ROUTED, 64, 1024, 5120, 4, 128),
             case(OP_ROUTED, 20, 2304, 8256, 8, 192),   # streaming kernel, low half
             case(OP_ROUTED, 20, 2304, 8224, 4, 32),    # streaming kernel, high half
             case(OP_LOWBIT, 13, 4096, 4096, 8, 0)]
    want = [call() for call, _ in cases]
    ws = torch.zeros(max(n for _, n in cases), dtype=torch.uint8, device="cuda")
    for _ in range(3):
        for order in (range(len(cases)), reversed(range(len(cases)))):
            for i in order:
                assert torch.equal(cases[i][0](workspace=ws), want[i])
    assert int(ws[:4].view(torch.int32).item()) == 0


@pytest.mark.parametrize("M", [33, 48, 64])
def test_weights_written_by_the_call_before(M):
    """From 33 rows on a call's weights may be another call's output, which the kernel before still writes when this one's starts (it takes eight
    of the SMs, so this one finds free ones at once)."""
    A, B = to_dev_bf16(inputs.activations(64, 1024, seed=1)), to_dev_bf16(inputs.weights(1024, 1024, seed=2))
    X = to_dev_bf16(inputs.activations(M, 1024, seed=3))
    W = dmr.dmr_dense_linear(A, B)
    torch.cuda.synchronize()
    want = dmr.dmr_dense_linear(X, W, OUT_F32)
    ws = [dmr.new_workspace(OP_DENSE, 64, 1024, 1024, QFormat(4, 0)) for _ in range(2)]
    Y = torch.empty_like(want)
    for _ in range(20):
        W.zero_()
        torch.cuda.synchronize()
        dmr.dmr_dense_linear(A, B, Y=W, workspace=ws[0])
        dmr.dmr_dense_linear(X, W, OUT_F32, Y=Y, workspace=ws[1])
        assert torch.equal(Y, want)


@pytest.mark.parametrize("bits,group", [(4, 128), (4, 64), (8, 320), (8, 0)])
@pytest.mark.parametrize("M,N", [(40, 2000), (65, 300), (128, 2000), (300, 130)])
def test_rows_longer_than_the_large_batches_take(M, N, bits, group):
    """More than 32768 inputs: exact for any number of rows, in launches of 128; routed rows are the unrouted ones whichever launch they fall into."""
    K = 40960
    assert dmr.dmr_describe_dispatch(OP_LOWBIT, M, N, K, QFormat(bits, group))["kernel"] == "small"
    W, X = inputs.weights(N, K, seed=N), inputs.activations(M, K, seed=M, outlier_frac=0.01)
    q, Xd, Wd = dmr.dmr_quantize(to_dev_bf16(W), QFormat(bits, group)), to_dev_bf16(X), to_dev_bf16(W)
    Y = dmr.dmr_lowbit_linear(Xd, q, OUT_F32)
    want = Xd.double() @ dmr.dmr_dequantize(q).double().T
    assert float((Y.double() - want).abs().max() / want.abs().max()) <= TOL
    mask = torch.from_numpy(inputs.precision_mask(M, 0.4, seed=M)).cuda()
    Yr = dmr.dmr_routed_linear(Xd, mask, Wd, q, OUT_F32)
    assert torch.equal(Yr, torch.where(mask[:, None] != 0, dmr.dmr_dense_linear(Xd, Wd, OUT_F32), Y))
