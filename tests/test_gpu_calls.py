"""The linears' Python calls: whatever the native marshalling does not take ends in the same errors as before, and streams, outputs and
workspaces that the caller passes are used."""
import pytest
import torch

import paper_2602_02711_b200 as dmr
from paper_2602_02711_b200 import binding, QFormat, OUT_BF16, OUT_F32
from paper_2602_02711_b200.binding import OP_DENSE, OP_LOWBIT, OP_ROUTED

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("native", [True, False])
@pytest.mark.parametrize("M", [0, 1, 40])
@pytest.mark.parametrize("out", [OUT_BF16, OUT_F32])
def test_given_outputs_workspaces_and_streams(M, out, native, monkeypatch):
    dmr.lib()
    if not native:
        monkeypatch.setattr(binding, "_calls", None)
    N, K = 200, 256
    X, W = torch.randn(M, K, device="cuda").bfloat16(), torch.randn(N, K, device="cuda").bfloat16()
    q, mask = dmr.dmr_quantize(W, QFormat(4, 64)), torch.ones(M, dtype=torch.uint8, device="cuda")
    dtype = torch.float32 if out == OUT_F32 else torch.bfloat16
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    for op, call in ((OP_LOWBIT, lambda **k: dmr.dmr_lowbit_linear(X, q, out, **k)), (OP_DENSE, lambda **k: dmr.dmr_dense_linear(X, W, out, **k)),
                     (OP_ROUTED, lambda **k: dmr.dmr_routed_linear(X, mask, W, q, out, **k))):
        want = call()
        for kw in ({}, {"stream": s}):
            Y, ws = torch.full((M, N), 7, dtype=dtype, device="cuda"), dmr.new_workspace(op, M, N, K, q.fmt)
            torch.cuda.synchronize()
            assert call(Y=Y, workspace=ws, **kw) is Y
            torch.cuda.synchronize()
            assert torch.equal(Y, want)


def test_refused_arguments_raise():
    N, K, M = 128, 128, 4
    X, W = torch.zeros(M, K, device="cuda", dtype=torch.bfloat16), torch.zeros(N, K, device="cuda", dtype=torch.bfloat16)
    q, Y = dmr.dmr_quantize(W, QFormat(4, 64)), torch.zeros(M, N, device="cuda", dtype=torch.bfloat16)
    mask, ws = torch.zeros(M, dtype=torch.uint8, device="cuda"), dmr.new_workspace(OP_ROUTED, M, N, K, q.fmt)
    for bad in (X.float(), X.cpu(), torch.zeros(K, M, device="cuda", dtype=torch.bfloat16).T, X[:, :64].contiguous()):
        for call in (lambda: dmr.dmr_lowbit_linear(bad, q, Y=Y, workspace=ws), lambda: dmr.dmr_dense_linear(bad, W, Y=Y, workspace=ws),
                     lambda: dmr.dmr_routed_linear(bad, mask, W, q, Y=Y, workspace=ws)):
            with pytest.raises(dmr.DmrError) as e:
                call()
            assert e.value.code == 1
    with pytest.raises(dmr.DmrError) as e:
        dmr.dmr_lowbit_linear(X, q, Y=Y, workspace=torch.zeros(16, dtype=torch.uint8, device="cuda"))
    assert e.value.code == 4
    with pytest.raises(dmr.DmrError) as e:
        dmr.dmr_dense_linear(X, W, OUT_F32, Y=Y, workspace=ws)
    assert e.value.code == 1
    with pytest.raises(dmr.DmrError) as e:
        dmr.dmr_routed_linear(X, mask[:3], W, q, Y=Y, workspace=ws)
    assert e.value.code == 1
