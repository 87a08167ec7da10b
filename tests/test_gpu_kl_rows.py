"""Step-wise KL: a token's value must not depend on where its row lies in memory or on how many tokens share the launch, and must
match the oracle at the edges of the row's vectors and parts."""
import numpy as np
import pytest
import torch

import oracle
import paper_2602_02711_b200 as dmr
from paper_2602_02711_b200 import inputs
from helpers import to_dev_bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("T,V", [
    (3, 1), (5, 7), (4, 17), (9, 4103),              # shorter than a vector, one vector and an end, ragged vectors
    (4, 16384), (5, 16387), (3, 65535), (6, 65537),  # rows cut into parts, ragged parts
    (320, 16391),                                    # more tokens than resident CTAs
])
def test_rows_at_any_offset_match_oracle(T, V, dtype):
    high, low = inputs.logit_pair(T, V, seed=V)
    if dtype == "bf16":
        hb, lb = inputs.f64_to_bf16_bits(high), inputs.f64_to_bf16_bits(low)
        hd, ld = to_dev_bf16(hb), to_dev_bf16(lb)
    else:
        hb, lb = high.astype(np.float32), low.astype(np.float32)
        hd, ld = torch.from_numpy(hb).cuda(), torch.from_numpy(lb).cuda()
    offs = torch.tensor([0, T], dtype=torch.int32).cuda()
    _, kt = dmr.dmr_stepwise_kl(hd, ld, offs)
    n = min(T, 12)
    _, want = oracle.stepwise_kl(hb[:n], lb[:n], [0, n])
    # the bound of the other KL tests: three fp32 terms of order 10, each good to a few 1e-7
    assert np.all(np.abs(kt[:n].cpu().numpy() - want) <= 5e-6 + 1e-4 * np.abs(want))
    for i in {0, 1, T - 1}:  # alone, at the start of a buffer
        _, one = dmr.dmr_stepwise_kl(hd[i:i + 1].clone(), ld[i:i + 1].clone(), torch.tensor([0, 1], dtype=torch.int32).cuda())
        assert torch.equal(one, kt[i:i + 1])
