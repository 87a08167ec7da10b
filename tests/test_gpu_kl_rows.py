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


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("V", [5000, 40003])
def test_masks_of_the_lowest_value_count_as_minus_infinity(V, dtype):
    """A mask may be written as -inf or as the type's lowest value: finite results, the same for both, whatever entries carry it (a thread's
    first ones, all of a thread's, all but one of a row)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(V)
    high = torch.randn((6, V), generator=g, device="cuda").mul_(2.5)
    low = high + 0.1 * torch.randn((6, V), generator=g, device="cuda")
    masked = torch.rand((6, V), generator=g, device="cuda") < 0.3
    masked[1, 16:4000] = True   # whole vectors of many threads
    masked[2] = False
    masked[2, 77] = True        # one entry
    masked[3, :V - 1] = True    # all but one
    offs = torch.tensor([0, 6], dtype=torch.int32).cuda()

    def kl(mask_high, mask_low, value):
        h = torch.where(mask_high, torch.full_like(high, value), high).to(dtype)
        l = torch.where(mask_low, torch.full_like(low, value), low).to(dtype)
        return dmr.dmr_stepwise_kl(h, l, offs)[1], h, l

    none, lowest = torch.zeros_like(masked), torch.finfo(dtype).min
    for mh, ml in ((masked, masked), (none, masked), (masked, none)):
        want, h, l = kl(mh, ml, float("-inf"))
        got = kl(mh, ml, lowest)[0]
        assert torch.isfinite(want).all() and torch.all((got - want).abs() <= 5e-6 + 1e-4 * want)  # the bound of the other KL tests
        if mh is masked:
            p, q = h.double().log_softmax(1), l.double().log_softmax(1)
            exact = torch.where(mh, 0.0, p.exp() * (p - q)).sum(1)
            assert torch.all((want - exact).abs() <= 5e-6 + 1e-4 * exact)
    everything = torch.ones_like(masked)
    for value in (float("-inf"), lowest):  # no distribution at all
        assert torch.isnan(kl(everything, none, value)[0]).all() and torch.isinf(kl(none, everything, value)[0]).all()
