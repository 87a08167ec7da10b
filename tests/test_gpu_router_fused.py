"""The one-launch router forward at the edges of its splits, against the float64 oracle: every head width it has an instance for,
widths that leave some of the sixteen CTAs of a cluster without features, one layer (the last layer is also the first), more tokens
than a cluster takes at a time, more sequences than clusters, and a repeated call on the same workspace."""
import numpy as np
import pytest
import torch

import oracle
import paper_2602_02711_b200 as dmr
from paper_2602_02711_b200 import inputs, RouterCfg

pytestmark = pytest.mark.gpu

TOL = 2e-5  # the bar of the other router tests: fp32 sums renormalised by every layer norm


@pytest.mark.parametrize("cfg_kw,B,L", [
    (dict(d=16, heads=1, ffn=16, layers=1, l_max=4, classes=2), 1, 1),
    (dict(d=48, heads=3, ffn=80, layers=1, l_max=8, classes=2), 3, 8),
    (dict(d=96, heads=3, ffn=208, layers=2, l_max=40, classes=5), 2, 37),
    (dict(d=256, heads=2, ffn=512, layers=2, l_max=128, classes=3), 2, 127),   # head width 128, keys in several steps
    (dict(d=384, heads=6, ffn=1536, layers=2, l_max=32, classes=2), 33, 32),   # several token blocks per cluster
    (dict(d=64, heads=4, ffn=128, layers=3, l_max=4, classes=2), 1000, 4),     # 143 sequences per cluster in the last layer
    (dict(d=48, heads=2, ffn=80, layers=2, l_max=8, classes=2), 3, 8),         # head width 24: layer by layer
])
def test_router_matches_oracle(cfg_kw, B, L):
    cfg = RouterCfg(**cfg_kw)
    p = inputs.router_params(**cfg_kw, seed=B)
    Z, n = inputs.router_embeddings(B, L, cfg_kw["d"], seed=L), inputs.router_lengths(B, L, seed=L)
    want = oracle.router_forward(Z, n, p, cfg_kw["heads"])
    params, Zd, nd = dmr.pack_router_params(p, cfg), torch.from_numpy(Z).cuda(), torch.from_numpy(n).cuda()
    ws = torch.full((dmr.lib().dmr_router_workspace_bytes(cfg, B, L),), 255, dtype=torch.uint8, device="cuda")  # NaN: nothing is assumed
    first, _ = dmr.dmr_router_forward(params, cfg, Zd, nd, score_class=1, workspace=ws)
    again, scores = dmr.dmr_router_forward(params, cfg, Zd, nd, score_class=1, workspace=ws)
    assert np.abs(first.cpu().numpy() - want).max() <= TOL
    assert torch.equal(first, again) and torch.equal(scores, again[:, 1].contiguous())


def test_inside_a_graph():
    kw = dict(d=384, heads=6, ffn=1536, layers=2, l_max=16, classes=2)
    cfg = RouterCfg(**kw)
    params = dmr.pack_router_params(inputs.router_params(**kw, seed=1), cfg)
    Z, n = torch.from_numpy(inputs.router_embeddings(5, 16, 384, seed=1)).cuda(), torch.from_numpy(inputs.router_lengths(5, 16, seed=1)).cuda()
    ws = torch.empty(dmr.lib().dmr_router_workspace_bytes(cfg, 5, 16), dtype=torch.uint8, device="cuda")
    want, _ = dmr.dmr_router_forward(params, cfg, Z, n, workspace=ws)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        got, _ = dmr.dmr_router_forward(params, cfg, Z, n, workspace=ws)
    for _ in range(3):
        got.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(got, want)


@pytest.mark.parametrize("ffn", [16, 80, 208, 400])
def test_features_that_some_ctas_have_none_of_after_a_kernel_that_left_nans(ffn):
    """Some of the sixteen CTAs of a cluster have no hidden features at these widths.  What the kernel before left in shared memory - here NaN
    in every word - must not reach the probabilities."""
    kw = dict(d=64, heads=4, ffn=ffn, layers=2, l_max=16, classes=2)
    cfg = RouterCfg(**kw)
    p = inputs.router_params(**kw, seed=3)
    Z, n = inputs.router_embeddings(20, 16, 64, seed=3), inputs.router_lengths(20, 16, seed=3)
    params, Zd, nd = dmr.pack_router_params(p, cfg), torch.from_numpy(Z).cuda(), torch.from_numpy(n).cuda()
    X, W = torch.full((16, 4096), float("nan"), device="cuda").bfloat16(), torch.full((4096, 4096), float("nan"), device="cuda").bfloat16()
    want = oracle.router_forward(Z, n, p, 4)
    for _ in range(5):
        dmr.dmr_dense_linear(X, W)
        got, _ = dmr.dmr_router_forward(params, cfg, Zd, nd)
        assert np.abs(got.cpu().numpy() - want).max() <= TOL


@pytest.mark.parametrize("cfg_kw,B,L,ways", [
    (dict(d=96, heads=6, ffn=96, layers=12, l_max=64, classes=2), 8, 32, 1),     # few tokens: one launch
    (dict(d=96, heads=6, ffn=96, layers=12, l_max=64, classes=2), 8, 64, 0),     # layer by layer
    (dict(d=256, heads=4, ffn=1024, layers=6, l_max=64, classes=2), 16, 64, 2),  # one launch or layer by layer, as the lengths are
    (dict(d=64, heads=4, ffn=128, layers=2, l_max=64, classes=3), 16, 64, 0),
    (dict(d=384, heads=6, ffn=1536, layers=8, l_max=64, classes=2), 24, 64, 2),
])
def test_choice_between_one_launch_and_layer_by_layer(cfg_kw, B, L, ways):
    """Both ways of a call whose lengths decide between them, in turn on one workspace; which kernels are enqueued depends on the sizes only."""
    cfg = RouterCfg(**cfg_kw)
    p = inputs.router_params(**cfg_kw, seed=B)
    Z = inputs.router_embeddings(B, L, cfg_kw["d"], seed=L)
    params, Zd = dmr.pack_router_params(p, cfg), torch.from_numpy(Z).cuda()
    ws = torch.full((dmr.lib().dmr_router_workspace_bytes(cfg, B, L),), 255, dtype=torch.uint8, device="cuda")
    layered = 2 + 7 * cfg_kw["layers"]
    for n in (np.full(B, L, np.int32), inputs.router_lengths(B, L, seed=L), np.ones(B, np.int32), np.full(B, L, np.int32)):
        before = dmr.dmr_launch_count()
        got, _ = dmr.dmr_router_forward(params, cfg, Zd, torch.from_numpy(n).cuda(), workspace=ws)
        assert dmr.dmr_launch_count() - before == (layered, 1, layered + 1)[ways]
        few = slice(0, B, max(1, B // 8))  # (sequences do not depend on one another)
        assert np.abs(got.cpu().numpy()[few] - oracle.router_forward(Z[few], n[few], p, cfg_kw["heads"])).max() <= TOL
