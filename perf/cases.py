"""Performance cases: the work a user of this library has it do, through its public entry points.

A serving program keeps the quantized (and, for routed steps, the bf16) weights of its decoder layers, one output buffer and one
workspace per linear, and calls the linears of a layer one after the other.  Offline it quantizes layers, scores action tokens
with the step-wise KL divergence, and online the router decides the precision of every step.  The layer shapes are the ones
`paper_2602_02711_b200.inputs` lists; tensors are drawn on the GPU from the seed with the distributions that module documents.

Interface: listed() -> cases, draw(rng) -> one more case, prepare(case, seed) -> state, run(state) -> outputs, work(case) and
tolerance(case).  A case is a dict of plain values; its "kind" says which of the paths below it takes.
"""
import math

import numpy as np
import torch

import paper_2602_02711_b200 as dmr
from paper_2602_02711_b200 import inputs
from paper_2602_02711_b200.binding import OP_DENSE, OP_LOWBIT, OP_ROUTED

LAYERS = {"7b": inputs.LAYER_7B, "14b": inputs.LAYER_14B, "32b": inputs.LAYER_32B}
BITS = {"w3": 3, "w4": 4, "w8": 8}
VOCAB = 151936           # the vocabulary of the logits the KL signal is formed from
OUTLIER_FRACTION = 0.01  # share of activation channels with outliers (x 20)
MAX_PRODUCT = 4096 * sum(n * k for n, k in inputs.LAYER_7B.values())  # rows x weights of the largest listed case


def listed():
    return [
        # One agent decoding one token on the low-precision model: the smallest layer call, weights read once for one row.
        {"name": "decode_w4_m1", "kind": "linear", "layer": "7b", "weights": "w4", "group": 128, "M": 1, "outliers": False},
        # Sixteen concurrent agents decoding together: the largest batch of the decode sweep.
        {"name": "decode_w4_m16", "kind": "linear", "layer": "7b", "weights": "w4", "group": 128, "M": 16, "outliers": False},
        # The most aggressive precision of the paper (W3A16, group 128) with a handful of agents.
        {"name": "decode_w3_m5", "kind": "linear", "layer": "7b", "weights": "w3", "group": 128, "M": 5, "outliers": False},
        # INT8 per-channel weights, wide layer, outlier activation channels, an odd batch between the decode tiles.
        {"name": "decode_w8_m13", "kind": "linear", "layer": "32b", "weights": "w8", "group": 0, "M": 13, "outliers": True},
        # Steps that the router sent to the high-precision model: the same layer with bf16 weights.
        {"name": "decode_bf16_m3", "kind": "linear", "layer": "7b", "weights": "bf16", "group": 0, "M": 3, "outliers": False},
        # A short prompt (or many agents at once) on the wide layer, group 64, ragged rows: between decode and prefill.
        {"name": "prefill_w4_g64_m201", "kind": "linear", "layer": "32b", "weights": "w4", "group": 64, "M": 201, "outliers": True},
        # A long prompt through the low-precision model: the largest case, bound by the tensor cores.
        {"name": "prefill_w4_m4096", "kind": "linear", "layer": "7b", "weights": "w4", "group": 128, "M": 4096, "outliers": False},
        # A prompt of ordinary, odd length through the high-precision model.
        {"name": "prefill_bf16_m1501", "kind": "linear", "layer": "7b", "weights": "bf16", "group": 0, "M": 1501, "outliers": False},
        # One decoding step of 64 concurrent agents, each on the precision its router chose (30 % high).
        {"name": "routed_w4_m64", "kind": "routed", "layer": "14b", "weights": "w4", "group": 128, "M": 64, "p_high": 0.3},
        # Making the low-precision copy of one layer.
        {"name": "quantize_w4", "kind": "quantize", "layer": "7b", "weights": "w4", "group": 128},
        # The router's training signal for a batch of action tokens.
        {"name": "kl_t777", "kind": "kl", "T": 777, "V": VOCAB, "dtype": "bf16"},
        # One agent asks the router for the precision of its next step: many small dependent launches.
        {"name": "router_b1", "kind": "router", "B": 1, "L": 32, "l_max": 32, "d": 384, "heads": 6, "ffn": 1536, "layers": 8, "rho": 0.4},
    ]


def _log_int(rng, lo, hi):
    """An integer of [lo, hi], spread evenly over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.99)))))))


def _weights(layer):
    return sum(n * k for n, k in LAYERS[layer].values())


def draw(rng):
    kind = rng.choice(["linear"] * 6 + ["routed", "quantize", "kl", "router"])
    if kind == "linear":
        layer = rng.choice(["7b", "14b", "32b"])
        weights, group = rng.choice([("w4", 128), ("w4", 128), ("w4", 64), ("w3", 128), ("w8", 0), ("bf16", 0)])
        # decode batches and prompts are equally common; the slower formats stop at half of the largest product
        most = MAX_PRODUCT // _weights(layer) // (1 if weights in ("w4", "bf16") else 2)
        M = _log_int(rng, 1, 32) if rng.random() < 0.5 else _log_int(rng, 33, most)
        return {"kind": kind, "layer": layer, "weights": weights, "group": group, "M": M, "outliers": rng.random() < 0.3}
    if kind == "routed":
        weights, group = rng.choice([("w4", 128), ("w4", 128), ("w8", 0), ("w3", 128)])
        return {"kind": kind, "layer": rng.choice(["7b", "14b"]), "weights": weights, "group": group, "M": _log_int(rng, 2, 256),
                "p_high": rng.choice([0.2, 0.3, 0.4, 0.7])}
    if kind == "quantize":
        weights, group = rng.choice([("w4", 128), ("w4", 64), ("w8", 0), ("w3", 128), ("w4", 0)])
        return {"kind": kind, "layer": rng.choice(["7b", "14b", "32b"]), "weights": weights, "group": group}
    if kind == "kl":
        return {"kind": kind, "T": _log_int(rng, 8, 1024), "V": rng.choice([VOCAB, VOCAB, rng.randrange(30000, VOCAB)]),
                "dtype": rng.choice(["bf16", "bf16", "f32"])}
    l_max = rng.choice([32, 64])
    return {"kind": kind, "B": _log_int(rng, 1, 64), "L": rng.randrange(2, l_max + 1), "l_max": l_max, "d": 384, "heads": 6, "ffn": 1536,
            "layers": 8, "rho": rng.choice([0.2, 0.4, 0.7])}


# ---- inputs ----------------------------------------------------------------------------------------------------------
class _Draw:
    """Tensors on the GPU from one seed, each call the next of its stream."""

    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(int(seed) * 7919 + 17)

    def normal(self, shape, sigma=1.0):
        return torch.randn(shape, generator=self.gen, device="cuda", dtype=torch.float32).mul_(sigma)

    def weight(self, N, K):
        return self.normal((N, K), inputs.WEIGHT_SIGMA).to(torch.bfloat16)

    def rows(self, M, K, outliers):
        x = self.normal((M, K), inputs.ACT_SIGMA)
        if outliers:
            x[:, torch.randperm(K, generator=self.gen, device="cuda")[:int(OUTLIER_FRACTION * K)]] *= 20.0
        return x.to(torch.bfloat16)

    def uniform(self, n):
        return torch.rand(n, generator=self.gen, device="cuda")


def _format(case):
    return dmr.QFormat(BITS[case["weights"]], case["group"]) if case["weights"] != "bf16" else dmr.QFormat(4, 0)


def prepare(case, seed):
    d = _Draw(seed)
    kind = case["kind"]
    state = {"kind": kind}
    if kind in ("linear", "routed"):
        fmt, M = _format(case), case["M"]
        op = OP_ROUTED if kind == "routed" else OP_DENSE if case["weights"] == "bf16" else OP_LOWBIT
        state["dense"] = op == OP_DENSE
        state["linears"] = []
        for N, K in LAYERS[case["layer"]].values():
            W = d.weight(N, K)
            state["linears"].append({
                "X": d.rows(M, K, case.get("outliers", False)),
                "W": W if op != OP_LOWBIT else None,
                "q": dmr.dmr_quantize(W, fmt) if op != OP_DENSE else None,
                "Y": torch.empty((M, N), dtype=torch.bfloat16, device="cuda"),
                "ws": dmr.new_workspace(op, M, N, K, fmt),
            })
        if kind == "routed":
            mask = (d.uniform(M) < case["p_high"]).to(torch.uint8)
            mask[0], mask[-1] = 1, 0  # both precisions are present, as work() assumes
            state["mask"] = mask
    elif kind == "quantize":
        state["fmt"] = _format(case)
        state["W"] = [d.weight(N, K) for N, K in LAYERS[case["layer"]].values()]
    elif kind == "kl":
        T, V = case["T"], case["V"]
        offsets = torch.from_numpy(inputs.step_offsets(T, 12, seed=T)).cuda()  # a batch of T tokens always has the same steps
        high = d.normal((T, V), 2.5)  # most steps agree closely, a tenth of the tokens deviates a lot
        top = torch.randint(0, V, (T, 3), generator=d.gen, device="cuda")
        high.scatter_add_(1, top, torch.tensor([9.0, 7.0, 6.0], device="cuda").expand(T, 3).contiguous())
        sigma = torch.where(d.uniform(T) < 0.1, 1.5, 0.1)
        low = d.normal((T, V)).mul_(sigma[:, None]).add_(high)
        dtype = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
        state["high"], state["low"], state["offsets"] = high.to(dtype), low.to(dtype), offsets
    else:
        kw = {k: case[k] for k in ("d", "heads", "ffn", "layers", "l_max")}
        kw["classes"] = 2
        cfg = dmr.RouterCfg(**kw)
        B, L = case["B"], case["L"]
        params = dmr.pack_router_params(inputs.router_params(**kw, seed=seed), cfg)
        # the threshold comes from the router's own scores on a calibration pool
        pool_z = d.normal((64, L, case["d"]))
        pool_n = torch.from_numpy(inputs.router_lengths(64, L, seed=seed)).cuda()
        _, pool = dmr.dmr_router_forward(params, cfg, pool_z, pool_n, score_class=1)
        lengths = inputs.router_lengths(B, L, seed=seed + 1) if B > 1 else np.array([L], dtype=np.int32)
        state.update(params=params, cfg=cfg, tau=dmr.dmr_router_calibrate(pool, case["rho"]), Z=d.normal((B, L, case["d"])),
                     lengths=torch.from_numpy(lengths).cuda(),
                     ws=torch.empty(dmr.lib().dmr_router_workspace_bytes(cfg, B, L), dtype=torch.uint8, device="cuda"))
    return state


# ---- one pass ----------------------------------------------------------------------------------------------------------
def run(state):
    kind = state["kind"]
    if kind == "linear":
        if state["dense"]:
            return [dmr.dmr_dense_linear(s["X"], s["W"], Y=s["Y"], workspace=s["ws"]) for s in state["linears"]]
        return [dmr.dmr_lowbit_linear(s["X"], s["q"], Y=s["Y"], workspace=s["ws"]) for s in state["linears"]]
    if kind == "routed":
        return [dmr.dmr_routed_linear(s["X"], state["mask"], s["W"], s["q"], Y=s["Y"], workspace=s["ws"]) for s in state["linears"]]
    if kind == "quantize":
        made = [dmr.dmr_quantize(W, state["fmt"], check=False) for W in state["W"]]
        return [[q.qweight, q.scales, q.zeros] for q in made]
    if kind == "kl":
        return dmr.dmr_stepwise_kl(state["high"], state["low"], state["offsets"])
    probs, scores = dmr.dmr_router_forward(state["params"], state["cfg"], state["Z"], state["lengths"], score_class=1, workspace=state["ws"])
    return probs, scores, dmr.dmr_router_mask(scores, state["tau"])


# ---- what a pass cannot do without ---------------------------------------------------------------------------------------
def _packed_bytes(N, K, case):
    g = case["group"] or K
    return N * K * BITS[case["weights"]] / 8 + 3 * N * (K // g)


def work(case):
    kind = case["kind"]
    nbytes = flops = 0.0
    if kind in ("linear", "routed"):
        for N, K in LAYERS[case["layer"]].values():
            if kind == "routed":
                nbytes += 2 * N * K + _packed_bytes(N, K, case)
            else:
                nbytes += 2 * N * K if case["weights"] == "bf16" else _packed_bytes(N, K, case)
            nbytes += 2 * case["M"] * (N + K)
            flops += 2.0 * case["M"] * N * K
    elif kind == "quantize":
        for N, K in LAYERS[case["layer"]].values():
            nbytes += 2 * N * K + _packed_bytes(N, K, case)
    elif kind == "kl":
        nbytes = 2.0 * case["T"] * case["V"] * (4 if case["dtype"] == "f32" else 2)
    else:
        d, ffn, B = case["d"], case["ffn"], case["B"]
        tokens = B * case["L"] if B == 1 else B * (case["L"] + 1) / 2  # valid entries: lengths are uniform in [1, L]
        layer, kv = 4 * d * d + 2 * d * ffn, 2 * d * d
        # past the keys and values of the last layer only the last valid step of a sequence is needed
        nbytes = 4.0 * (case["layers"] * layer + tokens * d)
        flops = 2.0 * (tokens * ((case["layers"] - 1) * layer + kv) + B * (layer - kv))
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times what the paths show against the same sums in 64 bits: bf16 outputs that round the other way (one unit in
    the last place is up to 2^-7 of a value: "max" 7.8e-3 seen everywhere; "rel" 5e-5 .. 3.4e-4), fp32 sums of the KL (5e-7, 1.7e-6)
    and the router's probabilities (4e-7, 9e-7)."""
    kind = case["kind"]
    if kind == "quantize":
        return "exact"
    if kind == "kl":
        return {"rel": 4e-6, "max": 2e-5}
    if kind == "router":
        return {"rel": 2e-6, "max": 4e-6}
    return {"rel": 1.2e-3, "max": 3e-2}
