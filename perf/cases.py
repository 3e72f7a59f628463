"""The work that a user of this framework has it do, as cases that can be timed.

Every case goes through the binding's public entry points, on the layer shapes of `synth.WORKLOADS` (the tiny layer, the
Mixtral-shaped layer, the fine-grained layer with shared experts, the width list {5,6,7,8}, the dense gated FFN):

  layer            one MoE layer call (`moe_forward`), decode and prefill
  stack            one layer of the decoder stack (`stack_layer`: RMSNorm + layer + residual, in place)
  routed           `route` first (a scheduler reads the histogram), then `moe_forward` on its result
  pack             MWQ quantization of one expert matrix (`pack_mwq`)
  pack_calibrated  the calibration-aware quantization (`pack_mwq_calibrated`)

A serving program keeps its packed weights, routers, workspace and output buffer; only the calls are a pass.
"""
from __future__ import annotations

import math

import torch

from paper_2504_15299_b200 import binding as B
from paper_2504_15299_b200 import synth

# the case's name for a shape -> its recipe
SHAPES = {"tiny": "tiny", "mixtral": "mixtral_decode", "finegrained": "finegrained", "mixtral_v2": "mixtral_v2",
          "dense": "dense_ffn"}
WIDTH_LISTS = ((2, 3, 4, 8), (2, 4, 8), (5, 6, 7, 8), (4, 8), (3, 5))


def _layer(name, op, shape, tokens, scales="tied", widths="drawn", gate="weights"):
    return {"name": name, "op": op, "shape": shape, "tokens": tokens, "scales": scales, "widths": widths, "gate": gate}


def listed():
    return [
        # the smallest call: a toy or test-sized layer, bound by launches and host work
        _layer("tiny_16", "layer", "tiny", 16),
        # a single chat: one token at a time
        _layer("mixtral_decode_1", "layer", "mixtral", 1),
        # one layer of a decoder stack serving sixteen sequences, widths from the learned bit-width routers
        _layer("mixtral_stack_16", "stack", "mixtral", 16, widths="router"),
        # a full decode batch (the benchmark's headline batch)
        _layer("mixtral_decode_64", "layer", "mixtral", 64),
        # an ordinary mixed batch, a ragged number of tokens, whose histogram a scheduler reads before the layer runs
        _layer("mixtral_routed_333", "routed", "mixtral", 333),
        # a prompt: prefill with skewed expert loads
        _layer("mixtral_prefill_2048", "layer", "mixtral", 2048, gate="zipf"),
        # fine-grained experts with shared ones: a large decode batch ...
        _layer("finegrained_256", "layer", "finegrained", 256),
        # ... and a prompt of ragged length with learned widths
        _layer("finegrained_prefill_1500", "layer", "finegrained", 1500, widths="router"),
        # free residual scales (one scale per extra bit, as calibration gives them): decode and prefill
        _layer("mixtral_free_decode_64", "layer", "mixtral", 64, scales="free"),
        _layer("mixtral_free_prefill_1024", "layer", "mixtral", 1024, scales="free"),
        # loading a model: one gate or up projection quantized and packed
        {"name": "pack_14336x4096", "op": "pack", "rows": 14336, "cols": 4096, "group": 128, "bits": "2,3,4,8", "scales": "tied"},
        # preparing a model: the same matrix with activation statistics and error compensation
        {"name": "pack_calibrated_14336x4096", "op": "pack_calibrated", "rows": 14336, "cols": 4096, "group": 128,
         "bits": "2,3,4,8", "scales": "free"},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["layer"] * 6 + ["stack", "routed", "pack", "pack_calibrated"])
    if op in ("pack", "pack_calibrated"):
        group = rng.choice((128, 128, 64))
        rows = _log_int(rng, 256, 14336)
        cols = group * _log_int(rng, 512 // group, (14336 if op == "pack" else 4096) // group)
        while rows * cols > 14336 * 4096:
            rows //= 2
        return {"op": op, "rows": rows, "cols": cols, "group": group, "bits": ",".join(map(str, rng.choice(WIDTH_LISTS))),
                "scales": "free" if op == "pack_calibrated" else rng.choice(("tied", "tied", "free"))}
    shape = rng.choice(("mixtral", "mixtral", "mixtral", "finegrained", "finegrained", "tiny", "mixtral_v2", "dense"))
    most = {"stack": 256, "routed": 1024, "layer": 2048}[op]
    c = _layer("", op, shape, _log_int(rng, 1, most), scales=rng.choice(("tied", "tied", "tied", "free")),
               widths=rng.choice(("drawn", "router")), gate=rng.choice(("weights", "weights", "zipf")))
    del c["name"]
    return c


def _config(case):
    free = 1 if case["scales"] == "free" else 0
    if case["op"] in ("pack", "pack_calibrated"):
        bits = tuple(int(b) for b in case["bits"].split(","))
        return B.Config(case["cols"], case["cols"], 1, 1, case["group"], bits, scale_mode=free)
    return B.Config.from_workload(synth.WORKLOADS[SHAPES[case["shape"]]], scale_mode=free)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed * 1000003 + 17)

    def normal(*shape, sigma=1.0):
        return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float32).mul_(sigma)

    cfg = _config(case)
    state = {"op": case["op"], "cfg": cfg}
    if case["op"] in ("pack", "pack_calibrated"):
        rows, cols = case["rows"], case["cols"]
        state["W"] = normal(rows, cols, sigma=0.02)
        if case["op"] == "pack_calibrated":
            # statistics of calibration activations with correlated columns of unequal energy: the second moments and the
            # upper Cholesky factor of (2 X X^T + lambda I)^-1, which the caller brings
            n = 2 * cols
            x = normal(n, cols)
            x = (x + 0.5 * x.roll(1, dims=1)) * torch.exp(0.5 * normal(cols))
            h = 2.0 * (x.T @ x).double() / n
            h.diagonal().add_(0.01 * h.diagonal().mean())
            inv = torch.cholesky_inverse(torch.linalg.cholesky(h))
            state["hc"] = torch.linalg.cholesky(inv, upper=True).float().contiguous()
            state["energy"] = x.square().sum(dim=0)
        return state

    wl = synth.WORKLOADS[SHAPES[case["shape"]]]
    T, K = case["tokens"], len(wl.bits)
    state["w"] = [B.pack_mwq(cfg, normal(*synth.expert_matrix_shape(wl, m), sigma=wl.sigma_w))
                  for _ in range(wl.n_experts + wl.n_shared) for m in range(3)]
    state["x"] = normal(T, wl.d_model).to(torch.bfloat16)
    if case["gate"] == "zipf":          # supplied router logits with a Zipf prior over the experts: unbalanced loads
        prior = -torch.log(torch.arange(1, wl.n_experts + 1, device="cuda", dtype=torch.float32))
        route = {"logits": normal(T, wl.n_experts) + prior}
    else:
        route = {"gate_w": normal(wl.n_experts, wl.d_model, sigma=wl.sigma_w).to(torch.bfloat16)}
    if case["widths"] == "router":
        route["bit_w"] = normal(wl.n_experts, K, wl.d_model, sigma=wl.sigma_w).to(torch.bfloat16)
    else:
        p = torch.tensor(wl.bit_probs, device="cuda").expand(T, -1)
        route["forced_bit_idx"] = torch.multinomial(p, wl.top_k, replacement=True, generator=gen).to(torch.int8)
    state["route"] = route
    state["workspace"] = torch.empty(B.workspace_bytes(cfg, T), dtype=torch.uint8, device="cuda")
    state["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    state["y"] = torch.empty_like(state["x"])
    state["xn"] = torch.empty_like(state["x"]) if case["op"] == "stack" else None
    return state


def run(state):
    op, cfg = state["op"], state["cfg"]
    if op == "pack":
        return B.pack_mwq(cfg, state["W"])
    if op == "pack_calibrated":
        return B.pack_mwq_calibrated(cfg, state["W"], state["hc"], state["energy"])
    ws, st, y = state["workspace"], state["status"], state["y"]
    if op == "layer":
        return B.moe_forward(cfg, state["x"], state["w"], y=y, workspace=ws, device_status=st, **state["route"])
    if op == "stack":
        y.copy_(state["x"])             # the step's hidden states arrive; the layer updates them in place
        return B.stack_layer(cfg, y, state["xn"], state["w"], workspace=ws, device_status=st, **state["route"])
    r = B.route(cfg, state["x"], workspace=ws, **state["route"])
    B.moe_forward(cfg, state["x"], state["w"], pre=r, y=y, workspace=ws, device_status=st)
    return {"y": y, "expert": r.topk_idx, "weight": r.topk_w, "width": r.bit_idx, "perm": r.perm, "inv_perm": r.inv_perm,
            "group_off": r.group_off}


def _matrix_bytes(rows, cols, group, bits, lowest, free):
    """Codes read at width `bits`, (scale, offset) of every row and group, with free scales one more scale per extra bit."""
    return rows * cols * bits / 8 + rows * (cols // group) * (4 + (2 * (bits - lowest) if free else 0))


def work(case):
    free = case["scales"] == "free"
    if case["op"] in ("pack", "pack_calibrated"):
        rows, cols = case["rows"], case["cols"]
        bits = [int(b) for b in case["bits"].split(",")]
        nbytes = rows * cols * 4 + _matrix_bytes(rows, cols, case["group"], bits[-1], bits[0], free)
        flops = rows * cols * (4 + 3 * (bits[-1] - bits[0]))
        if case["op"] == "pack_calibrated":          # every group's error leaves all later columns (a triangular update)
            nbytes += cols * cols * 4 / 2
            flops += rows * cols * (cols - case["group"])
        return {"bytes": float(nbytes), "flops": float(flops)}
    wl = synth.WORKLOADS[SHAPES[case["shape"]]]
    T, K = case["tokens"], len(wl.bits)
    p_width = [1.0 / K] * K if case["widths"] == "router" else list(wl.bit_probs)
    share = [1.0 / (e + 1) if case["gate"] == "zipf" else 1.0 for e in range(wl.n_experts)]
    share = [min(1.0, wl.top_k * s / sum(share)) for s in share]         # chance that a token selects the expert

    def expert(chance, bits):           # expected bytes: a width's own bits are read if any token needs them
        total, below = 0.0, 0
        for j, b in enumerate(bits):
            p = 1.0 - (1.0 - chance * sum(p_width[j:])) ** T
            for rows, cols in (synth.expert_matrix_shape(wl, m) for m in range(3)):
                full = _matrix_bytes(rows, cols, wl.group_size, b, bits[0], free)
                total += p * (full - (_matrix_bytes(rows, cols, wl.group_size, below, bits[0], free) if j else 0.0))
            below = b
        return total

    nbytes = sum(expert(s, wl.bits) for s in share)
    nbytes += wl.n_shared * sum(_matrix_bytes(*synth.expert_matrix_shape(wl, m), wl.group_size, wl.bits[-1], wl.bits[0], free)
                                for m in range(3))
    nbytes += 2 * T * wl.d_model * 2                                     # tokens in, results out
    nbytes += wl.n_experts * (4 * T if case["gate"] == "zipf" else 2 * wl.d_model)
    if case["widths"] == "router":
        nbytes += wl.n_experts * K * wl.d_model * 2
    flops = 2.0 * T * (wl.top_k + wl.n_shared) * 3 * wl.d_model * wl.d_ffn
    return {"bytes": float(nbytes), "flops": flops}


def tolerance(case):
    if case["op"] in ("pack", "pack_calibrated"):
        return "exact"                  # codes, scales and layout are pinned bit for bit
    # bf16 outputs (2^-9 per rounding) of products in 16-bit (fp16 or 15-bit integer) operands with fp32 accumulation, an
    # intermediate rounded to 16 bits on the way; routing (whole numbers) is pinned
    return {"rel": 5e-3, "max": 5e-2}
