"""The measured workloads of this framework: one MoE layer forward through its public entry points.

All cases use the DeepSeek-V3 layer shape of `synthetic.DSV3` (hidden 7168, intermediate 2048, 256 experts,
top-8) with `experts` of the 256 experts on this GPU: 32 (one of eight expert-parallel ranks, the busiest one) or
all 256.

A case is
  entry    "forward" (FP8 activations on the device), "hidden" (bf16 hidden states: router projection and input
           quantisation in front) or "host" (per-step tensors in pinned host memory, one synchronous call)
  tokens   batch size of the step
  experts  local experts
  skew     True: four hot experts (the skewed recipe of `synthetic.make_inputs`)
  layout   layout of the activation scales: 0 = [T, H/128], 1 = [H/128, T]
"""
import dataclasses

import torch

from paper_2608_14560_b200 import MoeFp8
from paper_2608_14560_b200 import synthetic as syn

MAX_TOKENS = 16384


def _case(entry, tokens, experts, skew=False, layout=0, name=None):
    c = {"entry": entry, "tokens": tokens, "experts": experts, "skew": skew, "layout": layout}
    return c if name is None else {"name": name, **c}


def listed():
    return [
        # one interactive request decoding: a single token, a few active experts, pure latency
        _case("forward", 1, 32, name="decode_T1_E32"),
        # a lightly loaded decode step on an expert-parallel rank
        _case("forward", 8, 32, name="decode_T8_E32"),
        # the median decode batch of the benchmark sweep
        _case("forward", 54, 32, name="decode_T54_E32"),
        # decode with the whole layer on one GPU: hundreds of experts with one or two rows each
        _case("forward", 33, 256, name="decode_T33_E256"),
        # decode inside a model: the layer starts from the bf16 hidden states
        _case("hidden", 16, 32, name="hidden_T16_E32"),
        # a heavily loaded decode step or a short prompt, just past a row-tile edge, scales laid out by a
        # producer that writes them block-major
        _case("forward", 257, 32, layout=1, name="prefill_T257_E32_scaleT"),
        # a chunk of a prompt, odd size
        _case("forward", 901, 32, name="prefill_T901_E32"),
        # chunked prefill inside a model, from bf16 hidden states
        _case("hidden", 1024, 32, name="hidden_T1024_E32"),
        # a step whose tensors live in host memory (CPU-side caller)
        _case("host", 512, 32, name="host_T512_E32"),
        # a long prompt on an expert-parallel rank: a few row tiles per expert, the last ones ragged
        _case("forward", 4096, 32, name="prefill_T4096_E32"),
        # prefill with badly balanced routing: a handful of hot experts take most rows
        _case("forward", 8192, 32, skew=True, name="prefill_T8192_E32_skew"),
        # the largest prefill: all experts local
        _case("forward", 16384, 256, name="prefill_T16384_E256"),
    ]


def draw(rng):
    entry = rng.choice(("forward", "forward", "forward", "hidden", "host"))
    experts = rng.choice((32, 32, 32, 256))
    tokens = max(1, min(MAX_TOKENS, int(round(MAX_TOKENS ** rng.random()))))
    if entry != "forward":
        # the projection and the host copies come on top of the layer: within the cost of the largest listed case
        tokens = min(tokens, 8192)
    skew = rng.random() < 0.25
    layout = 1 if rng.random() < 0.25 else 0
    return _case(entry, tokens, experts, skew, layout)


def _workload(case, seed):
    dims = dataclasses.replace(syn.DSV3, num_local_experts=case["experts"])
    return syn.Workload("case", case["tokens"], dims, seed=seed, skew=case["skew"])


def prepare(case, seed):
    dev = torch.device("cuda:0")
    wl = _workload(case, seed)
    d = wl.dims
    inp = syn.make_inputs(wl, dev)
    if not case["skew"]:  # (the skewed recipe puts its hot experts on the first rank)
        inp["local_expert_offset"] = _busiest_rank(_slots_of_experts(inp["router_logits"], inp["routing_bias"]),
                                                   case["experts"])
    if case["layout"]:
        inp["hidden_scale"] = inp["hidden_scale"].t().contiguous()
    eng = MoeFp8(d.hidden, d.intermediate, d.num_experts, d.num_local_experts, d.n_group, d.topk_group, d.top_k,
                 max_tokens=wl.tokens, hidden_scale_layout=case["layout"], device=dev)
    state = {"entry": case["entry"], "engine": eng, "inp": inp}
    if case["entry"] == "hidden":
        inp.update(syn.make_router_inputs(wl, dev))
        for k in ("hidden_fp8", "hidden_scale", "router_logits"):
            del inp[k]
    elif case["entry"] == "host":
        state["host"] = {k: inp.pop(k).cpu().pin_memory() for k in ("hidden_fp8", "hidden_scale", "router_logits")}
        state["host_out"] = torch.empty(wl.tokens, d.hidden, dtype=torch.bfloat16).pin_memory()
    return state


def run(state):
    eng = state["engine"]
    if state["entry"] == "forward":
        return eng.forward(state["inp"])
    if state["entry"] == "hidden":
        return eng.forward_from_hidden(state["inp"])
    return eng.forward_host(state["host"], state["inp"], state["host_out"])


def _slots_of_experts(logits, bias):
    """Rows of every expert: the eight best experts of the four best groups, a group scored by its two best."""
    T, E, G = logits.shape[0], syn.DSV3.num_experts, syn.DSV3.n_group
    biased = torch.sigmoid(logits) + bias.float()
    group = biased.view(T, G, E // G).topk(2, dim=-1).values.sum(-1)
    kept = torch.zeros_like(group).scatter_(1, group.topk(syn.DSV3.topk_group, dim=-1).indices, 1.0)
    biased = biased.masked_fill(kept.repeat_interleave(E // G, dim=1) == 0, -1.0e9)
    return torch.bincount(biased.topk(syn.DSV3.top_k, dim=-1).indices.flatten(), minlength=E)


def _busiest_rank(counts, experts):
    """First expert of the slice with the most active experts (then the most rows): an expert-parallel step waits
    for that rank."""
    per_rank = counts.view(-1, experts)
    return int(((per_rank > 0).sum(1) * 10 ** 6 + per_rank.sum(1)).argmax()) * experts


def _expected_load(case):
    """(local slots, active local experts) of a batch of this case, averaged over four draws of the input recipe's
    logits and biases."""
    T, E = case["tokens"], syn.DSV3.num_experts
    slots = active = 0.0
    draws = 4 if T <= 4096 else 1
    for i in range(draws):
        g = torch.Generator()
        g.manual_seed(1000 + i)
        logits = torch.randn(T, E, generator=g)
        bias = 0.1 * torch.randn(E, generator=g)
        first = 0
        if case["skew"]:
            boost = (1.0 + torch.randperm(E, generator=g)).pow(-1.1)
            boost[torch.tensor(syn.SKEW_HOT_EXPERTS)] = 3.0
            bias = bias + boost
        counts = _slots_of_experts(logits, bias)
        if not case["skew"]:
            first = _busiest_rank(counts, case["experts"])
        counts = counts[first: first + case["experts"]]
        slots += float(counts.sum()) / draws
        active += float((counts > 0).sum()) / draws
    return slots, active


def work(case):
    """Every active expert's weights and scales once, the step's inputs and output once; the two GEMMs of every
    local (token, expert) pair and, from hidden states, the router projection."""
    H, I, E, T = syn.DSV3.hidden, syn.DSV3.intermediate, syn.DSV3.num_experts, case["tokens"]
    slots, active = _expected_load(case)
    per_expert = 3 * I * H + 4 * 3 * (I // 128) * (H // 128)
    nbytes = active * per_expert + 2 * E + T * H * 2
    flops = slots * 2.0 * 3 * I * H
    if case["entry"] == "hidden":
        nbytes += T * H * 2 + E * H * 2
        flops += 2.0 * T * H * E
    else:
        nbytes += T * (H + H // 32 + 4 * E)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Measured against the same layer in 64 bits (8 to 3000 tokens): rel 2.35e-3, largest difference 0.023 of the
    # value -- the two bf16 roundings of the output and single re-quantised codes that land on the other side of
    # a rounding boundary.
    return {"rel": 0.01, "max": 0.1}
