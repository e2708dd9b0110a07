"""GPU parity: the CUDA path, called through the C ABI, against the CPU oracle
on the same seeded inputs.  Routing indices and the permutation are compared
bit for bit, the bf16 output with the tolerance of the workload definition."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
from paper_2608_14560_b200 import MoeFp8, MoeFp8Error
from paper_2608_14560_b200 import synthetic as syn

from parity import check_output, make_engine, run_and_compare

pytestmark = pytest.mark.gpu

SMALL = syn.LayerDims(hidden=512, intermediate=256, num_local_experts=32)


def _wl(tokens, dims=SMALL, seed=0, **kw):
    return syn.Workload(f"t{tokens}", tokens, dims, seed, **kw)


# ---- small layer, every token compared ------------------------------------
@pytest.mark.parametrize("tokens", [1, 7, 32, 33, 130, 512, 513, 1000])  # 512|513: launch-scheme boundary
def test_small_layer_all_tokens(cuda_device, tokens):
    st = run_and_compare(_wl(tokens, seed=tokens), cuda_device)
    assert st["frac"] >= 0.995


def test_small_layer_skewed_many_tiles_per_expert(cuda_device):
    # hot experts receive every token: several 128-row tiles per expert plus a ragged tail
    st = run_and_compare(_wl(1111, seed=9, skew=True), cuda_device)
    assert st["S"] > 4 * 1111


def test_all_experts_local(cuda_device):
    dims = dataclasses.replace(SMALL, num_local_experts=256)
    st = run_and_compare(_wl(333, dims, seed=5), cuda_device)
    assert st["S"] == 333 * 8


@pytest.mark.parametrize("off,eloc", [(32, 32), (224, 32), (5, 3), (0, 1)])
def test_local_expert_offsets(cuda_device, off, eloc):
    dims = dataclasses.replace(SMALL, num_local_experts=eloc)
    run_and_compare(_wl(200, dims, seed=off + eloc, local_expert_offset=off), cuda_device)


@pytest.mark.parametrize("tokens,eloc,off", [(9, 256, 0), (60, 256, 0), (80, 3, 5), (33, 1, 0), (70, 1, 7)])
def test_fused_small_batch_kernel_with_many_and_with_few_local_experts(cuda_device, tokens, eloc, off):
    # all experts local: a couple of hundred one- or two-row tiles; one local expert: every local row in one
    # expert, i.e. up to three sub-tiles of the same weights
    dims = dataclasses.replace(SMALL, num_local_experts=eloc)
    wl = _wl(tokens, dims, seed=300 + tokens + eloc, local_expert_offset=off)
    inp = syn.make_inputs(wl, cuda_device)
    eng = make_engine(wl, cuda_device)
    got = eng.forward(inp).clone()
    assert eng.last_launch_count() <= 2
    eng.set_small_batch_fusion(False)
    want = eng.forward(inp).clone()
    torch.cuda.synchronize()
    assert eng.status() == 0 and eng.last_launch_count() == 5
    assert torch.equal(got.view(torch.int16), want.view(torch.int16))
    eng.set_small_batch_fusion(True)
    run_and_compare(wl, cuda_device, inp=inp, eng=eng)
    eng.close()


def test_scale_layout_and_gate_order_flags(cuda_device):
    wl = _wl(97, seed=3)
    inp = syn.make_inputs(wl, cuda_device)
    inp_t = dict(inp, hidden_scale=inp["hidden_scale"].t().contiguous())
    run_and_compare(wl, cuda_device, inp=inp_t, hidden_scale_layout=1)
    I = wl.dims.intermediate
    inp_s = dict(inp, w13=torch.cat([inp["w13"][:, I:], inp["w13"][:, :I]], 1).contiguous(),
                 w13_scale=torch.cat([inp["w13_scale"][:, I // 128:], inp["w13_scale"][:, :I // 128]], 1).contiguous())
    run_and_compare(wl, cuda_device, inp=inp_s, gate_first=False)


# ---- degenerate cases -------------------------------------------------------
def test_zero_tokens_and_argument_errors(cuda_device):
    wl = _wl(0)
    inp = syn.make_inputs(wl, cuda_device)
    eng = make_engine(wl, cuda_device, max_tokens=16)
    out = eng.forward(inp)
    assert out.shape == (0, 512) and eng.last_launch_count() == 0
    big = syn.make_inputs(_wl(17), cuda_device)
    with pytest.raises(MoeFp8Error) as ei:
        eng.forward(big)  # T > max_tokens
    assert ei.value.rc == -1
    with pytest.raises(MoeFp8Error):
        eng.forward(dict(syn.make_inputs(_wl(4), cuda_device), local_expert_offset=250))
    with pytest.raises(MoeFp8Error):
        MoeFp8(hidden=500, device=cuda_device)
    eng.close()


def test_no_token_routes_locally(cuda_device):
    wl = _wl(64, seed=1)
    inp = syn.make_inputs(wl, cuda_device)
    inp["router_logits"][:, :32] = -20.0  # local experts (group 0) never win
    st = run_and_compare(wl, cuda_device, inp=inp)
    assert st["S"] == 0


@pytest.mark.parametrize("tokens", [1, 16, 17, 80])  # one launch | behind the routing kernel
def test_fused_kernel_without_a_tile_between_batches_that_have_some(cuda_device, tokens):
    inp = syn.make_inputs(_wl(tokens, seed=19), cuda_device)
    none = dict(inp, router_logits=inp["router_logits"].clone())
    none["router_logits"][:, :32] = -20.0
    eng = make_engine(_wl(tokens), cuda_device)
    run_and_compare(_wl(tokens, seed=19), cuda_device, inp=inp, eng=eng)
    want = eng.forward(inp).clone()
    for n in (1, 2, 3):  # (the two counter sets take turns)
        for _ in range(n):
            out = torch.full_like(want, float("nan"))
            eng.forward(none, out)
            assert not out.view(torch.int16).any()
        got = eng.forward(inp).clone()
        assert eng.status() == 0 and torch.equal(got.view(torch.int16), want.view(torch.int16))
    eng.close()


def test_every_token_on_the_same_experts(cuda_device):
    wl = _wl(300, seed=2)
    inp = syn.make_inputs(wl, cuda_device)
    inp["router_logits"][:] = -8.0
    inp["router_logits"][:, [1, 2, 3, 4, 40, 41, 80, 120]] = 6.0
    st = run_and_compare(wl, cuda_device, inp=inp)
    assert st["S"] == 4 * 300 and st["active"] == 4


def test_exact_score_ties_break_to_smaller_index(cuda_device):
    wl = _wl(50, seed=4)
    inp = syn.make_inputs(wl, cuda_device)
    inp["router_logits"][:] = 0.25
    inp["routing_bias"][:] = 0
    run_and_compare(wl, cuda_device, inp=inp)
    inp["router_logits"][:, 128:] = 0.5  # ties inside and across groups 4..7
    run_and_compare(wl, cuda_device, inp=inp)


def test_run_to_run_determinism_and_workspace_reuse(cuda_device):
    wl = _wl(500, seed=6)
    inp = syn.make_inputs(wl, cuda_device)
    eng = make_engine(wl, cuda_device, max_tokens=600)
    a = eng.forward(inp).clone()
    other = syn.make_inputs(_wl(77, seed=8), cuda_device)
    eng.forward(other)  # different T in between: stale scratch must not leak
    b = eng.forward(inp).clone()
    torch.cuda.synchronize()
    assert torch.equal(a.view(torch.int16), b.view(torch.int16))
    run_and_compare(_wl(77, seed=8), cuda_device, inp=other, eng=eng)
    eng.close()


def test_many_batch_sizes_back_to_back_on_one_handle(cuda_device):
    # 600 forwards in random order over batch sizes on both sides of every launch-scheme boundary: the counters
    # and scratch a forward leaves behind must never change the next one (bit-identical outputs, clean status)
    sizes = [1, 8, 32, 33, 128, 129, 512, 513, 700, 2048, 2049]
    inputs = {T: syn.make_inputs(_wl(T, seed=300 + T, skew=(T % 3 == 0)), cuda_device) for T in sizes}
    eng = make_engine(_wl(max(sizes)), cuda_device)
    want = {T: eng.forward(inputs[T]).clone() for T in sizes}
    torch.cuda.synchronize()
    assert eng.status() == 0
    order = np.random.default_rng(5).choice(len(sizes), 600)
    for i, k in enumerate(order):
        T = sizes[k]
        got = eng.forward(inputs[T])
        if i % 20 == 19:
            assert torch.equal(got.view(torch.int16), want[T].view(torch.int16)), f"forward {i}, T={T}"
            assert eng.status() == 0
    run_and_compare(_wl(129, seed=300 + 129, skew=True), cuda_device, inp=inputs[129], eng=eng)
    eng.close()


def test_host_entry_point_matches_device_entry_point(cuda_device):
    wl = _wl(260, seed=12)
    inp = syn.make_inputs(wl, cuda_device)
    eng = make_engine(wl, cuda_device)
    ref = eng.forward(inp).cpu()
    host_act = {k: inp[k].cpu().pin_memory() for k in ("hidden_fp8", "hidden_scale", "router_logits")}
    host_out = torch.empty(wl.tokens, 512, dtype=torch.bfloat16).pin_memory()
    eng.forward_host(host_act, inp, host_out)
    assert torch.equal(ref.view(torch.int16), host_out.view(torch.int16))
    eng.close()


@pytest.mark.parametrize("tokens", [300, 20])  # separate kernels | fused kernel
def test_host_calls_in_a_row_with_other_inputs_each(cuda_device, tokens):
    # on one handle and on a side stream, the batch before always half as long or twice as long; a forward from hidden
    # states, which fills the same staging areas, in between
    wl = _wl(tokens, seed=14)
    weights = syn.make_inputs(wl, cuda_device)
    eng = make_engine(wl, cuda_device)
    side = torch.cuda.Stream(device=cuda_device)
    r = syn.make_router_inputs(wl, cuda_device)
    want_hidden = eng.forward_from_hidden({**weights, **r}).clone()
    torch.cuda.synchronize()
    for i in range(4):
        b = syn.make_inputs(_wl(tokens if i % 2 else tokens // 2, seed=15 + i), cuda_device)
        acts = {k: b[k] for k in ("hidden_fp8", "hidden_scale", "router_logits")}
        want = eng.forward({**weights, **acts}).cpu()
        host = {k: v.cpu().pin_memory() for k, v in acts.items()}
        host_out = torch.empty(want.shape, dtype=torch.bfloat16).pin_memory()
        with torch.cuda.stream(side):
            eng.forward_host(host, weights, host_out)
            got_hidden = eng.forward_from_hidden({**weights, **r})
            for v in host.values():  # the call has returned: its buffers are the caller's again
                v.view(torch.uint8).fill_(0xFF)
        assert torch.equal(want.view(torch.int16), host_out.view(torch.int16)), f"call {i}"
        side.synchronize()
        assert eng.status() == 0
        assert torch.equal(got_hidden.view(torch.int16), want_hidden.view(torch.int16)), f"call {i}"
    eng.close()


@pytest.mark.parametrize("tokens", [300, 20])  # separate kernels | fused kernel
def test_a_rejected_call_has_enqueued_nothing(cuda_device, tokens):
    # the entry points that copy or compute something in front of the forward: after one that returned an argument
    # error the staging areas still hold what the last accepted call fed to the forward, and the next call is right
    wl = _wl(tokens, seed=16)
    inp = syn.make_inputs(wl, cuda_device)
    acts = {k: inp[k] for k in ("hidden_fp8", "hidden_scale", "router_logits")}
    other = {k: v.cpu().pin_memory() for k, v in syn.make_activations(wl, 17, cuda_device).items()}
    r = {"hidden_bf16": (torch.ones(tokens, 512, device=cuda_device) * 3).bfloat16(),
         "router_weight": torch.ones(256, 512, device=cuda_device).bfloat16()}
    host = {k: v.cpu().pin_memory() for k, v in acts.items()}
    host_out = torch.empty(tokens, 512, dtype=torch.bfloat16).pin_memory()
    eng = make_engine(wl, cuda_device)
    want = eng.forward(inp).cpu()
    shifted = torch.zeros(inp["w2"].numel() + 16, dtype=torch.uint8, device=cuda_device)[1:]
    for bad in ({"local_expert_offset": 250}, {"local_expert_offset": -1}, {"w2": shifted}, {"w13_scale": None}):
        for entry in (lambda w: eng.forward_host(other, w, host_out), lambda w: eng.forward_host_async(other, w, host_out),
                      lambda w: eng.forward_from_hidden({**w, **r})):
            eng.forward_host(host, inp, host_out)
            with pytest.raises(MoeFp8Error) as ei:
                entry({**inp, **bad})
            assert ei.value.rc == -1
            torch.cuda.synchronize()
            fed = eng.debug_export_inputs(tokens)
            assert torch.equal(fed["router_logits"], acts["router_logits"])
            assert torch.equal(fed["hidden_fp8"], acts["hidden_fp8"].view(torch.uint8))
            assert torch.equal(fed["hidden_scale"], acts["hidden_scale"])
    host_out.zero_()
    eng.forward_host(host, inp, host_out)
    assert eng.status() == 0 and torch.equal(host_out.view(torch.int16), want.view(torch.int16))
    eng.close()


def test_forward_on_a_side_stream_and_after_a_change_of_weights(cuda_device):
    # the forward is enqueued on the caller's current stream; the TMA descriptors of the weights are cached
    # per pointer pair and must be rebuilt when other weight tensors are passed
    wl = _wl(150, seed=21)
    inp_a = syn.make_inputs(wl, cuda_device)
    inp_b = syn.make_inputs(_wl(150, seed=22), cuda_device)
    fresh = make_engine(wl, cuda_device)
    want_b = fresh.forward(inp_b).clone()
    fresh.close()
    eng = make_engine(wl, cuda_device)
    side = torch.cuda.Stream(device=cuda_device)
    side.wait_stream(torch.cuda.current_stream(cuda_device))
    with torch.cuda.stream(side):
        eng.forward(inp_a)
        got_b = eng.forward(inp_b).clone()
    side.synchronize()
    assert eng.status() == 0
    assert torch.equal(want_b.view(torch.int16), got_b.view(torch.int16))
    run_and_compare(wl, cuda_device, inp=inp_a, eng=eng)
    eng.close()


# ---- the five benchmark workloads at full size -----------------------------
def _sample(T, n, seed):
    if T <= n:
        return None
    return np.sort(np.random.default_rng(seed).choice(T, n, replace=False)).astype(np.int32)


# Output: every token up to T = 1024, else 256 random tokens.  Per-slot rows (re-quantised intermediate and
# down-projection row): on the large workloads every row of the first and the last row tile of the largest
# expert segment, of the smallest non-empty segment and of the first tile of a median one -- whole tiles at the
# full K depth, on CTAs that have walked many tiles before them.
@pytest.mark.parametrize("cfg,n_sample,rows", [(0, 8, True), (1, 64, True), (2, 1024, "tiles"), (3, 256, "tiles")])
def test_benchmark_workloads_32_local_experts(cuda_device, cfg, n_sample, rows):
    wl = syn.CONFIGS[cfg]
    st = run_and_compare(wl, cuda_device, sample_tokens=_sample(wl.tokens, n_sample, cfg), check_rows=rows)
    print(wl.name, st)


@pytest.mark.parametrize("tokens,n_sample,rows", [(7, 7, True), (54, 54, True), (14107, 256, "tiles")])
def test_token_counts_quoted_in_the_paper(cuda_device, tokens, n_sample, rows):
    # the paper's table of workload regimes (short / median / long) quotes one latency each for T = 7, 54 and
    # 14107 tokens with 32 local experts
    base = syn.CONFIGS[1]
    wl = syn.Workload(f"dsv3_T{tokens}_E32", tokens, base.dims, base.seed, base.local_expert_offset,
                      base.scaling_factor, base.skew)
    st = run_and_compare(wl, cuda_device, sample_tokens=_sample(tokens, n_sample, tokens), check_rows=rows)
    print(wl.name, st)


def test_benchmark_workload_all_256_experts_local(cuda_device):
    wl = syn.CONFIGS[4]
    st = run_and_compare(wl, cuda_device, sample_tokens=_sample(wl.tokens, 256, 4), check_rows="tiles")
    assert st["S"] == wl.tokens * 8
    print(wl.name, st)


def test_routing_on_logits_far_outside_the_unit_range(cuda_device):
    # the fixed-operation sigmoid on its clamped tails and at large |logit|: indices and weights of the
    # kernel must equal the oracle's bit for bit there too, not only on N(0,1) logits
    wl = _wl(256, seed=31)
    inp = syn.make_inputs(wl, cuda_device)
    g = torch.Generator(device=cuda_device)
    g.manual_seed(77)
    mags = torch.tensor([8.0, 20.0, 87.0, 88.0, 100.0, 1e4, 0.015625, 3.0], device=cuda_device)
    pick = torch.randint(0, len(mags), inp["router_logits"].shape, generator=g, device=cuda_device)
    sign = torch.randint(0, 2, inp["router_logits"].shape, generator=g, device=cuda_device) * 2.0 - 1.0
    inp["router_logits"] = (mags[pick] * sign).contiguous()
    run_and_compare(wl, cuda_device, inp=inp)
    # a dense sweep of the benchmark's 1/64 grid over [-32, 32] and of large magnitudes, one value per expert column
    T = 4096 // 256 * 2
    grid = (torch.arange(-2048, 2048, device=cuda_device, dtype=torch.float32) / 64.0).view(-1, 256)
    big = (torch.arange(-2048, 2048, device=cuda_device, dtype=torch.float32) / 16.0).view(-1, 256)
    wl2 = _wl(T, seed=32)
    inp2 = syn.make_inputs(wl2, cuda_device)
    inp2["router_logits"] = torch.cat([grid, big]).contiguous()
    run_and_compare(wl2, cuda_device, inp=inp2)


def test_device_sigmoid_bits_equal_the_oracle(cuda_device):
    # every point of the benchmark's logit grid (k/64, |k| <= 2048), the clamp boundaries and 2^20 random
    # floats over the whole finite range: the kernel's sigmoid and the oracle's agree in every bit
    from paper_2608_14560_b200 import binding
    rng = np.random.default_rng(11)
    grid = (np.arange(-2048, 2049) / 64.0).astype(np.float32)
    edge = np.float32([0.0, -0.0, 87.0, -87.0, 88.0, -88.0, 88.5, -88.5, 100.0, -100.0, 1e4, -1e4, 3e38, -3e38,
                       1e-30, -1e-30, 1e-45, 0.34657359, -0.34657359])
    rnd_bits = rng.integers(0, 1 << 32, 1 << 20, dtype=np.uint64).astype(np.uint32)
    rnd = rnd_bits.view(np.float32)
    rnd = rnd[np.isfinite(rnd)]
    mid = (rng.standard_normal(1 << 18) * 6.0).astype(np.float32)
    x = np.concatenate([grid, edge, rnd, mid]).astype(np.float32)
    got = binding.debug_sigmoid(torch.from_numpy(x).to(cuda_device)).cpu().numpy()
    want = oracle.sigmoid(x)
    assert np.array_equal(got.view(np.uint32), want.view(np.uint32)), \
        f"{(got.view(np.uint32) != want.view(np.uint32)).sum()} of {x.size} sigmoid values differ"


def test_a_wait_that_runs_out_is_reported_and_the_handle_stays_usable(cuda_device):
    # The copy producer of GEMM1 is told to stop before its third pipeline stage and every wait limit is
    # shortened to 2^20 clocks: the consumers' waits give up, the kernel returns with a time-out code in the
    # status word (nothing traps, nothing spins without a bound), and the next forward on the same handle,
    # with the hook off again, is bit-identical to a forward on a fresh handle.
    wl = _wl(300, seed=41)
    inp = syn.make_inputs(wl, cuda_device)
    fresh = make_engine(wl, cuda_device)
    want = fresh.forward(inp).clone()
    torch.cuda.synchronize()
    fresh.close()
    eng = make_engine(wl, cuda_device)
    eng.debug_set_fault(skip_iteration=2, wait_clocks=1 << 20)
    eng.forward(inp)
    torch.cuda.synchronize()
    assert 1 <= eng.status() <= 5, f"expected a time-out code, got {eng.status()}"
    eng.debug_set_fault(-1, 0)
    got = eng.forward(inp).clone()
    torch.cuda.synchronize()
    assert eng.status() == 0
    assert torch.equal(got.view(torch.int16), want.view(torch.int16))
    run_and_compare(wl, cuda_device, inp=inp, eng=eng)
    eng.close()


@pytest.mark.parametrize("tokens,eloc", [(9, 32), (48, 32), (200, 32), (300, 32), (2000, 256)])
@pytest.mark.parametrize("clocks", [1 << 16, 1])  # 1: the roles give up before others have begun, copies still in flight
def test_an_abort_leaves_nothing_under_way(cuda_device, tokens, eloc, clocks):
    # one launch | fused behind the routing kernel | a launch per GEMM, overlapping | both GEMMs in one, the last with lists of
    # several tiles per CTA.  The copy producer stops at its first few stages, before and behind a full ring and a tile's
    # end: what was claimed and issued by then has to be waited for (status 5 would say that it was not all there), and the
    # forward that follows at once, whose CTAs get the shared and tensor memory, must be right
    wl = _wl(tokens, dataclasses.replace(SMALL, num_local_experts=eloc), seed=44)
    inp = syn.make_inputs(wl, cuda_device)
    eng = make_engine(wl, cuda_device)
    want = eng.forward(inp).clone()
    torch.cuda.synchronize()
    assert eng.status() == 0
    for skip in (0, 1, 2, 3, 4, 5, 6, 7, 9) + ((-1,) if clocks == 1 else ()):
        eng.debug_set_fault(skip_iteration=skip, wait_clocks=clocks)
        eng.forward(inp)
        eng.debug_set_fault(-1, 0)
        got = eng.forward(inp)
        torch.cuda.synchronize()
        assert eng.status() == 0
        assert torch.equal(got.view(torch.int16), want.view(torch.int16)), skip
        eng.debug_set_fault(skip_iteration=skip, wait_clocks=clocks)
        eng.forward(inp)
        torch.cuda.synchronize()
        assert eng.status() in (0, 1, 2, 3, 4, 8), skip
        eng.debug_set_fault(-1, 0)
    eng.close()


def test_stage_times_name_the_launches_of_a_forward(cuda_device):
    gemms = {"route_topk", "gather_rows", "gemm1_swiglu_quant", "gemm2", "combine"}
    joint = {"route_topk", "gather_rows", "grouped_mlp", "combine"}
    eng = make_engine(_wl(300), cuda_device)
    # (callers may keep the numbers)
    assert eng.stage_names()[:9] == ["route_topk", "count", "scan", "place", "gather_rows", "gemm1_swiglu_quant", "gemm2",
                                     "combine", "fused_small"]
    eng.set_stage_timing(True)
    for tokens, stages in ((9, {"fused_small"}), (40, {"route_topk", "fused_small"}), (200, gemms), (300, joint), (9, {"fused_small"})):
        inp = syn.make_inputs(_wl(tokens, seed=tokens), cuda_device)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        eng.forward(inp)
        b.record()
        times = eng.get_stage_times()
        torch.cuda.synchronize()
        assert {k for k, v in times.items() if v > 0} == stages and eng.last_launch_count() == len(stages)
        assert sum(times.values()) <= a.elapsed_time(b) + 1e-3
    eng.set_stage_timing(False)
    with pytest.raises(MoeFp8Error):
        eng.get_stage_times()
    eng.close()


# ---- the layer started from bf16 hidden states (router projection + input quantisation in front) ----------
def _from_hidden_case(wl, device, sample_tokens=None, **kw):
    d = wl.dims
    inp = syn.make_inputs(wl, device)
    r = syn.make_router_inputs(wl, device)
    eng = make_engine(wl, device, **kw)
    out = eng.forward_from_hidden({**inp, **r})
    fed = eng.debug_export_inputs(wl.tokens)
    dbg = eng.debug_export(wl.tokens, rows=False)
    torch.cuda.synchronize()
    assert int(dbg["status"].item()) == 0
    host = syn.to_host({**inp, **r})
    # projection and quantisation: bit for bit (the summation order of the projection is part of its definition)
    logits = oracle.router_logits(host["hidden_bf16"], host["router_weight"])
    assert np.array_equal(fed["router_logits"].cpu().numpy().view(np.uint32), logits.view(np.uint32)), \
        "router logits differ from the oracle's fixed-order sum"
    q, s = oracle.quantize_rows(host["hidden_bf16"])
    assert np.array_equal(fed["hidden_fp8"].cpu().numpy(), q)
    gs = fed["hidden_scale"].cpu().numpy()
    assert np.array_equal(gs.T if eng.cfg.hidden_scale_layout else gs, s)
    # routing from those logits: indices and weights bit for bit
    ridx, rw = oracle.route(logits, host["routing_bias"], d.n_group, d.topk_group, d.top_k, float(inp["scaling_factor"]))
    assert np.array_equal(dbg["topk_idx"].cpu().numpy(), ridx)
    assert np.array_equal(dbg["topk_w"].cpu().numpy(), rw)
    # output
    tokens = np.arange(wl.tokens, dtype=np.int32) if sample_tokens is None else sample_tokens
    full = dict(host, hidden_fp8=q, hidden_scale=s, router_logits=logits)
    from parity import oracle_forward_parallel
    ref = oracle_forward_parallel(full, d, tokens)
    gpu = out.view(torch.int16).cpu().numpy().view(np.uint16)[tokens]
    check_output(gpu, ref)
    eng.close()
    return int(((ridx >= wl.local_expert_offset) & (ridx < wl.local_expert_offset + d.num_local_experts)).sum())


@pytest.mark.parametrize("tokens", [1, 8, 33, 128, 129, 700])  # 128 | 129: the two tile shapes of the projection
def test_from_hidden_small_layer(cuda_device, tokens):
    _from_hidden_case(_wl(tokens, seed=60 + tokens), cuda_device)


@pytest.mark.parametrize("tokens,hidden", [(3, 256), (64, 768), (65, 256), (127, 1280), (128, 768), (128, 512), (129, 768), (129, 512),
                                           (257, 512), (2047, 256), (2048, 256), (2049, 512), (2053, 1280)])
def test_from_hidden_at_the_edges_of_the_projection_shapes(cuda_device, tokens, hidden):
    # the two warp tiles of the projection (up to 128 tokens and above) with ragged last tiles, K from fewer chunks than pipeline
    # stages up, and hidden sizes that the chunks of 512 do not divide
    dims = syn.LayerDims(hidden=hidden, intermediate=128, num_local_experts=32)
    _from_hidden_case(_wl(tokens, dims, seed=600 + tokens), cuda_device, sample_tokens=_sample(tokens, 64, tokens))


@pytest.mark.parametrize("tokens,hidden", [(1, 512), (63, 1024), (64, 2560)])
def test_from_hidden_of_small_batches_in_chunks_of_512(cuda_device, tokens, hidden):
    # fewer chunks than pipeline stages (1 and 2 of 4) and one more
    dims = syn.LayerDims(hidden=hidden, intermediate=128, num_local_experts=32)
    _from_hidden_case(_wl(tokens, dims, seed=650 + tokens), cuda_device)


def test_from_hidden_transposed_scale_layout(cuda_device):
    _from_hidden_case(_wl(77, seed=59), cuda_device, hidden_scale_layout=1)


@pytest.mark.parametrize("cfg,n_sample", [(1, 64), (2, 128)])
def test_from_hidden_benchmark_shapes(cuda_device, cfg, n_sample):
    wl = syn.CONFIGS[cfg]
    S = _from_hidden_case(wl, cuda_device, sample_tokens=_sample(wl.tokens, n_sample, cfg))
    assert S > 0


# ---- batches of at most 4 tokens: GEMM1's K range of every tile cut over several CTAs ------------------------
@pytest.mark.parametrize("tokens,eloc,off,seed", [(1, 32, 0, 3), (2, 32, 0, 1), (3, 32, 0, 2), (4, 32, 0, 0), (4, 1, 7, 5),
                                                  (4, 3, 5, 6), (4, 256, 0, 7), (1, 256, 0, 8)])
def test_k_split_of_very_small_batches_is_bit_identical(cuda_device, tokens, eloc, off, seed):
    # few tiles (the split is used) and, with all 256 experts local, many tiles (it is not); the full-size layer
    # has 56 K-blocks per GEMM1 tile, i.e. parts of 7 to 28 K-blocks
    dims = dataclasses.replace(syn.CONFIGS[0].dims, num_local_experts=eloc) if eloc <= 32 else dataclasses.replace(SMALL, num_local_experts=eloc)
    wl = syn.Workload(f"k{tokens}", tokens, dims, 700 + seed, local_expert_offset=off)
    inp = syn.make_inputs(wl, cuda_device)
    eng = make_engine(wl, cuda_device)
    eng.debug_set_k_split(False)
    want = eng.forward(inp).clone()
    eng.debug_set_k_split(True)
    for _ in range(3):  # the part counters of one forward must not disturb the next
        got = eng.forward(inp).clone()
    torch.cuda.synchronize()
    assert eng.status() == 0 and eng.last_launch_count() == 1
    assert torch.equal(got.view(torch.int16), want.view(torch.int16))
    run_and_compare(wl, cuda_device, inp=inp, eng=eng)
    eng.close()


# ---- row tiles of at most 32 rows inside the large-tile GEMM kernels: weights on the M side of the MMAs ------
@pytest.mark.parametrize("tokens,kw", [(100, {}), (200, {"skew": True}), (700, {}), (1111, {"skew": True}),
                                       (3000, {"local_expert_offset": 160})])
def test_short_row_tiles_are_bit_identical_to_full_row_tiles(cuda_device, tokens, kw):
    # the same forward with every row tile worked on as a full 128-row tile (hook off) and with the short ones
    # (an expert's last tile of at most 32 rows) taken the other way round, full and short tiles interleaved
    # in every CTA's work list
    wl = _wl(tokens, seed=500 + tokens, **kw)
    inp = syn.make_inputs(wl, cuda_device)
    eng = make_engine(wl, cuda_device)
    eng.debug_set_short_tiles(0)
    want = eng.forward(inp).clone()
    eng.debug_set_short_tiles(1)
    got = eng.forward(inp).clone()
    torch.cuda.synchronize()
    assert eng.status() == 0
    assert torch.equal(got.view(torch.int16), want.view(torch.int16))
    dbg = eng.debug_export(tokens, rows=False)
    counts = dbg["expert_count"].cpu().numpy()
    assert ((counts % 128 > 0) & (counts % 128 <= 32)).any(), "no short row tile in this workload"
    run_and_compare(wl, cuda_device, inp=inp, eng=eng)
    eng.close()


# ---- large-tile GEMM kernels on layers with fewer K-blocks per tile than the scale fetch runs ahead -----------
@pytest.mark.parametrize("hidden,inter,tokens,eloc,gate_first", [(256, 128, 700, 32, True), (256, 384, 300, 2, False),
                                                                 (768, 128, 90, 256, True), (1280, 640, 1000, 5, False)])
def test_large_tile_kernels_with_few_k_blocks_per_tile(cuda_device, hidden, inter, tokens, eloc, gate_first):
    # 1 to 10 K-blocks per tile against 4 pipeline stages, 8 factor slots and scales fetched 4 K-blocks ahead; one
    # CTA's list mixes short and full row tiles; w13 with the up projection first in two of the cases
    dims = syn.LayerDims(hidden=hidden, intermediate=inter, num_local_experts=eloc)
    wl = _wl(tokens, dims, seed=900 + hidden)
    inp = syn.make_inputs(wl, cuda_device)
    kw = {}
    if not gate_first:
        inp["w13"] = torch.cat([inp["w13"][:, inter:], inp["w13"][:, :inter]], 1).contiguous()
        inp["w13_scale"] = torch.cat([inp["w13_scale"][:, inter // 128:], inp["w13_scale"][:, :inter // 128]], 1).contiguous()
        kw["gate_first"] = False
    run_and_compare(wl, cuda_device, inp=inp, **kw)


# ---- both GEMMs in one launch: a GEMM2 tile waits for the GEMM1 tiles of its rows, in whatever CTA they are -----
@pytest.mark.parametrize("dims,tokens,kw", [
    (syn.LayerDims(hidden=512, intermediate=256, num_local_experts=1), 257, {}),       # fewer GEMM1 tiles than CTAs
    (syn.LayerDims(hidden=256, intermediate=128, num_local_experts=32), 300, {}),      # one column tile of GEMM1
    (syn.LayerDims(hidden=512, intermediate=1280, num_local_experts=32), 600, {}),     # GEMM2 tiles longer than GEMM1's
    (syn.LayerDims(hidden=1024, intermediate=512, num_local_experts=32), 2500, {"skew": True}),
    (syn.LayerDims(hidden=512, intermediate=256, num_local_experts=256), 2048, {}),
])
def test_one_launch_for_both_gemms(cuda_device, dims, tokens, kw):
    wl = _wl(tokens, dims, seed=1000 + tokens, **kw)
    inp = syn.make_inputs(wl, cuda_device)
    eng = make_engine(wl, cuda_device)
    want = eng.forward(inp).clone()
    for _ in range(5):  # the counters are set up anew by every forward
        got = eng.forward(inp)
    torch.cuda.synchronize()
    assert eng.last_launch_count() == 4 and eng.status() == 0
    assert torch.equal(got.view(torch.int16), want.view(torch.int16))
    run_and_compare(wl, cuda_device, inp=inp, eng=eng, sample_tokens=_sample(tokens, 256, 1))
    eng.close()


@pytest.mark.parametrize("tokens,eloc,skew", [(300, 8, False),     # at most one GEMM1 tile in a list
                                              (1200, 48, False),   # one or two
                                              (1200, 96, True),    # two and three, with short and full row tiles
                                              (1000, 256, False)])  # six and seven
def test_lists_of_gemm1_tiles_that_other_ctas_take_over(cuda_device, tokens, eloc, skew):
    # CTAs that have not started when others are through with their tiles, made certain: 1, 40 (beyond the first 32
    # entries of the table) and all but one of the CTAs never take their own lists.  The CTA that takes one over announces
    # the rows of its own and of the adopted lists, and everybody's GEMM2 tiles wait for them.
    dims = syn.LayerDims(hidden=512, intermediate=512, num_local_experts=eloc)
    wl = _wl(tokens, dims, seed=1100 + eloc, skew=skew)
    inp = syn.make_inputs(wl, cuda_device)
    eng = make_engine(wl, cuda_device)
    want = eng.forward(inp).clone()
    torch.cuda.synchronize()
    assert eng.last_launch_count() == 4 and eng.status() == 0
    sms = torch.cuda.get_device_properties(cuda_device).multi_processor_count
    for lists in (1, 40, sms - 1):
        eng.debug_set_unclaimed_lists(lists)
        for _ in range(3):
            got = eng.forward(inp)
        torch.cuda.synchronize()
        assert eng.status() == 0, lists
        assert torch.equal(got.view(torch.int16), want.view(torch.int16)), lists
    with pytest.raises(MoeFp8Error):
        eng.debug_set_unclaimed_lists(sms)
    eng.debug_set_unclaimed_lists(0)
    run_and_compare(wl, cuda_device, inp=inp, eng=eng, sample_tokens=_sample(tokens, 64, 1))
    eng.close()


@pytest.mark.parametrize("tokens", [90, 300])  # a launch per GEMM | both in one
def test_first_k_blocks_of_a_launch(cuda_device, tokens):
    # the first K-block of either issuer warp is the only one without an accumulator hand-over in front; here they are whole
    # GEMM1 tiles (two K-blocks), every CTA has one at most, and other rows lie in shared memory from the batch before
    dims = syn.LayerDims(hidden=256, intermediate=256, num_local_experts=32)
    inps = [syn.make_inputs(_wl(tokens, dims, seed=1150 + tokens + k), cuda_device) for k in range(2)]
    eng = make_engine(_wl(tokens, dims), cuda_device)
    for k, inp in enumerate(inps):
        run_and_compare(_wl(tokens, dims, seed=1150 + tokens + k), cuda_device, inp=inp, eng=eng)
    want = [eng.forward(i).clone() for i in inps]
    got = [eng.forward(inps[k % 2]).clone() for k in range(100)]
    torch.cuda.synchronize()
    assert eng.status() == 0
    assert all(torch.equal(g.view(torch.int16), want[k % 2].view(torch.int16)) for k, g in enumerate(got))
    eng.close()


def _route_round_robin(inp, tokens, active, away=0):
    # token t on eight experts in turn, of the first `active` ones and `away` experts of other ranks
    ids = torch.tensor(list(range(active)) + list(range(256 - away, 256)))
    idx = ids[(torch.arange(tokens)[:, None] * 8 + torch.arange(8)[None]) % len(ids)]
    inp["router_logits"][:] = -8.0
    inp["router_logits"].scatter_(1, idx.to(inp["router_logits"].device), 6.0)
    inp["routing_bias"][:] = 0


@pytest.mark.parametrize("active", [4, 9, 10, 16, 19, 25, 28])  # one row tile each: 16 GEMM1 and 28 GEMM2 tiles
def test_joint_launch_by_the_number_of_row_tiles(cuda_device, active):
    # fewer GEMM1 tiles than 148 CTAs (4, 9: 64 and 144, the first GEMM2 tile of every CTA dealt), one, two and three rounds of
    # them, all but a few CTAs without the last one (10: 160 tiles, 19: 304) or with it (16, 25, 28); and the same again with lists that
    # other CTAs take over
    wl = _wl(257, syn.DSV3, seed=1200 + active)
    inp = syn.make_inputs(wl, cuda_device)
    _route_round_robin(inp, 257, active, away=40 - active)
    eng = make_engine(wl, cuda_device, poison=False)
    run_and_compare(wl, cuda_device, inp=inp, eng=eng, sample_tokens=_sample(257, 24, active))
    assert eng.last_launch_count() == 4
    assert int((eng.debug_export(257, rows=False)["expert_count"] > 0).sum()) == active
    want = eng.forward(inp).clone()
    eng.debug_set_unclaimed_lists(50)
    got = eng.forward(inp)
    torch.cuda.synchronize()
    assert eng.status() == 0 and torch.equal(got.view(torch.int16), want.view(torch.int16))
    eng.close()


@pytest.mark.parametrize("hidden,inter,active", [(512, 256, 73), (512, 256, 74), (512, 256, 75),   # two and two tiles each
                                                 (256, 512, 37), (256, 512, 38), (256, 512, 148), (256, 512, 149),  # four and one
                                                 (1024, 128, 37), (1024, 128, 38), (1024, 128, 148), (1024, 128, 149)])  # one and four
def test_gemm2_tiles_dealt_and_from_the_counter(cuda_device, hidden, inter, active):
    # tiles of either GEMM on both sides of one for each of 148 CTAs: a launch per GEMM, overlapping | both GEMMs in one, and that
    # with lists that other CTAs take over
    dims = syn.LayerDims(hidden=hidden, intermediate=inter, num_local_experts=160)
    eng = make_engine(_wl(300, dims), cuda_device)
    for tokens, launches in ((100, 5), (300, 4)):
        wl = _wl(tokens, dims, seed=1250 + tokens + active)
        inp = syn.make_inputs(wl, cuda_device)
        _route_round_robin(inp, tokens, active)
        run_and_compare(wl, cuda_device, inp=inp, eng=eng, sample_tokens=_sample(tokens, 48, active), check_rows="tiles")
        assert eng.last_launch_count() == launches
        assert int((eng.debug_export(tokens, rows=False)["expert_count"] > 0).sum()) == active
        want = eng.forward(inp).clone()
        eng.debug_set_unclaimed_lists(50)
        got = [eng.forward(inp).clone() for _ in range(3)]
        torch.cuda.synchronize()
        assert eng.status() == 0 and all(torch.equal(g.view(torch.int16), want.view(torch.int16)) for g in got)
        eng.debug_set_unclaimed_lists(0)
    eng.close()


def test_two_handles_on_two_streams_share_the_gpu(cuda_device):
    # kernels whose CTAs wait for one another, from two streams at a time: a CTA may only depend on CTAs that run
    wls = [_wl(1500, seed=71), _wl(700, syn.LayerDims(hidden=1024, intermediate=512, num_local_experts=32), seed=72)]
    inps = [syn.make_inputs(w, cuda_device) for w in wls]
    engs = [make_engine(w, cuda_device) for w in wls]
    want = [e.forward(i).clone() for e, i in zip(engs, inps)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(device=cuda_device) for _ in wls]
    got = [None, None]
    for _ in range(20):
        for k in range(2):
            with torch.cuda.stream(streams[k]):
                got[k] = engs[k].forward(inps[k])
    torch.cuda.synchronize()
    for k in range(2):
        assert engs[k].status() == 0
        assert torch.equal(got[k].view(torch.int16), want[k].view(torch.int16))
        engs[k].close()


@pytest.mark.parametrize("sizes", [(9, 14), (48, 70), (12, 60), (16, 700), (75, 1500), (100, 200), (12, 150), (200, 1500)])
def test_fused_batches_on_two_streams(cuda_device, sizes):
    # the fused kernel beside another fused one, beside two GEMM launches that overlap and beside the joint one, and the latter two
    # beside each other: CTAs wait for one another, and the forwards follow each other closely (programmatic launches).  The waits give up early, so that a batch that only
    # got some of its CTAs would show as a time-out and not as a slow pass.
    wls = [_wl(t, syn.LayerDims(hidden=1024, intermediate=512, num_local_experts=32), seed=73 + t) for t in sizes]
    inps = [syn.make_inputs(w, cuda_device) for w in wls]
    engs = [make_engine(w, cuda_device) for w in wls]
    want = [e.forward(i).clone() for e, i in zip(engs, inps)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(device=cuda_device) for _ in wls]
    for e in engs:
        e.debug_set_fault(-1, 1 << 26)  # a few tens of milliseconds
    for _ in range(4):
        got = [[], []]
        for _ in range(25):
            for k in range(2):
                with torch.cuda.stream(streams[k]):
                    got[k].append(engs[k].forward(inps[k]))
        torch.cuda.synchronize()
        for k in range(2):
            assert engs[k].status() == 0
            assert all(torch.equal(g.view(torch.int16), want[k].view(torch.int16)) for g in got[k])
    for e in engs:
        e.close()


# ---- routing + counts + row tables in one launch, placement in the gather: block sizes and group splits ---------
@pytest.mark.parametrize("tokens,eloc,off", [(1, 32, 0), (7, 1, 3), (9, 64, 64), (129, 65, 20), (1023, 64, 0), (1024, 3, 5),
                                             (1025, 32, 32), (1025, 200, 56), (4999, 17, 0), (8193, 256, 0),
                                             (256, 256, 0), (257, 129, 100), (512, 128, 128), (513, 65, 0)])
def test_permutation_at_the_edges_of_its_blocks(cuda_device, tokens, eloc, off):
    # blocks of 8 tokens (up to 1024 tokens, 512 with more than 64 local experts and 256 with more than 128) and of 32, the
    # last block ragged; local expert counts on both sides of a power of two split the last block's threads into 1 to 32 groups
    dims = dataclasses.replace(syn.LayerDims(hidden=256, intermediate=128), num_local_experts=eloc)
    wl = _wl(tokens, dims, seed=40 + tokens, local_expert_offset=off)
    eng = make_engine(wl, cuda_device)
    eng.set_small_batch_fusion(False)
    run_and_compare(wl, cuda_device, eng=eng, sample_tokens=_sample(tokens, 64, tokens))
    joint = tokens > 256 and tokens * 8 * eloc // 256 <= 16384
    assert eng.last_launch_count() == (4 if joint else 5)
    eng.close()


@pytest.mark.parametrize("hidden", [256, 3840, 7424])  # 16, 240 and 464 16-byte chunks in a row
def test_gather_of_rows_whose_last_round_of_copies_is_half_a_warp(cuda_device, hidden):
    # a warp copies a row 224 chunks at a time; these leave 16 chunks, half a warp's, for the last round, in which
    # all lanes still take part in the exchange of the destination rows.  Every gathered byte and scale feeds GEMM1.
    dims = syn.LayerDims(hidden=hidden, intermediate=128, num_local_experts=64)
    for layout in (0, 1):
        wl = _wl(331, dims, seed=hidden + layout, skew=True)
        inp = syn.make_inputs(wl, cuda_device)
        if layout:
            inp["hidden_scale"] = inp["hidden_scale"].t().contiguous()
        run_and_compare(wl, cuda_device, inp=inp, hidden_scale_layout=layout)


# ---- batches of at most 80 tokens: gather, both GEMMs and the combine as one kernel; up to 16 tokens that ----
# ---- kernel also routes and permutes (every CTA for itself), and the forward is a single launch -------------
@pytest.mark.parametrize("tokens,kw", [(1, {}), (5, {}), (12, {}), (13, {}), (16, {"local_expert_offset": 64}),
                                       (17, {}), (32, {}), (23, {"skew": True}), (33, {}), (64, {"skew": True}),
                                       (80, {}), (80, {"skew": True, "local_expert_offset": 32})])
def test_fused_small_batch_kernel_is_bit_identical_to_the_separate_kernels(cuda_device, tokens, kw):
    wl = _wl(tokens, seed=80 + tokens, **kw)
    inp = syn.make_inputs(wl, cuda_device)
    eng = make_engine(wl, cuda_device)
    eng.set_small_batch_fusion(False)
    want = eng.forward(inp).clone()
    n_sep = eng.last_launch_count()
    eng.set_small_batch_fusion(True)
    got = eng.forward(inp).clone()
    torch.cuda.synchronize()
    assert eng.status() == 0
    assert eng.last_launch_count() == (1 if tokens <= 16 else 2) and n_sep == 5
    assert torch.equal(got.view(torch.int16), want.view(torch.int16))
    run_and_compare(wl, cuda_device, inp=inp, eng=eng)
    eng.close()


def test_fused_small_batch_kernel_transposed_scales_and_full_size_layer(cuda_device):
    wl = _wl(19, seed=90)
    inp = syn.make_inputs(wl, cuda_device)
    run_and_compare(wl, cuda_device, inp=dict(inp, hidden_scale=inp["hidden_scale"].t().contiguous()), hidden_scale_layout=1)
    base = syn.CONFIGS[0]
    for tokens in (1, 16, 32, 64):
        wl = syn.Workload(f"dsv3_T{tokens}_E32", tokens, base.dims, base.seed + tokens)
        inp = syn.make_inputs(wl, cuda_device)
        eng = make_engine(wl, cuda_device)
        eng.set_small_batch_fusion(False)
        want = eng.forward(inp).clone()
        eng.set_small_batch_fusion(True)
        for _ in range(3):  # counters left by one forward must not disturb the next
            got = eng.forward(inp).clone()
        torch.cuda.synchronize()
        assert eng.status() == 0
        assert torch.equal(got.view(torch.int16), want.view(torch.int16))
        run_and_compare(wl, cuda_device, inp=inp, eng=eng)
        eng.close()


@pytest.mark.parametrize("tokens,kw", [(200, {"skew": True}), (256, {}), (130, {"skew": True, "local_expert_offset": 96})])
def test_fused_kernel_with_a_raised_limit_cuts_experts_into_sub_tiles(cuda_device, tokens, kw):
    # beyond the default limit the caller may still ask for the fused kernel (up to 256 tokens): experts with
    # more than 32 rows are then worked on as several sub-tiles of 32 rows
    wl = _wl(tokens, seed=170 + tokens, **kw)
    inp = syn.make_inputs(wl, cuda_device)
    eng = make_engine(wl, cuda_device)
    want = eng.forward(inp).clone()
    assert eng.last_launch_count() == 5
    eng.set_small_batch_fusion(256)
    got = eng.forward(inp).clone()
    torch.cuda.synchronize()
    assert eng.status() == 0 and eng.last_launch_count() == 2
    assert torch.equal(got.view(torch.int16), want.view(torch.int16))
    dbg = run_and_compare(wl, cuda_device, inp=inp, eng=eng)
    eng.close()


@pytest.mark.parametrize("active", [8, 73, 74, 75, 148, 149, 200])
def test_fused_kernel_work_lists_around_full_rounds_of_ctas(cuda_device, active):
    # two GEMM1 and two GEMM2 tiles per active expert: fewer tiles than CTAs, exactly one and two per CTA, a few more
    dims = syn.LayerDims(hidden=512, intermediate=256, num_local_experts=256)
    wl = _wl(30, dims, seed=880 + active)
    inp = syn.make_inputs(wl, cuda_device)
    inp["router_logits"][:] = -8.0
    for t in range(30):
        inp["router_logits"][t, [(8 * t + j) % active for j in range(8)]] = 6.0
    eng = make_engine(wl, cuda_device)
    eng.set_small_batch_fusion(False)
    want = eng.forward(inp).clone()
    eng.set_small_batch_fusion(True)
    got = eng.forward(inp).clone()
    torch.cuda.synchronize()
    assert eng.status() == 0 and eng.last_launch_count() == 2
    assert torch.equal(got.view(torch.int16), want.view(torch.int16))
    assert int((eng.debug_export(30, rows=False)["expert_count"] > 0).sum()) == active
    eng.close()


@pytest.mark.parametrize("hidden,inter,active",
                         # two GEMM1 tiles each (2, 10, 40, 82 CTAs and none with one more), 28, 16 and 8 short GEMM2 tiles
                         [(h, 256, a) for h in (7168, 4096, 2048) for a in (75, 79, 94, 115, 148)]
                         # two GEMM2 tiles each: fewer than 148 CTAs, one, just at and above two for every CTA, of six K-blocks (all
                         # stages go out at once) and of seven
                         + [(512, i, a) for i in (768, 896) for a in (20, 74, 75, 147, 148, 149)])
def test_gemm2_tiles_of_the_fused_kernel_come_from_a_counter(cuda_device, hidden, inter, active):
    dims = syn.LayerDims(hidden=hidden, intermediate=inter, num_local_experts=160)
    wl = _wl(30, dims, seed=1300 + active)
    inp = syn.make_inputs(wl, cuda_device)
    _route_round_robin(inp, 30, active)
    eng = make_engine(wl, cuda_device, poison=False)
    eng.set_small_batch_fusion(False)
    want = eng.forward(inp).clone()
    eng.set_small_batch_fusion(True)
    for _ in range(2):
        got = eng.forward(inp).clone()
    torch.cuda.synchronize()
    assert eng.status() == 0 and eng.last_launch_count() == 2
    assert torch.equal(got.view(torch.int16), want.view(torch.int16))
    assert int((eng.debug_export(30, rows=False)["expert_count"] > 0).sum()) == active
    eng.close()


@pytest.mark.parametrize("tokens,skew,dims", [(81, False, SMALL), (81, True, SMALL), (200, True, SMALL), (256, False, SMALL),
                                              (150, False, syn.LayerDims(512, 512, num_local_experts=256)),
                                              (200, True, syn.LayerDims(512, 1024, num_local_experts=100))])
def test_two_gemm_launches_that_overlap(cuda_device, tokens, skew, dims):
    # GEMM2's launch starts while GEMM1's still runs and waits row tile by row tile; batches in a row on one handle, with
    # and without stage timing (which keeps the launches apart).  The two larger layers have lists of three and more GEMM1 tiles,
    # whose rows are announced together, and the skewed one short and full row tiles in them.
    eng = make_engine(_wl(tokens, dims), cuda_device)
    ref = make_engine(_wl(tokens, dims), cuda_device)
    ref.set_small_batch_fusion(256)
    inps = [syn.make_inputs(_wl(tokens, dims, seed=1700 + tokens + k, skew=skew), cuda_device) for k in range(3)]
    want = [ref.forward(i).clone() for i in inps]
    got = [eng.forward(inps[k % 3]).clone() for k in range(9)]
    eng.set_stage_timing(True)
    got += [eng.forward(i).clone() for i in inps]
    eng.set_stage_timing(False)
    got += [eng.forward(i).clone() for i in inps]
    torch.cuda.synchronize()
    assert eng.status() == 0 and ref.status() == 0 and eng.last_launch_count() == 5
    for k, g in enumerate(got):
        assert torch.equal(g.view(torch.int16), want[k % 3].view(torch.int16)), k
    eng.close()
    ref.close()


@pytest.mark.parametrize("hidden,inter,gate_first", [(256, 128, True), (256, 384, False), (768, 128, False)])
def test_fused_kernel_groups_take_turns_at_tiles_shorter_than_the_pipeline(cuda_device, hidden, inter, gate_first):
    # 1 to 6 K-blocks per tile against 6 stages, several tiles per CTA in both GEMMs, sub-tiles of more than 16 rows
    dims = syn.LayerDims(hidden=hidden, intermediate=inter, num_local_experts=256)
    for tokens in (14, 80):
        wl = _wl(tokens, dims, seed=1500 + hidden + inter + tokens, skew=tokens == 80)
        inp = syn.make_inputs(wl, cuda_device)
        eng = make_engine(wl, cuda_device, poison=False, gate_first=gate_first)
        eng.set_small_batch_fusion(False)
        want = eng.forward(inp).clone()
        eng.set_small_batch_fusion(True)
        got = eng.forward(inp).clone()
        torch.cuda.synchronize()
        assert eng.status() == 0 and eng.last_launch_count() == (1 if tokens <= 16 else 2)
        assert torch.equal(got.view(torch.int16), want.view(torch.int16))
        eng.close()


@pytest.mark.parametrize("hidden,inter,active", [(512, 256, 5), (1024, 128, 37), (1024, 128, 38), (256, 512, 37), (256, 512, 38)])
@pytest.mark.parametrize("tokens", [16, 17, 33, 70])
def test_fused_kernel_tiles_of_one_group_and_of_both(cuda_device, hidden, inter, active, tokens):
    # tiles for at most every CTA in both GEMMs, in GEMM1 only and in GEMM2 only, or one too many; sub-tiles of 16, 17, 32 and 1,
    # 32, 32 and 6 rows (three experts that every token goes to) beside short ones
    dims = syn.LayerDims(hidden=hidden, intermediate=inter, num_local_experts=160)
    wl = _wl(tokens, dims, seed=1550 + tokens + active)
    inp = syn.make_inputs(wl, cuda_device)
    _route_round_robin(inp, tokens, active - 3 if active > 11 else active)
    if active > 11:
        rest = torch.arange(tokens)[:, None] * 5 % (active - 3) + torch.arange(5)[None]
        idx = torch.cat([torch.arange(active - 3, active).expand(tokens, 3), rest % (active - 3)], 1)
        inp["router_logits"][:] = -8.0
        inp["router_logits"].scatter_(1, idx.to(cuda_device), 6.0)
    eng = make_engine(wl, cuda_device)
    eng.set_small_batch_fusion(False)
    want = eng.forward(inp).clone()
    eng.set_small_batch_fusion(True)
    got = [eng.forward(inp).clone() for _ in range(4)]
    torch.cuda.synchronize()
    assert eng.status() == 0 and eng.last_launch_count() == (1 if tokens <= 16 else 2)
    assert all(torch.equal(g.view(torch.int16), want.view(torch.int16)) for g in got)
    run_and_compare(wl, cuda_device, inp=inp, eng=eng, check_rows="tiles")
    eng.close()


@pytest.mark.parametrize("tokens,launches,eloc", [(16, 1, 32), (48, 2, 32), (3, 1, 256)])  # 3 tokens: K split
def test_a_wait_that_runs_out_in_the_fused_small_batch_kernel(cuda_device, tokens, launches, eloc):
    wl = _wl(tokens, dataclasses.replace(SMALL, num_local_experts=eloc), seed=43)
    inp = syn.make_inputs(wl, cuda_device)
    eng = make_engine(wl, cuda_device)
    want = eng.forward(inp).clone()
    torch.cuda.synchronize()
    assert eng.status() == 0 and eng.last_launch_count() == launches
    eng.debug_set_fault(skip_iteration=1, wait_clocks=1 << 20)
    eng.forward(inp)
    torch.cuda.synchronize()
    assert eng.status() in (1, 2, 3, 4, 5, 8), f"expected a time-out code, got {eng.status()}"
    eng.debug_set_fault(-1, 0)
    # the aborted call left its counters half counted; the calls after it alternate between the two counter
    # sets, each zeroing the other one, so all of them must be right
    for _ in range(4):
        got = eng.forward(inp).clone()
        torch.cuda.synchronize()
        assert eng.status() == 0
        assert torch.equal(got.view(torch.int16), want.view(torch.int16))
    eng.close()


def test_small_batches_of_changing_size_share_the_alternating_counters(cuda_device):
    # one handle, batch sizes on both sides of every launch scheme (one launch, routing kernel + fused kernel,
    # separate kernels) in turn: what one forward leaves in the workspace must not reach the next
    sizes = [7, 30, 3, 90, 16, 17, 1, 80, 12, 81, 9, 40]
    base = _wl(max(sizes), seed=47)
    inp = syn.make_inputs(base, cuda_device)
    eng = make_engine(base, cuda_device)
    ref = make_engine(base, cuda_device)
    ref.set_small_batch_fusion(False)
    for t in sizes:
        part = dict(inp, hidden_fp8=inp["hidden_fp8"][:t].contiguous(), hidden_scale=inp["hidden_scale"][:t].contiguous(),
                    router_logits=inp["router_logits"][:t].contiguous())
        got = eng.forward(part).clone()
        want = ref.forward(part).clone()
        torch.cuda.synchronize()
        assert eng.status() == 0 and ref.status() == 0
        assert eng.last_launch_count() == (1 if t <= 16 else 2 if t <= 80 else 5), t
        assert torch.equal(got.view(torch.int16), want.view(torch.int16)), t
    eng.close()
    ref.close()


def test_every_token_count_of_the_bench_sweep(cuda_device):
    # the token counts bench.py times on the 32-local-expert layer (the paper's three batch-size regimes), one
    # set of weights: routing and permutation on all tokens, the output on up to 48 sampled tokens each
    import bench
    base = syn.CONFIGS[1]
    ts = sorted(bench.SWEEP_TOKENS)
    big = syn.Workload("sweep", ts[-1], base.dims, base.seed)
    inp = syn.make_inputs(big, cuda_device)
    eng = make_engine(big, cuda_device, poison=False)
    for t in ts:
        wl = syn.Workload(f"dsv3_T{t}_E32", t, base.dims, base.seed)
        sub = {k: (v[:t] if k in ("hidden_fp8", "hidden_scale", "router_logits") else v) for k, v in inp.items()}
        st = run_and_compare(wl, cuda_device, inp=sub, sample_tokens=_sample(t, 48, t), check_rows=False, eng=eng)
        assert st["frac"] >= 0.995
    eng.close()


@pytest.mark.parametrize("tokens", [300, 40, 9])  # separate kernels | fused behind the routing kernel | one launch
def test_pipelined_host_entry_point_matches_device_entry_point(cuda_device, tokens):
    # five steps through moe_fp8_forward_host_async with three different batches in rotation (two staging sets
    # alternate inside the library): every step's host result equals the device-buffer forward of its batch
    wl = _wl(tokens, seed=13)
    batches = [syn.make_inputs(_wl(tokens, seed=13 + i), cuda_device) for i in range(3)]
    weights = batches[0]
    eng = make_engine(wl, cuda_device)
    want = []
    for b in batches:
        want.append(eng.forward({**weights, **{k: b[k] for k in ("hidden_fp8", "hidden_scale", "router_logits")}}).cpu())
    host_acts = [{k: b[k].cpu().pin_memory() for k in ("hidden_fp8", "hidden_scale", "router_logits")} for b in batches]
    host_outs = [torch.empty(tokens, 512, dtype=torch.bfloat16).pin_memory() for _ in range(5)]
    for i in range(5):
        eng.forward_host_async(host_acts[i % 3], weights, host_outs[i])
    eng.host_sync()
    assert eng.status() == 0
    for i in range(5):
        assert torch.equal(host_outs[i].view(torch.int16), want[i % 3].view(torch.int16)), f"step {i}"
    eng.close()


def test_a_batch_of_65536_tokens(cuda_device):
    # four times the largest benchmark batch: 528 352 padded rows, byte offsets beyond 2^32 in every row buffer
    base = syn.CONFIGS[1]
    wl = syn.Workload("dsv3_T65536_E32", 65536, base.dims, seed=65)
    st = run_and_compare(wl, cuda_device, sample_tokens=_sample(65536, 96, 65), check_rows="tiles", poison=False)
    assert st["S"] > 30000
