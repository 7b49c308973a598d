"""GPU parity, the wider cases: config 4 sampled from the plan (group ends and token-tile edges), the tensor-core kernels
at OLMoE shape in the batched-decode range and on single-expert group sizes (the kernel-level gate of Sec. 5.3), the
global-histogram grouping path, config 5 at its real size (16 OLMoE layers, teacher-forced), and guard bands around
every buffer the kernels write (the stand-in for a memory checker: no byte outside a buffer may change).
"""
import numpy as np
import pytest
import torch

from oracle import cache as ocache
from paper_2608_15383_b200 import synth

import helpers

pytestmark = pytest.mark.gpu
compare_plan = helpers.compare_plan


@pytest.fixture(scope="module")
def B():
    from paper_2608_15383_b200 import binding, build
    build.build()
    binding.lib()
    return binding


@pytest.fixture(scope="module")
def olmoe_layer(B):
    ora, bank = helpers.make_layer(synth.OLMOE, seed=2000)
    ora.max_cached = 64                                   # every expert stays dequantised (3.2 GB of host memory)
    return ora, bank


def tile_rows(cnt, bn):
    """First rows of the token tiles a group of `cnt` rows is cut into: ceil(cnt / bn) pieces of equal size rounded up
    to 16 rows (the rule of the tensor-core kernels' tile list; restated here only to CHOOSE which rows to sample)."""
    pieces = -(-cnt // bn)
    per = (-(-cnt // pieces) + 15) // 16 * 16
    return list(range(0, cnt, per))


@pytest.mark.parametrize("alpha", [0.0, 1.0])
def test_config4_prefill_olmoe_sampled_from_the_plan(B, olmoe_layer, alpha):
    """Config 4 (2048 tokens x top-8 over 64 experts, uniform and Zipf): the tokens behind the first and the last
    grouped row of every active expert and behind the rows on both sides of every token-tile edge are checked against
    the oracle, plus one row from the middle of every group."""
    ora, bank = olmoe_layer
    s = synth.OLMOE
    T = 2048
    hidden, ids, p = helpers.routed_inputs(s, T, seed=4000, alpha=alpha)
    cache = B.Cache(s, [bank], 64, max_tokens=T)
    sc = ocache.SlotCache(64, 64, 0, bytes_per_expert=cache.bytes_per_expert)
    out = cache.forward(0, hidden.cuda(), ids.cuda(), p.cuda())
    assert cache.last_path() == B.PATH_TENSOR
    compare_plan(cache, sc, ids)
    plan = cache.last_plan(0, ids.numel())
    tokens = set()
    for e in range(64):
        cnt, off = int(plan["counts"][e]), int(plan["offsets"][e])
        if cnt == 0:
            continue
        rows = {0, cnt // 2, cnt - 1}
        for n0 in tile_rows(cnt, 256)[1:]:
            rows.update((n0 - 1, n0))
        tokens.update(int(plan["perm"][off + r]) // s.top_k for r in rows)
    sample = sorted(tokens)
    assert 100 <= len(sample) <= 700                      # group ends of different experts often share a token
    y, ref = ora.forward(hidden[sample], ids[sample], p[sample])
    helpers.check_output(out[sample], y, ref, f"alpha={alpha}, {len(sample)} tokens")
    assert cache.status() == 0
    cache.close()


@pytest.mark.parametrize("T", [96, 128])
def test_small_n_tensor_core_kernels_at_olmoe_shape(B, olmoe_layer, T):
    """Batched decode with 768 and 1024 pairs at OLMoE shape: the 64-row, eight-stage tensor-core kernel shape, every
    token against the oracle."""
    ora, bank = olmoe_layer
    s = synth.OLMOE
    hidden, ids, p = helpers.routed_inputs(s, T, seed=7100 + T, alpha=1.0)
    y, ref = ora.forward(hidden, ids, p)
    cache = B.Cache(s, [bank], 64, max_tokens=T)
    cache.refuse_tensor_stream()                          # they take these calls where the device can run them
    out = cache.forward(0, hidden.cuda(), ids.cuda(), p.cuda())
    assert cache.last_path() == B.PATH_TENSOR_SMALL_N
    assert cache.last_tensor_kernels() == B.TENSOR_ROWS64
    helpers.check_output(out, y, ref, f"T={T}")
    cache.refuse_tensor_stream(False)
    out = cache.forward(0, hidden.cuda(), ids.cuda(), p.cuda())
    assert cache.last_path() == B.PATH_TENSOR_SMALL_N and cache.last_tensor_kernels() == B.TENSOR_STREAM
    helpers.check_output(out, y, ref, f"T={T}, streaming tensor-core kernels")
    assert cache.status() == 0
    cache.close()


@pytest.mark.parametrize("M", [641, 800, 1025, 1300])
def test_group_size_sweep_reaches_the_tensor_core_kernels(B, M):
    """One expert, k = 1, group sizes past the streaming kernels' range: both tensor-core kernel shapes on a single
    group with ragged tiles (641 = 10 tiles of 64 rows + 1 row; 1300 = 6 tiles of 224 rows, the last one short),
    every row against the dequantised reference (Sec. 5.3 checks group sizes against such a reference)."""
    s = synth.Shape(d_model=2048, d_ff=1024, num_experts=2, top_k=1)
    if not hasattr(test_group_size_sweep_reaches_the_tensor_core_kernels, "layer"):
        test_group_size_sweep_reaches_the_tensor_core_kernels.layer = helpers.make_layer(s, seed=77)
    ora, bank = test_group_size_sweep_reaches_the_tensor_core_kernels.layer
    hidden = synth.hidden_states(s, M, seed=900 + M)
    ids = torch.ones((M, 1), dtype=torch.int32)
    p = torch.rand((M, 1), generator=torch.Generator().manual_seed(M)) + 0.5
    y, ref = ora.forward(hidden, ids, p)
    cache = B.Cache(s, [bank], 2, max_tokens=M)
    out = cache.forward(0, hidden.cuda(), ids.cuda(), p.cuda())
    assert cache.last_path() == (B.PATH_TENSOR_SMALL_N if M <= 1024 else B.PATH_TENSOR)
    helpers.check_output(out, y, ref, f"M={M}")
    assert cache.status() == 0
    cache.close()


def test_global_histogram_grouping_path(B):
    """A key space of 8192 (256 experts, 128 slots, waves of 4) with more than 2048 pairs: grouping by global histogram
    and one CTA per key (the scheme behind the single-CTA and the chunked ones).  Plan, state and counters bit for
    bit against the oracle over several calls; output against the oracle and against the resident run."""
    s = synth.Shape(d_model=128, d_ff=128, num_experts=256, top_k=4)
    ora, bank = helpers.make_layer(s, seed=321)
    T = 600
    cache = B.Cache(s, [bank], 128, max_tokens=T, wave_cap=4)
    assert cache.n_keys == 8192
    full = B.Cache(s, [bank], s.num_experts, max_tokens=T)
    sc = ocache.SlotCache(s.num_experts, 128, 4, bytes_per_expert=cache.bytes_per_expert)
    for step in range(3):
        hidden, ids, p = helpers.routed_inputs(s, T, seed=8100 + step, alpha=0.3)
        h, i, w = hidden.cuda(), ids.cuda(), p.cuda()
        out = cache.forward(0, h, i, w)
        compare_plan(cache, sc, ids)
        ref_out = full.forward(0, h, i, w)
        assert torch.equal(out.view(torch.int16), ref_out.view(torch.int16)), step
    y, ref = ora.forward(hidden, ids, p)
    helpers.check_output(out, y, ref, "key space 8192")
    assert cache.status() == 0 and full.status() == 0
    cache.close()
    full.close()


def test_config5_real_size_teacher_forced(B):
    """Config 5 at the paper's geometry (Sec. 4.1: 16 sparse layers, 64 experts, top-8, 2048 / 1024), 16 slots, 16
    tokens, one step: per layer the plan, state and counters bit for bit against the oracle's cache model, and the
    output of sampled tokens against the oracle fed with the GPU's layer input and routing (teacher forcing)."""
    s, L, T, C = synth.OLMOE, 16, 16, 16
    layers = []
    for l in range(L):
        wg, wu, wd = synth.expert_weights(s, 6000 + l, device="cuda")
        layers.append((helpers.OracleLayer(s, wg, wu, wd), B.pack_bank(s, wg, wu, wd)))
    cache = B.Cache(s, [bank for _, bank in layers], C, max_tokens=T)
    models = [ocache.SlotCache(s.num_experts, C, 0, bytes_per_expert=cache.bytes_per_expert) for _ in range(L)]
    stack = synth.SyntheticStack(s, L, seed=41, alpha=0.5, device="cuda")
    h = synth.hidden_states(s, T, seed=4).cuda()
    waves = []
    for l in range(L):
        bias = None if stack.bias[l] is None else stack.bias[l].float().contiguous()
        ids, w = B.exmoe_route(s, h, stack.routers[l], bias)
        out = cache.forward(l, h, ids, w).clone()
        plan = compare_plan(cache, models[l], ids.cpu(), layer=l)
        waves.append(plan.n_waves)
        sample = [0, 5, 10, T - 1]                           # four tokens per layer: up to 32 experts to dequantise
        y, ref = layers[l][0].forward(h[sample].cpu(), ids[sample].cpu(), w[sample].cpu())
        helpers.check_output(out[sample], y, ref, f"layer {l}")
        layers[l][0]._deq.clear()
        h = (h.float() + out.float() + stack.draw_noise(T)[0]).to(torch.bfloat16)
    assert max(waves) >= 2 and cache.status() == 0
    assert bool(torch.isfinite(h.float()).all())
    cache.close()


def guarded_out(T, H):
    """An output tensor inside a larger one filled with a pattern; returns (view, whole, first, last)."""
    pad = 4096
    whole = torch.full((T * H + 2 * pad,), -1.0, dtype=torch.bfloat16, device="cuda")      # 0xBF80 everywhere
    return whole[pad:pad + T * H].view(T, H), whole, pad, pad + T * H


def out_guards_intact(whole, first, last):
    torch.cuda.synchronize()
    return bool((whole[:first] == -1.0).all()) and bool((whole[last:] == -1.0).all())


@pytest.mark.parametrize("case", ["pairwise", "in-CTA grouping, several waves", "streaming", "tensor small-N", "tensor large-N",
                                  "chunked grouping", "host copies", "prefetch"])
def test_no_kernel_writes_outside_its_buffers(B, case):
    """Slot memory, workspace and the output each sit between margins filled with a pattern; one call per kernel path,
    both miss paths and the prefetch; afterwards every margin byte is unchanged (and the result is still right)."""
    s = synth.MID
    if not hasattr(test_no_kernel_writes_outside_its_buffers, "layer"):
        test_no_kernel_writes_outside_its_buffers.layer = helpers.make_layer(s, seed=5)
    ora, bank = test_no_kernel_writes_outside_its_buffers.layer
    T, C, Cw, want = {"pairwise": (2, 16, 0, B.PATH_PAIR), "in-CTA grouping, several waves": (5, 6, 3, B.PATH_SMALL),
                      "streaming": (40, 6, 0, B.PATH_STREAM), "tensor small-N": (200, 6, 3, B.PATH_TENSOR_SMALL_N),
                      "tensor large-N": (300, 16, 0, B.PATH_TENSOR), "chunked grouping": (700, 6, 0, B.PATH_TENSOR),
                      "host copies": (40, 5, 2, B.PATH_STREAM), "prefetch": (3, 8, 0, None)}[case]
    if case == "chunked grouping":                           # beyond 8192 pairs: fewer are grouped together with the row copy
        T = 2100
    cache = B.Cache(s, [bank], C, max_tokens=T, wave_cap=Cw, guard_bytes=1 << 16)
    if case == "host copies":
        cache.set_miss_path(B.MISS_HOST_COPIES)
    hidden, ids, p = helpers.routed_inputs(s, T, seed=9300 + T, alpha=0.5)
    y, ref = ora.forward(hidden, ids, p)
    out, whole, first, last = guarded_out(T, s.d_model)
    if case == "prefetch":
        cache.prefetch(0, ids.cuda().reshape(-1)[:8].contiguous())
    for _ in range(2):                                       # a cold cache, then hits and LRU replacement
        cache.forward(0, hidden.cuda(), ids.cuda(), p.cuda(), out=out)
    if want is not None:
        assert cache.last_path() == want
    assert cache.guards_intact() and out_guards_intact(whole, first, last)
    helpers.check_output(out, y, ref, case)
    assert cache.status() == 0
    cache.close()


@pytest.mark.parametrize("slots, wave_cap", [(64, 0), (20, 7)])
def test_streaming_tensor_core_kernels_write_only_their_buffers(B, olmoe_layer, slots, wave_cap):
    """The same margins around the streaming tensor-core kernels, which the small shape above does not reach: one wave and several,
    with the rows of the last token in the buffers' last rows."""
    ora, bank = olmoe_layer
    s, T = synth.OLMOE, 101
    cache = B.Cache(s, [bank], slots, max_tokens=T, wave_cap=wave_cap, guard_bytes=1 << 16)
    hidden, ids, p = helpers.routed_inputs(s, T, seed=9350, alpha=1.0)
    out, whole, first, last = guarded_out(T, s.d_model)
    for _ in range(2):
        cache.forward(0, hidden.cuda(), ids.cuda(), p.cuda(), out=out)
    assert cache.last_tensor_kernels() == B.TENSOR_STREAM
    assert cache.guards_intact() and out_guards_intact(whole, first, last)
    sample = list(range(0, T, 5))
    y, ref = ora.forward(hidden[sample], ids[sample], p[sample])
    helpers.check_output(out[sample], y, ref, f"{slots} slots")
    assert cache.status() == 0
    cache.close()


def test_static_entry_point_writes_only_its_output(B):
    s = synth.MID
    ora, bank = test_no_kernel_writes_outside_its_buffers.layer if hasattr(test_no_kernel_writes_outside_its_buffers, "layer") \
        else helpers.make_layer(s, seed=5)
    T = 4
    hidden, ids, p = helpers.routed_inputs(s, T, seed=9400)
    y, ref = ora.forward(hidden, ids, p)
    out, whole, first, last = guarded_out(T, s.d_model)
    stream = torch.cuda.Stream()                             # not the default stream
    stream.wait_stream(torch.cuda.current_stream())
    B.exmoe_moe_forward_static_status()                      # the word is sticky: drop what an earlier caller left
    B.exmoe_moe_forward_static(s, bank.cuda().reshape(-1), hidden.cuda(), ids.cuda(), p.cuda(), out, stream=stream)
    stream.synchronize()
    assert out_guards_intact(whole, first, last)
    helpers.check_output(out, y, ref, "static, side stream")
    assert B.exmoe_moe_forward_static_status() == 0
    bad = ids.clone()
    bad[1, 0] = -3
    B.exmoe_moe_forward_static(s, bank.cuda().reshape(-1), hidden.cuda(), bad.cuda(), p.cuda(), out, stream=stream)
    assert B.exmoe_moe_forward_static_status() == B.EXMOE_ERR_BAD_EXPERT_ID      # reported, then cleared
    assert B.exmoe_moe_forward_static_status() == 0
    # a shape whose down kernel would need 264 KB of shared memory is refused before anything is queued
    big = synth.Shape(d_model=256, d_ff=4096, num_experts=32, top_k=32)
    with pytest.raises(B.ExmoeError) as ei:
        B.exmoe_moe_forward_static(big, bank.cuda().reshape(-1), torch.zeros((1, 256), dtype=torch.bfloat16, device="cuda"),
                                   torch.zeros((1, 32), dtype=torch.int32, device="cuda"),
                                   torch.zeros((1, 32), dtype=torch.float32, device="cuda"),
                                   torch.zeros((1, 256), dtype=torch.bfloat16, device="cuda"))
    assert ei.value.code == B.EXMOE_ERR_SHAPE


def test_zero_tokens_through_the_abi_and_host_copy_bytes(B):
    """T = 0 reaches the C entry points (no early return in the binding); the host-buffer call copies what T needs,
    not what max_tokens would."""
    s = synth.MID
    ora, bank = helpers.make_layer(s, seed=5)
    cache = B.Cache(s, [bank], s.num_experts, max_tokens=2048)
    empty_h = torch.empty((0, s.d_model), dtype=torch.bfloat16, device="cuda")
    empty_i = torch.empty((0, s.top_k), dtype=torch.int32, device="cuda")
    empty_w = torch.empty((0, s.top_k), dtype=torch.float32, device="cuda")
    assert cache.forward(0, empty_h, empty_i, empty_w).shape == (0, s.d_model)
    assert cache.forward_host(0, empty_h.cpu(), empty_i.cpu(), empty_w.cpu()).shape == (0, s.d_model)
    B.exmoe_moe_forward_static(s, bank.cuda().reshape(-1), empty_h, empty_i, empty_w, torch.empty_like(empty_h))
    hidden, ids, p = helpers.routed_inputs(s, 1, seed=9500)
    y, ref = ora.forward(hidden, ids, p)
    out = cache.forward_host(0, hidden, ids, p)
    helpers.check_output(out, y, ref, "host call, T = 1 of max_tokens = 2048")
    assert cache.last_host_copy_bytes() == s.d_model * 2 + 2 * s.top_k * 4       # 1056 bytes, not 2 MB
    assert cache.status() == 0
    cache.close()


@pytest.mark.parametrize("T", [16, 128, 2048])
def test_graph_replay_of_the_larger_paths_is_bit_identical_to_plain_launches(B, olmoe_layer, T):
    """bench.py times every leg as a CUDA-graph replay: the streaming kernels (T = 16), the 64-row tensor-core shape
    (T = 128) and the 256-row one (T = 2048, config 4) must give, replayed from a graph over two rotating input sets,
    the very bits of their plain launches (which the other tests hold to the oracle)."""
    _, bank = olmoe_layer
    s = synth.OLMOE
    cache = B.Cache(s, [bank], 64, max_tokens=T)
    cache.refuse_tensor_stream()                          # T = 128: the 64-row shape; the kernels that it stands in for are below
    inputs = [tuple(x.cuda() for x in helpers.routed_inputs(s, T, seed=8800 + T + i, alpha=0.5)) for i in range(2)]
    plain = [cache.forward(0, h, i, w).clone() for h, i, w in inputs]
    want = {16: B.PATH_STREAM, 128: B.PATH_TENSOR_SMALL_N, 2048: B.PATH_TENSOR}[T]
    assert cache.last_path() == want
    assert T == 16 or cache.last_tensor_kernels() == (B.TENSOR_ROWS64 if T == 128 else B.TENSOR_ROWS256)
    outs = [torch.zeros_like(plain[0]) for _ in inputs]
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        for (h, i, w), o in zip(inputs, outs):
            cache.forward(0, h, i, w, out=o, stream=stream)
    for rep in range(2):
        for o in outs:
            o.zero_()
        with torch.cuda.stream(stream):
            g.replay()
        stream.synchronize()
        for o, p in zip(outs, plain):
            assert torch.equal(o.view(torch.int16), p.view(torch.int16)), f"T={T} replay {rep}"
    assert cache.status() == 0
    cache.close()


@pytest.mark.parametrize("T", [100, 140])
def test_graph_replay_of_the_streaming_tensor_core_kernels(B, olmoe_layer, T):
    """The same for the streaming tensor-core kernels, on both sides of 1024 pairs: two layer calls per graph, replayed on rows
    and routing that change between the replays."""
    _, bank = olmoe_layer
    s = synth.OLMOE
    cache = B.Cache(s, [bank, bank], 64, max_tokens=T)
    inputs = [tuple(x.cuda() for x in helpers.routed_inputs(s, T, seed=8900 + T + i, alpha=0.5)) for i in range(3)]
    plain = [[cache.forward(l, *x).clone() for l in range(2)] for x in inputs]
    assert cache.last_tensor_kernels() == B.TENSOR_STREAM
    held, outs = [x.clone() for x in inputs[0]], [torch.zeros_like(plain[0][0]) for _ in range(2)]
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        for l in range(2):
            cache.forward(l, *held, out=outs[l], stream=stream)
    for i in (1, 2, 0):
        for x, y in zip(held, inputs[i]):
            x.copy_(y)
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            g.replay()
        stream.synchronize()
        for o, p in zip(outs, plain[i]):
            assert torch.equal(o.view(torch.int16), p.view(torch.int16)), i
    assert cache.status() == 0
    cache.close()


@pytest.mark.parametrize("d_model, E, k, T, slots", [
    (512, 16, 4, 161, 16),             # 644 pairs, just past the streaming kernels: segments of five pairs, the last one short
    (512, 16, 4, 300, 6),              # several waves: keys are (wave, slot)
    (2304, 4, 1, 700, 4),              # rows of more than 256 16-byte pieces (two passes of a warp); one pair per token
    (512, 16, 4, 2048, 16),            # 8192 pairs, the most that the one-launch grouping takes
    (512, 16, 4, 2049, 16)])           # ... and the first call behind it
def test_grouping_together_with_the_row_copy(B, d_model, E, k, T, slots):
    """Tensor-core calls whose pairs are grouped and whose rows are copied in one launch: plan, permutation and state bit
    for bit, every 16th token and the last one against the oracle (the repository's output tolerance)."""
    s = synth.Shape(d_model, 256, E, k)
    ora, bank = helpers.make_layer(s, seed=31 + d_model + E)
    hidden, ids, p = helpers.routed_inputs(s, T, seed=5100 + T, alpha=1.0)
    cache = B.Cache(s, [bank], slots, max_tokens=T)
    sc = ocache.SlotCache(E, slots, 0, bytes_per_expert=cache.bytes_per_expert)
    out = cache.forward(0, hidden.cuda(), ids.cuda(), p.cuda())
    assert cache.last_path() in (B.PATH_TENSOR_SMALL_N, B.PATH_TENSOR)
    compare_plan(cache, sc, ids)
    sample = list(range(0, T, 16)) + [T - 1]
    y, ref = ora.forward(hidden[sample], ids[sample], p[sample])
    helpers.check_output(out[sample], y, ref, f"{d_model} {E} {k} {T}")
    assert cache.status() == 0
    bad = ids.clone()
    bad[T // 2] = -1                                      # a token without a valid expert: zero row, the others unchanged
    out2 = cache.forward(0, hidden.cuda(), bad.cuda(), p.cuda())
    keep = torch.arange(T) != T // 2
    assert not out2[T // 2].any() and cache.status() != 0
    assert torch.equal(out2[keep].view(torch.int16), out[keep].view(torch.int16))
    cache.close()


@pytest.mark.parametrize("T", [81, 95])
def test_streaming_kernels_past_their_own_grouping(B, olmoe_layer, T):
    """648 and 760 pairs over 64 experts, fewer than 12 per expert: the streaming kernels on the grouping kernel's plan,
    every token against the oracle, and bit for bit the same from a cache with misses and several waves."""
    ora, bank = olmoe_layer
    s = synth.OLMOE
    hidden, ids, p = helpers.routed_inputs(s, T, seed=7300 + T, alpha=1.0)
    y, ref = ora.forward(hidden, ids, p)
    cache = B.Cache(s, [bank], 64, max_tokens=T)
    out = cache.forward(0, hidden.cuda(), ids.cuda(), p.cuda())
    assert cache.last_path() == B.PATH_STREAM
    compare_plan(cache, ocache.SlotCache(64, 64, 0, bytes_per_expert=cache.bytes_per_expert), ids)
    helpers.check_output(out, y, ref, f"T={T}")
    part = B.Cache(s, [bank], 24, max_tokens=T, wave_cap=10)
    out2 = part.forward(0, hidden.cuda(), ids.cuda(), p.cuda())
    assert torch.equal(out2.view(torch.int16), out.view(torch.int16))
    assert cache.status() == 0 and part.status() == 0
    cache.close(); part.close()


@pytest.mark.parametrize("E, k, T, path", [(64, 8, 80, "PATH_STREAM"), (64, 8, 81, "PATH_TENSOR_SMALL_N"), (96, 7, 110, "PATH_TENSOR_SMALL_N"),
                                           (128, 4, 300, "PATH_TENSOR")])
def test_streaming_kernels_end_at_640_pairs(B, E, k, T, path):
    """... however few rows that is per expert (but for 2048 x 1024): what they cost under skewed routing the host cannot see."""
    s = synth.Shape(256, 128, E, k)
    ora, bank = helpers.make_layer(s, seed=71 + E)
    hidden, ids, p = helpers.routed_inputs(s, T, seed=5600 + T, alpha=1.0)
    cache = B.Cache(s, [bank], E, max_tokens=T)
    out = cache.forward(0, hidden.cuda(), ids.cuda(), p.cuda())
    assert cache.last_path() == getattr(B, path) and cache.status() == 0
    y, ref = ora.forward(hidden[::9], ids[::9], p[::9])
    helpers.check_output(out[::9], y, ref, f"E={E} T={T}")
    cache.close()


@pytest.mark.parametrize("d_model, d_ff, E, k, slots, last", [
    (512, 256, 64, 4, 64, 160),        # 640 pairs
    (1024, 768, 24, 4, 24, 84),        # 14 rows per expert (288 weight tiles: more than SMs)
    (512, 256, 16, 4, 16, 112),        # 28 rows per expert (64 weight tiles)
    (2816, 256, 6, 6, 6, 28),          # 22 blocks do not split into four ranges: 28 rows per expert come first
    (1664, 640, 32, 4, 32, 48),        # 13 and 5 blocks: 192 pairs
    (1664, 640, 32, 4, 8, 48)])        # ... and the same with misses
def test_where_the_streaming_kernels_end(B, d_model, d_ff, E, k, slots, last):
    """The last token count that goes to the streaming kernels and the first that does not."""
    s = synth.Shape(d_model, d_ff, E, k)
    ora, bank = helpers.make_layer(s, seed=81 + d_model)
    cache = B.Cache(s, [bank], slots, max_tokens=last + 1)
    for T, path in ((last, B.PATH_STREAM), (last + 1, B.PATH_TENSOR_SMALL_N)):
        hidden, ids, p = helpers.routed_inputs(s, T, seed=5700 + T, alpha=0.5)
        out = cache.forward(0, hidden.cuda(), ids.cuda(), p.cuda())
        assert cache.last_path() == path and cache.status() == 0
        y, ref = ora.forward(hidden[::17], ids[::17], p[::17])
        helpers.check_output(out[::17], y, ref, f"T={T}")
    cache.close()


@pytest.mark.parametrize("E, k, T", [
    (16, 5, 5),                        # 25 pairs: the smallest streaming call
    (128, 4, 160),                     # the most experts and pairs that the streaming kernels group themselves
    (132, 4, 160),                     # ... and the first size that takes the grouping kernel's plan
    (16, 3, 43)])                      # groups of eight, nine and more rows: remainders of the eight-row passes
def test_edges_of_the_streaming_kernels_own_grouping(B, E, k, T):
    s = synth.Shape(256, 128, E, k)
    ora, bank = helpers.make_layer(s, seed=41 + E + k)
    hidden, ids, p = helpers.routed_inputs(s, T, seed=5300 + T + E, alpha=0.3)
    y, ref = ora.forward(hidden, ids, p)
    cache = B.Cache(s, [bank], E, max_tokens=T)
    out = cache.forward(0, hidden.cuda(), ids.cuda(), p.cuda())
    assert cache.last_path() == B.PATH_STREAM
    compare_plan(cache, ocache.SlotCache(E, E, 0, bytes_per_expert=cache.bytes_per_expert), ids)
    helpers.check_output(out, y, ref, f"E={E} k={k} T={T}")
    assert cache.status() == 0
    cache.close()


@pytest.mark.parametrize("E, wave_cap, k, T", [(16, 8, 4, 8), (16, 8, 4, 16), (16, 4, 2, 200), (64, 32, 1, 25), (16, 0, 4, 16)])
def test_ids_beyond_the_experts_in_a_larger_key_space(B, E, wave_cap, k, T):
    """Every expert resident and a wave_cap below the number of experts: the key space (ceil(E / wave_cap) * E) is larger
    than the expert count, and ids E .. keys - 1 are as invalid as any other id out of range: sticky status, no
    contribution, the other tokens' bits unchanged.  Layer 0 of a cache of several layers: the slots such an id would
    name lie inside the slot memory."""
    s = synth.Shape(256, 128, E, k)
    ora, bank = helpers.make_layer(s, seed=61 + E)
    hidden, ids, p = helpers.routed_inputs(s, T, seed=5500 + T, alpha=0.3)
    cache = B.Cache(s, [bank] * 5, E, max_tokens=T, wave_cap=wave_cap)
    clean = cache.forward(0, hidden.cuda(), ids.cuda(), p.cuda())
    assert cache.last_path() == B.PATH_STREAM and cache.status() == 0
    y, ref = ora.forward(hidden, ids, p)
    helpers.check_output(clean, y, ref, "clean")
    bad = ids.clone()
    bad[1], bad[T - 2, 0], bad[T // 2, k - 1] = E, -1, 2 * E - 1
    out = cache.forward(0, hidden.cuda(), bad.cuda(), p.cuda())
    assert cache.status() == B.EXMOE_ERR_BAD_EXPERT_ID
    hit = torch.zeros(T, dtype=torch.bool)
    hit[[1, T // 2, T - 2]] = True
    assert torch.equal(out[~hit].view(torch.int16), clean[~hit].view(torch.int16))
    assert not out[1].any()
    kept = torch.where((bad >= 0) & (bad < E), bad, torch.full_like(bad, -1))
    y, ref = ora.forward(hidden, kept, p)
    helpers.check_output(out, y, ref, "invalid ids add nothing")
    compare_plan(cache, ocache.SlotCache(E, E, wave_cap, bytes_per_expert=cache.bytes_per_expert), kept)
    cache.close()


@pytest.mark.parametrize("T", [1, 4, 40])
def test_activation_scaling_over_magnitudes(B, T):
    """The decode and streaming kernels scale every 128-wide block of a row into FP16 by a power of two: rows of 1e-6 to
    1e6, a row with one block of zeros and rows with one element 4096 times the others keep the repository's tolerance,
    each row by itself (an element 2^-12 of its block's largest still has all eight of its bits: FP16 reaches 2^-24
    below 1, scaled blocks start at 2^15)."""
    s = synth.MID
    ora, bank = helpers.make_layer(s, seed=55)
    base, ids, p = helpers.routed_inputs(s, T, seed=5400 + T, alpha=0.5)
    cache = B.Cache(s, [bank], s.num_experts, max_tokens=T)
    for what in (1e-6, 1e-3, 1e3, 1e6, "zero block", "outlier"):
        hidden = base.clone()
        if what == "zero block":
            hidden[:, 128:256] = 0
        elif what == "outlier":
            hidden[:, 77] = 4096.0
        else:
            hidden = (hidden.float() * what).to(torch.bfloat16)
        y, ref = ora.forward(hidden, ids, p)
        out = cache.forward(0, hidden.cuda(), ids.cuda(), p.cuda())
        for t in range(0, T, 7):
            helpers.check_output(out[t:t + 1], y[t:t + 1], ref[t:t + 1], f"T={T} row {t} {what}")
    assert cache.status() == 0
    cache.close()


@pytest.mark.parametrize("T", [1, 2, 3])
def test_largest_panels_of_the_bulk_down_kernel(B, T):
    """Seven selected experts of eleven blocks: the shape that fills the shared memory of the by-token down kernel."""
    s = synth.Shape(1024, 1408, 12, 7)
    ora, bank = helpers.make_layer(s, seed=91)
    hidden, ids, p = helpers.routed_inputs(s, T, seed=5800 + T, alpha=0.5)
    cache = B.Cache(s, [bank], 12, max_tokens=T)
    out = cache.forward(0, hidden.cuda(), ids.cuda(), p.cuda())
    y, ref = ora.forward(hidden, ids, p)
    helpers.check_output(out, y, ref, f"T={T}")
    assert cache.last_path() == B.PATH_PAIR and cache.status() == 0
    cache.close()


@pytest.mark.parametrize("T", [3, 12, 60, 300])
def test_reading_the_plan_leaves_the_status_alone(B, T):
    """One invalid id raises the sticky status once: reading the plan afterwards (which some calls form only then) does not
    raise it again."""
    s = synth.MID
    _, bank = helpers.make_layer(s, seed=95)
    hidden, ids, p = helpers.routed_inputs(s, T, seed=5900 + T)
    ids[T // 2, 1] = -3
    cache = B.Cache(s, [bank], s.num_experts, max_tokens=T)
    cache.forward(0, hidden.cuda(), ids.cuda(), p.cuda())
    assert cache.status() == B.EXMOE_ERR_BAD_EXPERT_ID
    assert cache.last_plan(0, ids.numel())["counts"].sum() == T * s.top_k - 1
    assert cache.status() == 0
    cache.close()


def test_streaming_tensor_core_kernels_at_tile_edges(B):
    """Groups of 1 to 129 rows (tiles of 64, their remainders and 16-row steps) on odd numbers of K blocks (17 and 11) and of
    weight tiles (17): the first and last rows of every token tile against the oracle, and the same bits in waves of 20 experts."""
    s = synth.Shape(d_model=2176, d_ff=1408, num_experts=48, top_k=1)
    ora, bank = helpers.make_layer(s, seed=4100)
    sizes = [1, 15, 16, 17, 31, 32, 33, 47, 48, 49, 63, 64, 65, 80, 127, 128, 129, 2]
    ids = torch.tensor([[(5 * e + 3) % 48] for e, n in enumerate(sizes) for _ in range(n)], dtype=torch.int32)
    T = ids.shape[0]
    ids = ids[torch.randperm(T, generator=torch.Generator().manual_seed(1))].contiguous()
    hidden = synth.hidden_states(s, T, seed=4200)
    p = torch.rand((T, 1), generator=torch.Generator().manual_seed(2)) + 0.5
    cache = B.Cache(s, [bank], 48, max_tokens=T)
    out = cache.forward(0, hidden.cuda(), ids.cuda(), p.cuda())
    assert cache.last_path() == B.PATH_TENSOR_SMALL_N and cache.status() == 0
    assert cache.last_tensor_kernels() == B.TENSOR_STREAM
    sample = set()
    for e in range(48):
        rows = (ids[:, 0] == e).nonzero()[:, 0].tolist()
        for n0 in tile_rows(len(rows), 64) if rows else []:
            sample.update(rows[i] for i in (n0 - 1, n0, len(rows) - 1) if i >= 0)
    sample = sorted(sample)
    y, ref = ora.forward(hidden[sample], ids[sample], p[sample])
    helpers.check_output(out[sample], y, ref, f"{len(sample)} tokens")
    cache.close()
    part = B.Cache(s, [bank], 20, max_tokens=T)
    again = part.forward(0, hidden.cuda(), ids.cuda(), p.cuda())
    assert torch.equal(out.view(torch.int16), again.view(torch.int16)) and part.status() == 0
    part.close()
    for miss in (B.MISS_DEVICE_FETCH, B.MISS_HOST_COPIES):         # 18 experts fit 20 slots: several waves need a smaller cap
        part = B.Cache(s, [bank], 20, max_tokens=T, wave_cap=7)
        part.set_miss_path(miss)
        again = part.forward(0, hidden.cuda(), ids.cuda(), p.cuda())
        assert part.last_tensor_kernels() == B.TENSOR_STREAM and part.last_plan(0, T)["n_waves"] == 3
        assert torch.equal(out.view(torch.int16), again.view(torch.int16)) and part.status() == 0
        part.close()


def test_streaming_tensor_core_kernels_with_more_tiles_than_they_list(B):
    """A CTA keeps the first 128 entries of the tile list in shared memory and reads the rest past L1: 160 experts with rows."""
    s = synth.Shape(d_model=2048, d_ff=512, num_experts=160, top_k=1)
    ora, bank = helpers.make_layer(s, seed=4500)
    T = 900
    ids = (torch.arange(T, dtype=torch.int32) * 7 % 160)[torch.randperm(T, generator=torch.Generator().manual_seed(3))].view(T, 1).contiguous()
    hidden = synth.hidden_states(s, T, seed=4510)
    p = torch.rand((T, 1), generator=torch.Generator().manual_seed(4)) + 0.5
    cache = B.Cache(s, [bank], 160, max_tokens=T)
    out = cache.forward(0, hidden.cuda(), ids.cuda(), p.cuda())
    assert cache.last_tensor_kernels() == B.TENSOR_STREAM and (cache.last_plan(0, T)["counts"] > 0).sum() == 160
    sample = [int((ids[:, 0] == e).nonzero()[0]) for e in range(160)]
    y, ref = ora.forward(hidden[sample], ids[sample], p[sample])
    helpers.check_output(out[sample], y, ref, "a row of every expert")
    assert cache.status() == 0
    cache.close()


@pytest.mark.parametrize("slots", [64, 20])
def test_streaming_tensor_core_kernels_with_invalid_ids(B, olmoe_layer, slots):
    """Pairs with an id outside the experts add nothing and are reported; a call without any valid id gives zeros, and the next
    good call is right again."""
    ora, bank = olmoe_layer
    s, T = synth.OLMOE, 100
    hidden, ids, p = helpers.routed_inputs(s, T, seed=4600, alpha=0.5)
    bad = ids.clone()
    bad[::3, 2], bad[1::7, 5], bad[50] = -1, 64, 1 << 30
    cache = B.Cache(s, [bank], slots, max_tokens=T)
    sample = list(range(0, T, 10)) + [1, 49, 51, 99]
    for what in (bad, torch.full_like(ids, -7), ids):
        out = cache.forward(0, hidden.cuda(), what.cuda(), p.cuda())
        assert cache.last_tensor_kernels() == B.TENSOR_STREAM
        assert cache.status() == (0 if what is ids else B.EXMOE_ERR_BAD_EXPERT_ID)
        y, ref = ora.forward(hidden[sample], what[sample], p[sample])
        if (what == -7).all():
            assert not out.any()
        else:
            helpers.check_output(out[sample], y, ref, "ids")
            assert not (what is bad and out[50].any())
    cache.close()


@pytest.mark.parametrize("slots", [16, 6])
def test_chunked_grouping_after_a_call_with_an_invalid_id(B, slots):
    """More than 8192 pairs: the arrival counter and the bad-id word of the chunked grouping are ready again for the next call, and
    neither keeps what an earlier call found, with the experts resident or not."""
    s, T = synth.MID, 2100
    _, bank = helpers.make_layer(s, seed=5)
    hidden, ids, p = (x.cuda() for x in helpers.routed_inputs(s, T, seed=4700, alpha=0.5))
    bad = ids.clone()
    bad[T - 1, 3] = 16
    fresh = B.Cache(s, [bank], slots, max_tokens=T)
    good = fresh.forward(0, hidden, ids, p)
    cache = B.Cache(s, [bank], slots, max_tokens=T)
    for what in (bad, ids, bad, bad, ids):
        out = cache.forward(0, hidden, what, p)
        assert cache.status() == (0 if what is ids else B.EXMOE_ERR_BAD_EXPERT_ID)
        plan = cache.last_plan(0, ids.numel())
        assert plan["counts"].sum() == ids.numel() - (what is bad)
        assert torch.equal(out[:-1].view(torch.int16), good[:-1].view(torch.int16))
        assert torch.equal(out[-1].view(torch.int16), good[-1].view(torch.int16)) == (what is ids)
    fresh.close()
    cache.close()


@pytest.mark.parametrize("T", [96, 140])
def test_device_that_cannot_run_the_streaming_tensor_core_kernels(B, olmoe_layer, T):
    """Where the device refuses these kernels their shared memory or registers, the other tensor-core kernels take the call
    (with the rows in their own order), on both sides of 1024 pairs; nothing is combined from an earlier call's buffers."""
    ora, bank = olmoe_layer
    s = synth.OLMOE
    cache = B.Cache(s, [bank], 64, max_tokens=T)
    hidden, ids, p = helpers.routed_inputs(s, T, seed=7600 + T, alpha=0.5)
    first = cache.forward(0, hidden.cuda(), ids.cuda(), p.cuda()).clone()
    assert cache.last_tensor_kernels() == B.TENSOR_STREAM
    cache.refuse_tensor_stream()
    hidden = hidden.flip(0).contiguous()                 # other rows than those that the buffers hold
    out = cache.forward(0, hidden.cuda(), ids.cuda(), p.cuda())
    assert cache.last_tensor_kernels() == (B.TENSOR_ROWS64 if T * s.top_k <= 1024 else B.TENSOR_ROWS256)
    y, ref = ora.forward(hidden, ids, p)
    helpers.check_output(out, y, ref, f"T={T}, refused")
    cache.refuse_tensor_stream(False)
    out = cache.forward(0, hidden.flip(0).contiguous().cuda(), ids.cuda(), p.cuda())
    assert cache.last_tensor_kernels() == B.TENSOR_STREAM and torch.equal(out.view(torch.int16), first.view(torch.int16))
    assert cache.status() == 0
    cache.close()


@pytest.mark.parametrize("shape, T, kind", [
    (synth.OLMOE, 96, "STREAM"),                                                 # the first call behind the streaming kernels
    (synth.OLMOE, 128, "STREAM"), (synth.OLMOE, 129, "STREAM"), (synth.OLMOE, 144, "STREAM"), (synth.OLMOE, 145, "ROWS256"),
    (synth.Shape(2048, 1408, 60, 4), 256, "STREAM"), (synth.Shape(2048, 1408, 60, 4), 257, "ROWS256"),
    (synth.Shape(2560, 1280, 40, 4), 240, "STREAM"), (synth.Shape(2560, 1280, 40, 4), 241, "ROWS64"),     # 24 rows per expert, one more pair each
    (synth.Shape(1920, 1408, 60, 4), 200, "ROWS64"),                             # d_model
    (synth.Shape(2048, 640, 92, 4), 200, "ROWS64"), (synth.Shape(2048, 640, 93, 4), 200, "STREAM")])       # 99.5 and 100.5 blocks per SM
def test_range_of_the_streaming_tensor_core_kernels(B, shape, T, kind):
    """Which tensor-core kernels take a call, at the edges of the rule; rounding apart, both give the same rows."""
    bank = B.pack_bank(shape, *synth.expert_weights(shape, 4300, device="cuda"))
    cache = B.Cache(shape, [bank], shape.num_experts, max_tokens=T)
    hidden, ids, p = (x.cuda() for x in helpers.routed_inputs(shape, T, seed=4310 + T, alpha=1.0))
    out = cache.forward(0, hidden, ids, p).float()
    assert cache.last_tensor_kernels() == getattr(B, "TENSOR_" + kind)
    cache.refuse_tensor_stream()
    other = cache.forward(0, hidden, ids, p).float()
    assert cache.last_tensor_kernels() != B.TENSOR_STREAM
    assert torch.linalg.norm(out - other) <= 2 * helpers.REL_FRO * torch.linalg.norm(other)      # each within REL_FRO of the oracle
    assert cache.status() == 0
    cache.close()


def test_streaming_tensor_core_kernels_with_large_activations(B):
    """Activations up to binary32's end in one block of 128: the block's sum of code x activation must not overflow where the
    layer's own values do not (up values near 1e37, gates near 1, outputs near 1e36)."""
    s = synth.Shape(d_model=2048, d_ff=1024, num_experts=64, top_k=8)
    wg, wu, wd = synth.expert_weights(s, 4400)
    wg[:, :, 128:] = 0                                   # gates read the first block, up projections the second
    wu[:, :, :128] = 0
    wu[:, :, 256:] = 0
    ora, bank = helpers.OracleLayer(s, wg, wu, wd), B.pack_bank(s, wg, wu, wd)
    T = 100
    hidden, ids, p = helpers.routed_inputs(s, T, seed=4410)
    hidden[:, 128:256] = (hidden[:, 128:256].float().clamp(-3, 3) * 1e38).to(torch.bfloat16)
    cache = B.Cache(s, [bank], 64, max_tokens=T)
    out = cache.forward(0, hidden.cuda(), ids.cuda(), p.cuda())
    assert cache.last_tensor_kernels() == B.TENSOR_STREAM
    sample = list(range(0, T, 9))
    y, ref = ora.forward(hidden[sample], ids[sample], p[sample])
    assert 1e35 < abs(ref).max() < 3e38
    helpers.check_output(out[sample], y, ref, "activations of 3e38")
    assert cache.status() == 0
    cache.close()


@pytest.mark.parametrize("k, T", [(1, 300), (2, 300), (3, 61), (3, 300), (5, 256), (5, 257), (8, 256), (8, 257), (11, 130), (11, 300)])
def test_combine_with_its_rows_requested_ahead(B, k, T):
    """Two, four and eight rows requested together, by top_k and on both sides of 131,072 threads (256 tokens of d_model 2048), where
    top_k is less than that, equal, and no multiple; some pairs without a valid id."""
    s = synth.Shape(d_model=2048, d_ff=128, num_experts=16, top_k=k)
    ora, bank = helpers.make_layer(s, seed=4800 + k)
    hidden, ids, p = helpers.routed_inputs(s, T, seed=4810 + T)
    ids[T // 2, k - 1] = -1
    ids[T - 1, 0] = 16
    cache = B.Cache(s, [bank], 16, max_tokens=T)
    out = cache.forward(0, hidden.cuda(), ids.cuda(), p.cuda())
    sample = sorted({0, 1, T // 2, T // 2 + 1, T - 2, T - 1} | set(range(0, T, 37)))
    y, ref = ora.forward(hidden[sample], ids[sample], p[sample])
    helpers.check_output(out[sample], y, ref, f"top-{k}, {T} tokens")
    assert cache.status() == B.EXMOE_ERR_BAD_EXPERT_ID
    cache.close()
