"""GPU parity of the fused router (Eq. 1) against the oracle router, through the C ABI.

The top-k choice is an integer decided by floating point: the kernel decides in binary32 (its own precision),
the oracle in binary64.  So the comparison is: identical ids wherever the oracle's logits separate the experts
by more than the binary32 rounding of a 2048-term sum; where the kernel's choice differs, the two experts must
be such a near-tie in the oracle (the choice is then valid either way); weights within binary32 rounding.
"""
import numpy as np
import pytest
import torch

from oracle import router as orouter
from paper_2608_15383_b200 import synth

import helpers

pytestmark = pytest.mark.gpu

NEAR_TIE = 2e-5          # logit gap below which binary32 and binary64 may order two experts differently


@pytest.fixture(scope="module")
def B():
    from paper_2608_15383_b200 import binding, build
    build.build()
    binding.lib()
    return binding


def check(shape, hidden, w_router, bias, ids_gpu, w_gpu):
    ids_ref, p_ref, z = orouter.route(hidden.float().numpy(), w_router.float().numpy(), shape.top_k,
                                      None if bias is None else bias.double().numpy())
    ids_gpu, w_gpu = ids_gpu.cpu().numpy(), w_gpu.cpu().numpy()
    assert ids_gpu.dtype == np.int32 and ids_gpu.shape == ids_ref.shape
    n_diff = 0
    for t in range(ids_ref.shape[0]):
        assert len(set(ids_gpu[t].tolist())) == shape.top_k                      # k distinct, valid experts
        assert ((ids_gpu[t] >= 0) & (ids_gpu[t] < shape.num_experts)).all()
        full = orouter.softmax(z[t])
        np.testing.assert_allclose(w_gpu[t], full[ids_gpu[t]], rtol=2e-5, atol=1e-9)   # weights of what it chose
        assert np.all(np.diff(w_gpu[t]) <= 1e-9)                                 # descending
        if np.array_equal(ids_gpu[t], ids_ref[t]):
            continue
        n_diff += 1
        for j in range(shape.top_k):                                             # any difference is a near-tie
            if ids_gpu[t, j] != ids_ref[t, j]:
                assert abs(z[t, ids_gpu[t, j]] - z[t, ids_ref[t, j]]) < NEAR_TIE, (t, j)
    return n_diff


@pytest.mark.parametrize("shape,T,alpha", [(synth.TINY, 16, 0.0), (synth.MID, 33, 1.0), (synth.OLMOE, 1, 0.0),
                                           (synth.OLMOE, 64, 1.0), (synth.OLMOE, 300, 0.5)])
def test_router_matches_oracle(B, shape, T, alpha):
    hidden = synth.hidden_states(shape, T, seed=11 + T)
    w_router = synth.router_weights(shape, seed=5)
    bias = synth.zipf_bias(shape.num_experts, alpha, seed=9) if alpha else None
    ids, w = B.exmoe_route(shape, hidden.cuda(), w_router.cuda(), None if bias is None else bias.cuda())
    torch.cuda.synchronize()
    n_diff = check(shape, hidden, w_router, bias, ids, w)
    assert n_diff <= max(1, T // 50)                      # near-ties are rare with random inputs
    # the harness router (torch, binary32) makes the same choices up to the same near-ties
    ids_t, w_t = helpers.route(hidden.cuda(), w_router.cuda(), shape.top_k, None if bias is None else bias.cuda())
    same = (ids_t == ids).all(dim=1).float().mean().item()
    assert same >= 0.95


def test_router_ties_and_edge_cases(B):
    shape = synth.Shape(d_model=128, d_ff=128, num_experts=8, top_k=3)
    w_router = torch.zeros((8, 128), dtype=torch.bfloat16)
    w_router[2, 0] = w_router[5, 0] = 1.0                 # experts 2 and 5 tie at the top, the rest tie at zero
    hidden = torch.zeros((2, 128), dtype=torch.bfloat16)
    hidden[0, 0] = 3.0
    ids, w = B.exmoe_route(shape, hidden.cuda(), w_router.cuda())
    assert ids[0].tolist() == [2, 5, 0]                   # ties to the lower id
    assert ids[1].tolist() == [0, 1, 2]                   # all logits equal
    np.testing.assert_allclose(w[1].cpu().numpy(), [1 / 8] * 3, rtol=1e-6)
    ids_ref, p_ref, _ = orouter.route(hidden.float().numpy(), w_router.float().numpy(), 3)
    assert np.array_equal(ids.cpu().numpy(), ids_ref)
    np.testing.assert_allclose(w.cpu().numpy(), p_ref, rtol=1e-6)
    # T = 0 is a no-op; bad shapes are refused
    B.exmoe_route(shape, torch.empty((0, 128), dtype=torch.bfloat16, device="cuda"), w_router.cuda())
    with pytest.raises(B.ExmoeError) as ei:
        B.exmoe_route(synth.Shape(d_model=100, d_ff=128, num_experts=8, top_k=3), hidden.cuda(), w_router.cuda())
    assert ei.value.code == B.EXMOE_ERR_SHAPE


def test_router_feeds_the_layer(B):
    """Router output goes straight into exmoe_moe_forward: the layer result equals the one on the harness router's
    ids wherever the two routers agree (they do on these inputs)."""
    import helpers
    shape = synth.MID
    ora, bank = helpers.make_layer(shape, seed=77)
    hidden = synth.hidden_states(shape, 12, seed=3)
    w_router = synth.router_weights(shape, seed=4)
    ids, w = B.exmoe_route(shape, hidden.cuda(), w_router.cuda())
    cache = B.Cache(shape, [bank], shape.num_experts, max_tokens=16)
    out = cache.forward(0, hidden.cuda(), ids, w)
    y, ref = ora.forward(hidden, ids.cpu(), w.cpu())
    helpers.check_output(out, y, ref, "router-fed layer")
    cache.close()


@pytest.mark.parametrize("shape,T", [(synth.OLMOE, 47), (synth.OLMOE, 48), (synth.OLMOE, 51), (synth.OLMOE, 223), (synth.OLMOE, 225),
                                     (synth.OLMOE, 2303), (synth.OLMOE, 2337), (synth.Shape(1280, 128, 72, 5), 300),
                                     (synth.Shape(1280, 128, 72, 5), 2310), (synth.Shape(128, 128, 3, 2), 240),
                                     (synth.Shape(512, 128, 16, 4), 896), (synth.Shape(512, 128, 16, 4), 4000),
                                     (synth.Shape(512, 128, 16, 4), 191), (synth.Shape(512, 128, 16, 4), 895),
                                     (synth.Shape(2048, 128, 32, 8), 599),
                                     (synth.Shape(256, 128, 8, 2), 49), (synth.Shape(256, 128, 8, 2), 1536), (synth.Shape(1000, 128, 20, 3), 300),
                                     (synth.Shape(1024, 128, 256, 8), 130), (synth.Shape(1024, 128, 256, 8), 515), (synth.Shape(8192, 128, 64, 8), 530),
                                     (synth.Shape(256, 128, 132, 4), 2050), (synth.Shape(512, 128, 1030, 3), 50)])
def test_choice_does_not_depend_on_the_batch_size(B, shape, T):
    """Every form of the kernel (one or four tokens per cluster, tensor cores with 16 or 32 tokens per CTA; last tiles
    partly filled, an expert count that is no multiple of 64) picks the experts that one token at a time picks.  Near-ties
    are planted: rows of the router matrix that differ from another in one element by one BF16 ulp, and equal rows.
    Weights agree to binary32 rounding: logits of a few units off by 1e-6 at most, so 2e-5 relative as in `check`."""
    hidden = synth.hidden_states(shape, T, seed=3).cuda()
    w = synth.router_weights(shape, seed=4)
    for e in range(1, shape.num_experts, 3):
        w[e] = w[e - 1]
        if e % 2:
            w[e, e % shape.d_model] *= 1.0 + 2.0 ** -7
    w = w.cuda()
    ids, p = B.exmoe_route(shape, hidden, w)
    for t0 in range(0, T, 40):                            # 40 tokens: the one-token-per-cluster form
        i1, p1 = B.exmoe_route(shape, hidden[t0:t0 + 40].contiguous(), w)
        assert torch.equal(ids[t0:t0 + 40], i1)
        torch.testing.assert_close(p[t0:t0 + 40], p1, rtol=2e-5, atol=1e-9)


@pytest.mark.parametrize("T", [192, 193, 197])
def test_choice_where_the_tensor_core_form_begins(B, T):
    test_choice_does_not_depend_on_the_batch_size(B, synth.OLMOE, T)


@pytest.mark.parametrize("T", [223, 224])
def test_choice_where_the_tensor_core_form_begins_for_short_rows(B, T):
    test_choice_does_not_depend_on_the_batch_size(B, synth.Shape(512, 128, 48, 8), T)


@pytest.mark.parametrize("d_model, E, k", [(2048, 64, 8), (512, 16, 4), (4096, 96, 8), (128, 8, 2)])
@pytest.mark.parametrize("kind", ["normal", "positive"])
def test_weights_of_the_tensor_core_form_are_no_further_off(B, d_model, E, k, kind):
    """Against 64 bits, on the ids of the call: the mixture weights of a batch that takes the tensor cores are no further
    off than those of the same tokens in calls of 40 (binary32 sums).  1.1: the ratio of two root mean squares over some
    thousand errors each moves by a few per cent from seed to seed."""
    s = synth.Shape(d_model, 128, E, k)
    T = 2400
    hidden, w = synth.hidden_states(s, T, seed=11).cuda(), synth.router_weights(s, seed=12).cuda()
    if kind == "positive":
        hidden, w = hidden.abs(), w.abs() * 0.05
    p = torch.softmax(hidden.double() @ w.double().T, dim=1)

    def rms(ids, wt):
        ref = torch.gather(p, 1, ids.long())
        return ((wt.double() - ref) / ref).pow(2).mean().sqrt().item()

    parts = [B.exmoe_route(s, hidden[t:t + 40].contiguous(), w) for t in range(0, T, 40)]
    small = rms(torch.cat([x[0] for x in parts]), torch.cat([x[1] for x in parts]))
    for n in (400, T):                                    # 16 and 32 experts per CTA
        calls = [B.exmoe_route(s, hidden[t:t + n].contiguous(), w) for t in range(0, T, n)]
        large = rms(torch.cat([x[0] for x in calls]), torch.cat([x[1] for x in calls]))
        assert large <= 1.1 * small, (n, large, small)


def test_near_ties_in_rows_of_one_sign(B):
    """Rows whose products all have one sign, the largest in front: where sums in one accumulator lose most.  Near-ties as
    in test_choice_does_not_depend_on_the_batch_size, in the tail of the rows."""
    s = synth.Shape(4096, 128, 64, 8)
    hidden, w = synth.hidden_states(s, 320, seed=5).abs(), synth.router_weights(s, seed=6).abs() * 0.02
    hidden[:, :64] *= 64
    w[:, :64] *= 64
    for e in range(1, 64, 2):
        w[e] = w[e - 1]
        w[e, 100 + e] *= 1.0 + 2.0 ** -7
        w[e, 2000 + 16 * e:2008 + 16 * e] *= 1.0 + 2.0 ** -7
    hidden, w = hidden.cuda(), w.cuda()
    ids, p = B.exmoe_route(s, hidden, w)
    for t in range(0, 320, 40):
        i1, p1 = B.exmoe_route(s, hidden[t:t + 40].contiguous(), w)
        assert torch.equal(ids[t:t + 40], i1)
        torch.testing.assert_close(p[t:t + 40], p1, rtol=2e-5, atol=1e-9)


@pytest.mark.parametrize("what", ["small hidden states", "zero hidden states", "fewer than k unmasked", "masked with -inf", "all but one far below",
                                  "subnormal probabilities", "large logits"])
def test_choice_where_probabilities_cannot_tell(B, what):
    """Logits that differ and share a binary32 probability (closer than expf resolves, or so far below the largest that the
    probabilities are subnormal or zero) are ordered by id in every form: a batch that takes the tensor cores chooses what
    calls of 40 tokens choose."""
    s = synth.OLMOE
    E, k, T = s.num_experts, s.top_k, 400
    hidden, w, bias = synth.hidden_states(s, T, seed=21), synth.router_weights(s, seed=22), None
    g = torch.Generator().manual_seed(23)
    rows = torch.randperm(E, generator=g)
    if what == "small hidden states":
        hidden = (hidden.float() * torch.logspace(-12, -1, T)[:, None]).to(torch.bfloat16)
    elif what == "zero hidden states":
        hidden = torch.zeros_like(hidden)
        bias = torch.randint(0, 40, (E,), generator=g).float() * 1e-9
    elif what == "large logits":
        bias = torch.rand(E, generator=g) * 90.0
        bias[rows[:k]] = 90.0 + torch.arange(k) * 1e-6
    else:
        bias = torch.zeros(E)
        if what == "subnormal probabilities":
            bias[rows[3:]] = -torch.linspace(80.0, 115.0, E - 3)
        elif what == "all but one far below":
            bias[rows[1:]] = -200.0
        else:
            bias[rows[k - 2:]] = -1e4 if what == "fewer than k unmasked" else float("-inf")
    hidden, w, bias = hidden.cuda(), w.cuda(), None if bias is None else bias.cuda()
    ids, p = B.exmoe_route(s, hidden, w, bias)
    for t in range(0, T, 40):
        i1, p1 = B.exmoe_route(s, hidden[t:t + 40].contiguous(), w, bias)
        assert torch.equal(ids[t:t + 40], i1), t
        torch.testing.assert_close(p[t:t + 40], p1, rtol=2e-5, atol=1e-9)
