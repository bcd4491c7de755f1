"""GPU-vs-oracle parity through the C ABI (run with -m gpu on a B200)."""
import os

import numpy as np
import pytest

import gen
import oracle

pytestmark = pytest.mark.gpu


def _pair(*a, **kw):
    from parity_util import Pair
    return Pair(*a, **kw)


def _bias(seed, E, alpha, n_seq):
    return np.stack([gen.router_bias(seed, 0, s, alpha, E) for s in range(n_seq)])


def test_tiny_config_32_decode_tokens_cold_start():
    """Config 1: d=256, F=512, 8 experts, top-2, 4 slots, 32 single-token calls."""
    c = gen.config_by_name("tiny")
    P = _pair(c.d_model, c.d_ff, c.n_experts, c.top_k, c.cache_slots[0], seed=c.seed)
    P.set_bias(_bias(c.seed, c.n_experts, c.alphas[0], 1), None)
    misses = 0
    for step in range(c.decode_steps):
        x = gen.hidden_states(c.seed, 0, "decode", step, 1, c.d_model)
        _, o = P.step(x)
        misses += o["stats"]["misses"]
    assert misses >= 2          # cold start: the first call misses both experts
    P.close()


@pytest.mark.parametrize("d,F,E,k,C", [
    (512, 200, 16, 4, 5),       # ragged d_ff (25 units), waves when T*k > C
    (1024, 64, 8, 2, 2),        # cache as small as top-k
    (2048, 96, 12, 3, 12),      # everything resident after warm-up
    (3072, 40, 6, 2, 3),
    (4096, 72, 5, 2, 4),        # widest rows (two ring entries per 8 rows)
])
def test_shapes_and_token_counts(d, F, E, k, C):
    P = _pair(d, F, E, k, C, seed=100 + d // 256)
    n_seq = 3
    P.set_bias(_bias(7, E, 0.5, n_seq), None)
    step = 0
    for T in (1, 3, 8, 1, 19, 70, 2, 1):
        seq = (np.arange(T) * n_seq // max(T, 1)).astype(np.int32)
        P.set_bias(P.bias, seq)
        x = gen.hidden_states(100 + d, 0, "decode", step, T, d)
        P.step(x)
        step += 1
    eos, tot = P.gpu.layer.cache_state()
    assert tot["hits"] + tot["misses"] > 0
    P.close()


@pytest.mark.parametrize("d,E,k,n_seq", [(4096, 6, 2, 40), (2048, 33, 2, 32), (256, 64, 8, 33), (2304, 3, 1, 5)])
def test_decode_router_over_its_token_groups_and_sequences(d, E, k, n_seq):
    """The decode router's warps by experts and token groups, one and two halves of a row, more sequences than lanes:
    logits, indices and traces bit for bit with every expert resident (more pairs than slots, no more experts)."""
    P = _pair(d, 16, E, k, E, seed=90 + E)
    bias = _bias(90, E, 0.5, n_seq)
    for step, T in enumerate((1, 2, 3, 5, 7, 8)):
        P.set_bias(bias, ((np.arange(T) * 11 + n_seq - 1) % n_seq).astype(np.int32))
        P.step(gen.hidden_states(90 + E, 0, "decode", step, T, d))
    P.close()


@pytest.mark.parametrize("T", [1, 4, 8])
def test_decode_router_takes_sequences_that_the_kernel_ahead_writes(T):
    """token_seq is the output of the kernel directly ahead (a prompt through experts of zeros), over what was no valid
    sequence before, with more sequences than a warp has lanes: the router may be running by then, and must not have
    looked a bias up with what it found."""
    import torch
    from paper_2602_11192_b200.runner import current_stream_ptr, to_dev_bf16
    d, E, k, n_seq = 512, 12, 2, 40
    A, P = _pair(d, 16, E, k, E, seed=97), _pair(d, 16, E, k, E, seed=98)
    A.gpu.store.zero_()
    bias = _bias(97, E, 0.5, n_seq)
    bias_dev, seq = torch.from_numpy(bias).cuda(), torch.empty((9, d // 2), dtype=torch.int32, device="cuda")
    P.gpu.layer.set_router_bias(bias_dev, seq, n_seq)
    x = [gen.hidden_states(98, 0, "decode", i, T, d) for i in range(4)]
    xd, xa = [to_dev_bf16(v) for v in x], to_dev_bf16(gen.hidden_states(97, 0, "prefill", 0, 9, d))
    out = torch.empty((T, d), dtype=torch.int16, device="cuda")
    for step in range(4):
        seq.fill_(0x7FFFFFF0 if step % 2 else -5)
        A.gpu.layer.forward(current_stream_ptr(), xa, 9, seq)
        P.gpu.layer.forward(current_stream_ptr(), xd[step], T, out)
        torch.cuda.synchronize()
        assert int(seq.abs().max()) == 0
        idx, _, logits = oracle.route(x[step], P.w_r, k, bias, np.zeros(T, np.int32))
        assert np.array_equal(P.gpu.layer.last_logits(T).view(np.uint32), logits.view(np.uint32))
        assert np.array_equal(P.gpu.layer.last_routing(T)[0], idx)
    A.close()
    P.close()


@pytest.mark.parametrize("T,E,k,C", [(1, 64, 8, 64), (1, 40, 3, 5), (3, 12, 2, 6), (8, 33, 8, 33), (8, 16, 2, 4), (20, 12, 2, 6)])
def test_hidden_states_and_biases_that_are_not_finite(T, E, k, C):
    """One token's hidden state holds NaNs (all its logits are NaN: the lowest ids are taken, once each), another's experts
    are masked with a bias of -inf but for k - 1 of them, a third's are all +inf: every token has k distinct experts, the
    call's requests are no more than its pairs, and the other tokens' results are the oracle's."""
    d = 512
    P = _pair(d, 16, E, k, C, seed=130 + E)
    bias = np.zeros((3, E), np.float32)
    bias[1, :] = -np.inf
    bias[1, E - (k - 1):] = 0.0
    bias[2, :] = np.inf
    for step in range(3):
        x = gen.hidden_states(130 + E, 0, "decode", step, T, d)
        bad = step % T
        x[bad, ::7] = 0x7FC1 if step != 1 else 0xFFFF
        seq = np.zeros(T, np.int32)
        if T > 2:
            seq[(bad + 1) % T], seq[(bad + 2) % T] = 1, 2
        P.set_bias(bias, seq)
        res = P.gpu.forward_np(x)
        idx, _ = P.gpu.layer.last_routing(T)
        assert idx.min() >= 0 and idx.max() < E and all(len(set(r)) == k for r in idx.tolist())
        assert idx[bad].tolist() == list(range(k))
        good = [t for t in range(T) if t != bad and seq[t] != 2]
        if T > 2:
            assert sorted(idx[(bad + 1) % T].tolist()) == [0] + list(range(E - (k - 1), E))
            assert idx[(bad + 2) % T].tolist() == list(range(k))
        st = res["stats"]
        assert st["status"] == 0 and st["n_distinct"] == len(np.unique(idx)) == st["hits"] + st["misses"]
        cnt, off, perm = P.gpu.layer.last_gather(T)
        assert np.array_equal(cnt, np.bincount(idx.reshape(-1), minlength=E)) and sorted(perm.tolist()) == list(range(T * k))
        if good:
            sub_bias, sub_seq = bias, seq[good]
            idx_o, gate_o, _ = oracle.route(x[good], P.w_r, k, sub_bias, sub_seq)
            assert np.array_equal(idx[good], idx_o)
            y = oracle.ffn_combine(x[good], idx_o, gate_o, P.weights, P.F, 0)
            from parity_util import rel_err_per_token
            assert rel_err_per_token(res["out_bits"][good], y).max() <= 8e-3
    # and the cache is in order: every resident expert in one slot
    eos, _ = P.gpu.layer.cache_state()
    held = [e for e in eos.tolist() if e >= 0]
    assert len(set(held)) == len(held)
    P.close()


@pytest.mark.parametrize("store,d,E,k,n_shared", [("bf16", 512, 64, 32, 3), ("q4slots", 512, 9, 1, 0), ("bf16", 256, 1, 1, 0), ("bf16", 4096, 5, 4, 1)])
def test_one_token_calls_take_their_requests_from_records_of_their_own(store, d, E, k, n_shared):
    """One-token calls, fetching (announced by the plan's word) and then all resident (announced by the records, of
    which a warp's lanes are too few for 32 experts and 3 shared ones), between calls of two tokens."""
    P = _pair(d, 24, E, k, E, seed=95 + E, n_shared=n_shared, store=store)
    P.set_bias(_bias(95, E, 0.3, 2), None)
    for step, T in enumerate((1, 1, 2, 1, 1, 1, 2, 1)):
        P.step(gen.hidden_states(95 + E, 0, "decode", step % 3, T, d))
    P.close()


@pytest.mark.parametrize("policy", ["lru", "count"])
def test_what_follows_a_decode_call_sees_all_that_its_planner_wrote(policy):
    """The smallest layer, whose FFN kernel takes hardly longer than the rest of the planning it overlaps.  The kernel
    directly behind it (programmatically launched: another layer's call that takes the statistics as its hidden state)
    reads the statistics of this very call; preloads queued behind calls, with nothing waiting in between, leave the
    cache as the oracle has it."""
    import torch
    from paper_2602_11192_b200.runner import current_stream_ptr, to_dev_bf16
    d, F, E, k, C = 256, 8, 12, 2, 6
    P, R = _pair(d, F, E, k, C, seed=101), _pair(d, F, E, k, E, seed=102)
    P.set_policy(policy, 0.9 if policy == "count" else 0.0)
    # (whole numbers as bf16 patterns are denormal: the reader's router scales them up)
    R.gpu.set_router(np.full((E, d), 0x4E80, np.uint16))
    s = current_stream_ptr()
    out = torch.empty((1, d), dtype=torch.int16, device="cuda")
    xs = [gen.hidden_states(101, 0, "decode", i, 1, d) for i in range(40)]
    xd = [to_dev_bf16(x) for x in xs]
    rec = torch.zeros(d // 2, dtype=torch.int32, device="cuda")      # a hidden state that begins with a statistics record
    for i, x in enumerate(xs):
        P.gpu.layer.forward(s, xd[i], 1, out, rec)
        R.gpu.layer.forward(s, rec, 1, out)
        torch.cuda.synchronize()
        seen = R.gpu.layer.last_logits(1).copy()
        R.gpu.layer.forward(s, rec, 1, out)
        torch.cuda.synchronize()
        assert np.array_equal(seen.view(np.uint32), R.gpu.layer.last_logits(1).view(np.uint32)), "call %d" % i
        assert int(rec[10]) == i + 1                                 # call_no
        P.cache.call(oracle.route(x, P.w_r, k, None, None)[0])
    rs = np.random.default_rng(101)
    for rnd in range(10):
        for i, x in enumerate(xs[:8]):
            P.gpu.layer.forward(s, xd[i], 1, out, rec)
            ids = rs.permutation(E)[:2].astype(np.int32)
            P.gpu.layer.preload(ids)
            P.cache.call(oracle.route(x, P.w_r, k, None, None)[0])
            P.cache.preload(ids.tolist())
        P.gpu.layer.forward(s, xd[8], 1, out, rec)
        P.cache.call(oracle.route(xs[8], P.w_r, k, None, None)[0])
        torch.cuda.synchronize()
        eos, _, tot = P.cache.state()
        eos_g, tot_g = P.gpu.layer.cache_state()
        assert np.array_equal(eos_g, eos) and tot_g == tot
        assert np.array_equal(P.gpu.layer.cache_counts(E).view(np.uint32), P.cache.counts().view(np.uint32))
    P.close()
    R.close()


@pytest.mark.parametrize("d,F", [(256, 8), (2048, 64)])
def test_one_token_calls_in_a_chain_read_what_the_call_ahead_wrote(d, F):
    """Layers whose hidden state is the output of the layer ahead, in two buffers that take turns (so every SM has held
    older contents of the same addresses), all resident: queued back to back, the bits of calls that are waited for."""
    import torch
    from paper_2602_11192_b200.runner import current_stream_ptr, to_dev_bf16
    E, k, n_layers = 8, 2, 5
    Ps = [_pair(d, F, E, k, E, seed=110 + l) for l in range(n_layers)]
    s = current_stream_ptr()
    for l, P in enumerate(Ps):
        P.gpu.layer.preload(np.arange(E, dtype=np.int32))
        P.set_bias(_bias(110 + l, E, 0.5, 1), None)
    buf = torch.empty((2, d), dtype=torch.int16, device="cuda")
    xs = torch.stack([to_dev_bf16(gen.hidden_states(110, 0, "decode", i, 1, d))[0] for i in range(20)])

    def chain(wait):
        outs = torch.empty((len(xs), n_layers, d), dtype=torch.int16, device="cuda")
        for i in range(len(xs)):
            buf[0].copy_(xs[i])
            for l, P in enumerate(Ps):
                P.gpu.layer.forward(s, buf[l % 2], 1, buf[(l + 1) % 2])
                if wait:
                    torch.cuda.synchronize()
                    outs[i, l].copy_(buf[(l + 1) % 2])
            outs[i, -1].copy_(buf[n_layers % 2])
        torch.cuda.synchronize()
        return outs.cpu().numpy()

    want = chain(True)
    for _ in range(5):
        assert np.array_equal(chain(False)[:, -1], want[:, -1])
    for P in Ps:
        P.close()


@pytest.mark.parametrize("F", [48, 600])
def test_wide_model_with_many_tokens_keeps_its_token_operands_in_tensor_memory(F):
    """d_model 4096 with 5 to 8 tokens per call: where that saves an SM a tile (d_ff 600: twelve rows of three experts), the decode
    kernel writes the hidden states' tensor-core operands into tensor memory once and reads them from there (the shared memory goes
    to taller weight tiles).  Calls whose missed experts the kernel fetches itself (token-expert pairs <= slots), with a
    shared expert, between calls of fewer tokens that take the shared-memory form; then the same bits
    again from a warm cache (the sum over the SMs is exact, so residency must not change the output)."""
    d, E, k, C = 4096, 20, 2, 16
    P = _pair(d, F, E, k, C, seed=77, n_shared=1)
    P.set_bias(_bias(9, E, 0.5, 4), None)
    outs = {}
    for rnd in range(2):
        for step, T in enumerate((8, 5, 2, 7, 6, 1, 8)):
            P.set_bias(P.bias, (np.arange(T) % 4).astype(np.int32))
            res, o = P.step(gen.hidden_states(77, 0, "decode", step, T, d))
            if rnd == 0:
                outs[step] = res["out_bits"].copy()
            else:
                assert np.array_equal(outs[step], res["out_bits"]), "output bits depend on the cache state"
    assert not P.gpu.layer.last_call_used_gemm()
    P.close()


@pytest.mark.parametrize("store,d,F,k,n_shared,C", [
    ("bf16", 256, 1768, 2, 0, 3), ("bf16", 256, 1760, 2, 0, 3),      # the least rows per SM for four groups of warps, and less
    ("bf16", 512, 888, 2, 0, 4), ("bf16", 512, 880, 2, 0, 4),        # the same for two groups
    ("bf16", 512, 3608, 1, 0, 4), ("bf16", 768, 1200, 2, 1, 2),      # d_ff that ends inside a tile; missed experts stored by either group
    ("bf16", 1024, 1768, 2, 0, 2),
    ("bf16", 1280, 72, 2, 0, 3), ("bf16", 1792, 1768, 1, 1, 4),      # one group, widths of their own
    ("bf16", 1536, 72, 2, 0, 3), ("bf16", 2304, 72, 2, 0, 2), ("bf16", 2560, 200, 2, 1, 4), ("bf16", 2816, 72, 2, 0, 3),
    ("bf16", 3072, 72, 2, 0, 3), ("bf16", 3328, 72, 2, 0, 3), ("bf16", 3584, 48, 2, 1, 2), ("bf16", 3840, 48, 2, 1, 4),
    ("bf16", 3072, 1480, 2, 0, 4), ("bf16", 3328, 1480, 2, 0, 3),    # token operands in tensor memory from some number of tokens on
    ("bf16", 3584, 1480, 2, 0, 4), ("bf16", 3840, 888, 1, 1, 2), ("bf16", 4096, 888, 1, 1, 4),
    ("q4slots", 512, 1768, 2, 0, 3), ("q4slots", 512, 64, 2, 0, 3),  # 4-bit slots: two groups and one
    ("q4slots", 1024, 1768, 2, 0, 2), ("q4slots", 1024, 72, 2, 1, 3),
    ("q4slots", 2048, 1768, 2, 0, 4), ("q4slots", 4096, 72, 2, 0, 3),
    ("q4slots", 2048, 144, 2, 0, 3), ("q4slots", 2048, 152, 2, 0, 3),  # one group below two rows per SM, and two
])
def test_decode_kernels_of_every_width_and_grouping(store, d, F, k, n_shared, C):
    """Decode calls of 1 to 8 tokens, missed experts fetched by the kernel or by the host, element by element against the
    oracle; then the same bits from whatever the cache holds by then."""
    E = 4
    P = _pair(d, F, E, k, C, seed=800 + d // 256, n_shared=n_shared, store=store)
    P.set_bias(_bias(25, E, 0.5, 2), None)
    outs = {}
    for rnd in range(2):
        for step, T in enumerate((1, 4, 5, 2, 8)):
            P.set_bias(P.bias, (np.arange(T) % 2).astype(np.int32))
            x = gen.hidden_states(801, 0, "decode", step, T, d)
            if rnd == 0:
                res, _ = P.step(x)
                outs[step] = res["out_bits"].copy()
            elif T * k <= C or C == E:               # (in compute groups a token's sum depends on what is resident)
                assert np.array_equal(P.gpu.forward_np(x)["out_bits"], outs[step]), T
    P.close()


def test_largest_supported_sizes_and_empty_call():
    """d_model, n_experts and top_k at their limits; T * k = 64 is the largest call the fused
    decode planner takes, T = 3 already goes through the general kernels; T = 0 is a no-op."""
    from paper_2602_11192_b200 import MelinoeError, MoELayer
    with pytest.raises(MelinoeError) as ei:
        MoELayer(8192, 64, 8, 2, 2)                 # wider than the decode kernel's accumulators cover
    assert ei.value.status == 6
    import torch
    from paper_2602_11192_b200.runner import current_stream_ptr
    d, F, E, k, C = 4096, 64, 64, 32, 32
    P = _pair(d, F, E, k, C, seed=41)
    for step, T in enumerate((1, 2, 3, 9, 1)):
        P.step(gen.hidden_states(41, 0, "decode", step, T, d), tokens=[0, T - 1] if T > 1 else None)
    x = torch.zeros((1, d), dtype=torch.int16, device="cuda")
    y = torch.full((1, d), 7, dtype=torch.int16, device="cuda")
    before = P.gpu.layer.cache_state()
    P.gpu.layer.forward(current_stream_ptr(), x, 0, y)
    torch.cuda.synchronize()
    assert int(y.min()) == 7 and int(y.max()) == 7          # nothing written
    after = P.gpu.layer.cache_state()
    assert np.array_equal(before[0], after[0]) and before[1] == after[1]
    P.close()


def test_full_cache_has_only_compulsory_misses():
    E, k = 8, 2
    P = _pair(256, 64, E, k, E, seed=3)
    seen = set()
    for step in range(24):
        x = gen.hidden_states(3, 0, "decode", step, 1, 256)
        _, o = P.step(x)
        for e, s, hit, ev in o["req"].tolist():
            assert ev == -1 and bool(hit) == (e in seen)
            seen.add(e)
    _, tot = P.gpu.layer.cache_state()
    assert tot["misses"] == len(seen) and tot["evictions"] == 0
    P.close()


def test_output_does_not_depend_on_cache_size_or_history():
    d, F, E, k = 512, 64, 8, 2
    xs = [gen.hidden_states(5, 0, "decode", s, 2, d) for s in range(6)]
    outs = {}
    for C in (2, 5, 8):
        P = _pair(d, F, E, k, C, seed=5)
        outs[C] = [P.step(x)[0]["out_bits"] for x in xs]
        # warm second pass over the same inputs: same outputs
        again = [P.step(x)[0]["out_bits"] for x in xs]
        for a, b in zip(outs[C], again):
            assert np.array_equal(a, b)
        P.close()
    for C in (5, 8):
        for a, b in zip(outs[C], outs[2]):
            assert np.array_equal(a, b)


def test_shared_experts_and_batch():
    d, F, E, k, C = 512, 48, 10, 3, 4
    P = _pair(d, F, E, k, C, seed=9, n_shared=2)
    P.set_bias(_bias(9, E, 0.3, 4), np.arange(4, dtype=np.int32))
    for step in range(5):
        x = gen.hidden_states(9, 0, "decode", step, 4, d)
        P.step(x)
    P.set_bias(P.bias, (np.arange(37) % 4).astype(np.int32))
    P.step(gen.hidden_states(9, 0, "prefill", 0, 37, d))
    P.close()


def test_prefill_then_decode_with_waves():
    """More distinct experts than slots in one call: the misses come in waves."""
    d, F, E, k, C = 512, 64, 16, 4, 4
    P = _pair(d, F, E, k, C, seed=11)
    x = gen.hidden_states(11, 0, "prefill", 0, 40, d)
    _, o = P.step(x)
    assert o["stats"]["n_distinct"] > C and o["stats"]["groups"] >= 3
    for step in range(6):
        P.step(gen.hidden_states(11, 0, "decode", step, 1, d))
    P.close()


@pytest.mark.parametrize("d,F,E,k,C,n_shared,Ts", [
    (512, 256, 8, 2, 8, 0, (40, 300, 9)),        # everything fits the cache: one compute group after warm-up
    (256, 128, 16, 4, 5, 0, (130, 64)),          # more distinct experts than slots: miss waves
    (1024, 384, 6, 2, 3, 2, (257, 20)),          # shared experts, ragged last m-tile
    (512, 256, 4, 2, 4, 0, (600, 385, 40)),      # many tokens per expert, ragged
    (1024, 384, 4, 2, 2, 1, (700,)),             # many tokens per expert with a shared expert and miss waves
    (256, 256, 2, 2, 2, 0, (1100, 520)),         # every token to both experts: nine m-tiles (CTA pairs, the last one half empty)
    (512, 1032, 6, 3, 3, 1, (130, 64)),          # a launch for each GEMM of a wave
])
def test_prefill_grouped_gemm(d, F, E, k, C, n_shared, Ts):
    """Calls of more than 8 tokens run the tensor-core grouped GEMM (d_ff a multiple of 128)."""
    P = _pair(d, F, E, k, C, seed=200 + d // 256, n_shared=n_shared)
    n_seq = 4
    bias = _bias(21, E, 0.5, n_seq)
    step = 0
    for T in Ts:
        P.set_bias(bias, (np.arange(T) % n_seq).astype(np.int32))
        x = gen.hidden_states(300 + d, 0, "prefill", step, T, d)
        # the oracle evaluates a spread of tokens (first, last and every 7th): the FFN is per token
        tokens = sorted(set([0, 1, T - 2, T - 1] + list(range(0, T, 7))))
        P.step(x, tokens=tokens)
        assert P.gpu.layer.last_call_used_gemm()
        step += 1
    # and decode-sized calls on the same handle afterwards (streaming kernel), sharing the cache state
    P.set_bias(bias, np.zeros(2, np.int32))
    P.step(gen.hidden_states(300 + d, 0, "decode", 0, 2, d))
    assert not P.gpu.layer.last_call_used_gemm()
    P.close()


@pytest.mark.parametrize("store,d,F,E,k,n_shared,Ts", [
    ("bf16", 256, 8, 2, 1, 0, (9, 33)),                # one row group of hidden units: less than a weight tile and a k-block
    ("bf16", 512, 200, 3, 3, 1, (15, 17, 127, 129)),   # every expert sees every token: chunks of 16, 32, 128 and 2 x 80 tokens; d_ff ends inside a tile
    ("bf16", 256, 328, 2, 2, 0, (256, 257, 258, 300)), # CTA pairs: 256 tokens in one chunk, 257 in two; d_ff ends inside the pair's second tile
    ("q4slots", 512, 200, 3, 3, 1, (9, 16, 129)),      # the same of 4-bit codes, with a shared expert
    ("q4slots", 1024, 264, 4, 2, 0, (70,)),            # codes of a column group in both halves of their 128 bytes
    ("q4slots", 4096, 136, 2, 1, 0, (20,)),
    ("bf16", 2048, 1416, 2, 1, 1, (9, 140)),           # d_ff of 22 tiles and an eighth of one; GEMM 2 of 23 k-blocks, the last an eighth
    ("q4slots", 2048, 1416, 2, 1, 1, (9, 300)),        # the same of 4-bit codes; chunks of up to 256 tokens
    ("q4slots", 512, 64, 2, 2, 0, (256, 257)),         # one and two chunks; GEMM 2 of a single k-block
    ("bf16", 512, 200, 3, 3, 1, (32, 64, 65)),         # rows fetched by index up to 64 tokens, copied from 65 on
    ("q4slots", 512, 72, 6, 2, 0, (96, 97)),           # single CTAs up to 32 pairs per expert, pairs of CTAs beyond
    ("bf16", 256, 520, 5, 2, 1, (9, 64, 65, 700)),     # a launch for each GEMM; rows by index and copied
    ("bf16", 768, 1160, 3, 2, 0, (70, 300)),
    ("q4slots", 512, 1416, 4, 2, 1, (64, 65, 513)),    # one launch of single CTAs, then two of pairs
    ("q4slots", 512, 264, 16, 2, 1, (200, 256)),       # single CTAs, a shared expert of two chunks: tiles expanded for each
    ("bf16", 1024, 6144, 2, 1, 0, (512, 513)),         # two launches up to 256 pairs per expert, one beyond
    ("q4slots", 1024, 2560, 2, 1, 0, (512, 513)),
])
def test_grouped_gemm_at_the_edges_of_its_tiles(store, d, F, E, k, n_shared, Ts):
    """Token counts around the steps of the tensor-core operation's N and d_ff that ends inside weight tiles and
    k-blocks, element by element against the oracle."""
    P = _pair(d, F, E, k, E, seed=400 + d // 256 + F, n_shared=n_shared, store=store)
    for step, T in enumerate(Ts):
        tokens = sorted(set([0, 1, T - 2, T - 1] + list(range(0, T, 5))))
        P.step(gen.hidden_states(401 + d, 0, "prefill", step, T, d), tokens=tokens)
    P.close()


@pytest.mark.parametrize("T,d", [(20, 1024), (200, 1024), (200, 512)])
def test_prompts_of_two_layers_on_two_streams(T, d):
    """GEMM 2's items wait for GEMM 1's of whichever CTA has them, or its launch for GEMM 1's: with two layers' launches competing
    for the SMs, queued back to back on a stream each, both give the bits that they give alone."""
    import torch
    from paper_2602_11192_b200.runner import to_dev_bf16
    F, E, k = 1024, 16, 4
    Ps = [_pair(d, F, E, k, E, seed=520 + l) for l in range(2)]
    streams = [torch.cuda.Stream() for _ in Ps]
    xs = [to_dev_bf16(gen.hidden_states(520 + l, 0, "prefill", 0, T, d)) for l in range(2)]
    for P in Ps:
        P.gpu.layer.preload(np.arange(E, dtype=np.int32))
        P.set_bias(_bias(24, E, 0.5, 1), None)
        P.gpu.layer.reserve(T)
    outs = torch.empty((2, 20, T, d), dtype=torch.int16, device="cuda")
    want = []
    for P, s, x in zip(Ps, streams, xs):
        y = torch.empty((T, d), dtype=torch.int16, device="cuda")
        torch.cuda.synchronize()
        P.gpu.layer.forward(s.cuda_stream, x, T, y)
        torch.cuda.synchronize()
        want.append(y.cpu().numpy())
    for i in range(20):
        for l, (P, s, x) in enumerate(zip(Ps, streams, xs)):
            P.gpu.layer.forward(s.cuda_stream, x, T, outs[l, i])
    torch.cuda.synchronize()
    for l, P in enumerate(Ps):
        for i in range(20):
            assert np.array_equal(outs[l, i].cpu().numpy(), want[l]), (l, i)
        P.close()


@pytest.mark.parametrize("E,k,Ts", [(1, 1, (9, 700)), (5, 5, (296, 297, 1200)), (33, 3, (592, 593)), (64, 32, (65, 600)), (16, 2, (2500,))])
def test_router_and_token_lists_at_the_edges_of_their_tiles(E, k, Ts):
    """Token counts on both sides of the changes of the router's tile (148 SMs: one token per warp up to 296, two up
    to 592, then four), expert counts that do not fill its groups, more router blocks than the planning kernel
    keeps in registers, 512 pairs in a block: logits, indices, token lists and the trace bit for bit."""
    d, F = 512, 16
    P = _pair(d, F, E, k, E, seed=500 + E)
    P.set_bias(_bias(23, E, 0.5, 3), None)
    for step, T in enumerate(Ts):
        P.set_bias(P.bias, (np.arange(T) % 3).astype(np.int32))
        P.step(gen.hidden_states(501 + E, 0, "prefill", step, T, d), tokens=[0, T // 2, T - 1])
    P.close()


@pytest.mark.parametrize("T,d,E,k", [(9, 512, 12, 2), (400, 512, 12, 2), (600, 4096, 64, 32), (1500, 2048, 64, 32)])
def test_prompts_read_a_router_matrix_that_the_kernel_ahead_writes(T, d, E, k):
    """Only decode calls may read the router matrix before the work ahead of them has finished: here it is the output of
    the kernel directly ahead of a prompt, which may be running by then."""
    import torch
    from paper_2602_11192_b200.runner import current_stream_ptr, to_dev_bf16
    A, P = _pair(d, 16, E, k, E, seed=121), _pair(d, 16, E, 2, E, seed=122)
    A.gpu.layer.preload(np.arange(E, dtype=np.int32))
    w = torch.zeros((E, d), dtype=torch.int16, device="cuda")
    P.gpu.layer.set_router(w)
    x = gen.hidden_states(122, 0, "prefill", 0, T, d)
    xd, out = to_dev_bf16(x), torch.empty((T, d), dtype=torch.int16, device="cuda")
    for step in range(4):
        xa = to_dev_bf16(gen.hidden_states(121, 0, "prefill", step, E, d))
        A.gpu.layer.forward(current_stream_ptr(), xa, E, w)
        P.gpu.layer.forward(current_stream_ptr(), xd, T, out)
        torch.cuda.synchronize()
        idx, _, logits = oracle.route(x, w.cpu().numpy().view(np.uint16), 2, None, None)
        assert np.array_equal(P.gpu.layer.last_logits(T).view(np.uint32), logits.view(np.uint32))
        assert np.array_equal(P.gpu.layer.last_routing(T)[0], idx)
    A.close()
    P.close()


def test_prefill_router_breaks_ties_towards_the_lowest_expert_id():
    """More than 8 tokens go through the general router kernel: with a zero router matrix the logits are
    the bias alone, and a bias with equal entries makes ties that must go to the lowest ids (Eq. 1 with
    the tie rule of the oracle's strict-greater arg-max); all-equal logits select experts 0 .. k-1."""
    d, F, E, k, C = 512, 64, 12, 3, 6
    P = _pair(d, F, E, k, C, seed=81)
    P.w_r = np.zeros_like(P.w_r)
    P.gpu.set_router(P.w_r)
    bias = np.zeros((3, E), np.float32)
    bias[0, [2, 5, 7, 9, 11]] = 1.0            # five tied winners: 2, 5, 7 are taken
    bias[1, :] = 0.25                          # everything equal: 0, 1, 2
    bias[2, [10, 4]] = 3.0                     # two clear winners, then the lowest of the tied rest: 4, 10, 0
    for T in (20, 9, 33):
        seq = (np.arange(T) % 3).astype(np.int32)
        P.set_bias(bias, seq)
        _, o = P.step(gen.hidden_states(81, 0, "prefill", T, T, d), tokens=[0, 1, 2, T - 1])
        for t in range(T):
            want = {0: [2, 5, 7], 1: [0, 1, 2], 2: [4, 10, 0]}[int(seq[t])]
            assert o["idx"][t].tolist() == want
    # the same ties through the decode router (at most 8 tokens)
    P.set_bias(bias, np.arange(3, dtype=np.int32))
    _, o = P.step(gen.hidden_states(81, 0, "decode", 0, 3, d))
    assert o["idx"].tolist() == [[2, 5, 7], [0, 1, 2], [4, 10, 0]]
    P.close()


def test_a_failed_host_copy_leaves_the_handle_usable():
    """Error path of a partly queued call.  The failure is made on the host: a hook makes the first
    host-issued expert copy of the call report an error instead of being issued (nothing faults or
    waits on the device).  The call returns the error, later calls return it too until the cache is
    reset, the stream can be synchronised, and after the reset the layer works again."""
    import torch
    from paper_2602_11192_b200 import MelinoeError, lib
    from paper_2602_11192_b200.runner import current_stream_ptr, to_dev_bf16
    d, F, E, k, C = 512, 128, 8, 2, 4
    P = _pair(d, F, E, k, C, seed=83)
    T = 40                                              # grouped-GEMM path: the host issues the copies
    x = gen.hidden_states(83, 0, "prefill", 0, T, d)
    xd = to_dev_bf16(x)
    out = torch.zeros((T, d), dtype=torch.int16, device="cuda")
    lib().melinoe_debug_fail_host_copy(1)
    with pytest.raises(MelinoeError) as ei:
        P.gpu.layer.forward(current_stream_ptr(), xd, T, out)
    assert ei.value.status == 3
    lib().melinoe_debug_fail_host_copy(0)
    torch.cuda.synchronize()                            # whatever was queued runs to its end
    with pytest.raises(MelinoeError) as ei:
        P.gpu.layer.forward(current_stream_ptr(), xd, T, out)
    assert ei.value.status == 3                         # sticky
    with pytest.raises(MelinoeError):
        P.gpu.layer.cache_state()
    P.reset()                                           # clears the error; both sides start cold again
    P.step(x, tokens=[0, 7, T - 1])
    P.step(gen.hidden_states(83, 0, "decode", 0, 2, d))
    P.close()


def test_a_gather_whose_plan_never_comes_reports_it():
    """The gather of a long call waits for the plan's word, bounded.  With a word that nobody sets the wait runs out, the
    kernel ends and the handle says so, instead of leaving the lists and rows of the call before to be computed with."""
    import torch
    from paper_2602_11192_b200 import MelinoeError, lib
    from paper_2602_11192_b200.runner import current_stream_ptr
    P = _pair(512, 128, 8, 2, 8, seed=84)
    x = gen.hidden_states(84, 0, "prefill", 0, 70, 512)
    P.step(x, tokens=[0, 69])
    assert lib().melinoe_debug_gather_without_plan(P.gpu.layer._h, current_stream_ptr()) == 0
    torch.cuda.synchronize()
    with pytest.raises(MelinoeError) as ei:
        P.gpu.layer.cache_state()
    assert ei.value.status == 5
    P.reset()
    P.step(x, tokens=[0, 69])
    P.close()


def test_request_trace_records_calls_without_synchronising():
    """The request trace: 24 calls (decode-sized ones through the fused planner, two larger ones through the
    general planner) are queued back to back with no synchronisation in between; afterwards the ring holds
    the last 16 calls' records, each equal to what the oracle says of that call: routing indices, gates,
    request records in order, hit and miss counts."""
    import torch
    from paper_2602_11192_b200.budget import read_trace
    from paper_2602_11192_b200.runner import current_stream_ptr, to_dev_bf16
    d, F, E, k, C = 512, 64, 12, 2, 4
    P = _pair(d, F, E, k, C, seed=87)
    L = P.gpu.layer
    max_tok, cap = 8, 16
    rb = L.trace_record_bytes(max_tok)
    assert rb == (32 + 16 * E + 8 * max_tok * k + 15) // 16 * 16
    buf = torch.zeros(cap * rb, dtype=torch.uint8, device="cuda")
    L.set_trace(buf, buf.numel(), max_tok)
    Ts = [1, 3, 8, 1, 20, 2, 1, 5] * 3
    xs = [gen.hidden_states(87, 0, "decode", i, T, d) for i, T in enumerate(Ts)]
    outs = [torch.empty((T, d), dtype=torch.int16, device="cuda") for T in Ts]
    xd = [to_dev_bf16(x) for x in xs]
    s = current_stream_ptr()
    for x, o, T in zip(xd, outs, Ts):
        L.forward(s, x, T, o)                       # nothing waits here
    torch.cuda.synchronize()
    assert L.trace_count() == len(Ts)
    recs = read_trace(buf.cpu().numpy(), cap, E, k, max_tok)
    want = []
    for x in xs:
        idx, gate, _ = oracle.route(x, P.w_r, k)
        want.append((idx, gate, P.cache.call(idx)))
    for n in range(len(Ts) - cap, len(Ts)):
        r = recs[n % cap]
        idx, gate, req = want[n]
        nt = min(Ts[n], max_tok)
        assert r["call_no"] == n + 1 and r["n_tokens"] == Ts[n] and r["status"] == 0
        assert np.array_equal(r["idx"], idx[:nt]) and np.allclose(r["gate"], gate[:nt], rtol=1e-5, atol=1e-7)
        assert np.array_equal(r["req"], req)
        assert r["hits"] == int(req[:, 2].sum()) and r["misses"] == len(req) - int(req[:, 2].sum())
    L.set_trace(None, 0, 0)
    L.forward(s, xd[0], Ts[0], outs[0])
    torch.cuda.synchronize()
    assert L.trace_count() == len(Ts)               # switched off: nothing more is recorded
    P.close()


def test_forward_host_matches_forward_and_is_deterministic():
    import torch
    from paper_2602_11192_b200.runner import current_stream_ptr
    d, F, E, k, C = 512, 64, 8, 2, 3
    P = _pair(d, F, E, k, C, seed=13)
    xs = [gen.hidden_states(13, 0, "decode", s, 3, d) for s in range(5)]
    a = [P.step(x)[0]["out_bits"] for x in xs]
    P.reset()
    hx = torch.empty((3, d), dtype=torch.int16, pin_memory=True)
    hy = torch.empty((3, d), dtype=torch.int16, pin_memory=True)
    hs = torch.zeros(12, dtype=torch.int32, pin_memory=True)
    for i, x in enumerate(xs):
        hx.copy_(torch.from_numpy(x.view(np.int16)))
        P.gpu.layer.forward_host(current_stream_ptr(), hx, 3, hy, hs)
        torch.cuda.synchronize()
        assert np.array_equal(hy.numpy().view(np.uint16), a[i])
        assert int(hs[0]) == 0 and int(hs[1]) == 3
        P.cache.call(oracle.route(x, P.w_r, k)[0])
    # pageable host buffers take the staged route and give the same bits
    P.gpu.layer.reset_cache()
    py, ps = np.empty((3, d), np.int16), np.zeros(12, np.int32)
    for i, x in enumerate(xs):
        px = np.ascontiguousarray(x.view(np.int16))
        P.gpu.layer.forward_host(current_stream_ptr(), px, 3, py, ps)
        torch.cuda.synchronize()
        assert np.array_equal(py.view(np.uint16), a[i])
        assert int(ps[0]) == 0 and int(ps[1]) == 3
    P.close()


def test_preload_fills_the_cache_before_the_first_token():
    d, F, E, k, C = 256, 32, 8, 2, 4
    P = _pair(d, F, E, k, C, seed=15)
    x = gen.hidden_states(15, 0, "decode", 0, 1, d)
    idx, _, _ = oracle.route(x, P.w_r, k)
    P.preload(sorted(idx[0].tolist()))
    _, o = P.step(x)
    assert o["stats"]["misses"] == 0 and o["stats"]["hits"] == k
    eos, tot = P.gpu.layer.cache_state()
    assert tot["misses"] == k and set(eos[:k].tolist()) == set(idx[0].tolist())
    P.close()


@pytest.mark.parametrize("policy", ["lru", "count"])
def test_preload_is_queued_and_matches_the_oracle(policy):
    """Preloads in the middle of a stream of calls (on a warm cache: ids that are resident, ids that
    evict, a full list of cache_slots ids), queued without any host synchronisation between them and
    the calls around them; slot table, totals, counts and the following calls' traces and outputs
    agree with the oracle; then the pooled variant for a batch."""
    d, F, E, k, C = 512, 64, 12, 2, 5
    P = _pair(d, F, E, k, C, seed=17)
    if policy == "count":
        P.set_policy("count", 0.9)
    step = 0
    for ids in ([3, 7], [7, 1, 9, 3, 0], [11], [2, 2, 5]):
        P.preload(ids)
        for _ in range(2):
            P.step(gen.hidden_states(17, 0, "decode", step, 3, d))
            step += 1
    lists = np.array([[4, 6, 8], [6, 8, 10], [8, 1, 4], [0, 8, 6]], np.int32)
    want = oracle.pool_prefetch(lists, E, C)
    assert want.tolist() == [8, 6, 4, 0, 1]
    P.gpu.layer.preload_pooled(lists)
    P.cache.preload(want)
    P.step(gen.hidden_states(17, 0, "decode", step, 4, d))
    eos, _ = P.gpu.layer.cache_state()
    P.close()


@pytest.mark.parametrize("gamma", [1.0, 0.9, 0.5])
def test_count_policy_trace_matches_the_oracle(gamma):
    """Definition C.1's discounted-count eviction (gamma = 1: LFU): requests, victims, compute
    groups' results and the fp32 counts agree with the oracle call by call, decode and prefill."""
    d, F, E, k, C = 256, 64, 16, 2, 4
    P = _pair(d, F, E, k, C, seed=31)
    P.set_policy("count", gamma)
    bias = np.stack([gen.router_bias(31, 0, s, 0.3, E) for s in range(4)])
    n_evict = 0
    for step in range(40):
        T = (1, 3, 8)[step % 3]
        P.set_bias(bias, (np.arange(T) % 4).astype(np.int32))
        _, out = P.step(gen.hidden_states(31, 0, "decode", step, T, d))
        n_evict += int((out["req"][:, 3] >= 0).sum())
    assert n_evict > 20
    P.set_bias(bias, (np.arange(40) % 4).astype(np.int32))
    P.step(gen.hidden_states(31, 0, "prefill", 0, 40, d))     # many misses in one call: one wave each at worst
    # back to LRU on the same cache contents: the trace follows the LRU oracle again
    P.set_policy("lru")
    P.set_bias(bias, np.zeros(1, np.int32))
    for step in range(6):
        P.step(gen.hidden_states(31, 0, "decode", 100 + step, 1, d))
    P.close()


def test_count_policy_with_shared_experts_and_batches():
    """The count policy on a stack with always-resident shared experts (their requests sit between
    the hits and the miss waves in the launch order) and token batches."""
    d, F, E, k, C = 256, 64, 12, 3, 4
    P = _pair(d, F, E, k, C, seed=35, n_shared=2)
    P.set_policy("count", 0.9)
    for step, T in enumerate((4, 1, 8, 2, 30, 1, 5)):
        P.step(gen.hidden_states(35, 0, "decode", step, T, d))
    P.close()


def test_count_policy_preload_and_lfu_keeps_the_hot_experts():
    d, F, E, k, C = 256, 32, 8, 2, 4
    P = _pair(d, F, E, k, C, seed=33)
    P.set_policy("count", 1.0)
    P.preload([5, 1, 6, 2])
    assert np.array_equal(P.gpu.layer.cache_counts(E), P.cache.counts())
    for step in range(12):
        P.step(gen.hidden_states(33, 0, "decode", step, 2, d))
    with pytest.raises(Exception):
        P.gpu.layer.set_policy("count", 1.5)
    P.close()


def test_q4_host_store_matches_the_oracle_and_a_bf16_store_of_the_same_weights():
    """4-bit host store: the misses move 4-bit blobs, the layer computes with the weights the format
    defines.  Against the oracle on its own dequantised weights (tolerance), and bit for bit against
    a second layer whose bf16 store holds those dequantised weights."""
    from paper_2602_11192_b200.runner import LayerSetup
    d, F, E, k, C = 512, 128, 12, 2, 4
    P = _pair(d, F, E, k, C, seed=51, store="q4")
    assert P.bytes_per_miss == 3 * (d * F // 2 + d * F // 32)
    ref = LayerSetup(d, F, E, k, C)
    ref.set_experts(P.weights, [])
    ref.set_router(P.w_r)
    n_miss = 0
    for step, T in enumerate((1, 2, 8, 1, 20, 3, 1, 1)):
        x = gen.hidden_states(51, 0, "decode", step, T, d)
        res, out = P.step(x)
        n_miss += out["stats"]["misses"]
        assert np.array_equal(res["out_bits"], ref.forward_np(x)["out_bits"])
    assert n_miss > 10
    # preload goes through the same expansion
    P.reset()
    ref.layer.reset_cache()
    P.preload([3, 7])
    ref.layer.preload(np.array([3, 7], np.int32))
    x = gen.hidden_states(51, 0, "decode", 99, 4, d)
    res, _ = P.step(x)
    assert np.array_equal(res["out_bits"], ref.forward_np(x)["out_bits"])
    ref.close()
    P.close()


@pytest.mark.parametrize("d,F,E,k,C,n_shared", [(512, 128, 12, 2, 4, 0), (1024, 72, 16, 4, 8, 1), (2048, 64, 16, 8, 8, 0),
                                                (4096, 40, 8, 2, 4, 0)])
def test_q4_slots_match_the_oracle(d, F, E, k, C, n_shared):
    """4-bit cache slots: host link and HBM carry 4-bit blobs only, the FFN kernel expands the codes in
    registers.  Routing, cache trace and statistics bit for bit, activations element-wise, against the
    oracle on the weights the format defines; calls of 1..8 tokens (fetched by the kernel itself), of
    more tokens than slots allow (copies issued by the host) and of several launches; both entry points."""
    P = _pair(d, F, E, k, C, seed=61, n_shared=n_shared, store="q4slots")
    from paper_2602_11192_b200 import melinoe_moe_expert_bytes_q4
    assert P.bytes_per_miss == melinoe_moe_expert_bytes_q4(d, F) and P.gpu.layer.slots == "q4"
    n_miss = 0
    for step, T in enumerate((1, 1, 2, 8, 5, 1, 19, 3, 1, 4)):
        x = gen.hidden_states(61, 0, "decode", step, T, d)
        entry = "static" if T <= 8 and T * k <= 64 and step % 2 == 1 else "forward"
        res, out = P.step(x, entry=entry)
        n_miss += out["stats"]["misses"]
        assert not P.gpu.layer.last_call_used_gemm()
    assert n_miss > 6
    P.set_policy("count", 0.9)
    P.reset()
    P.preload(list(range(min(C, 3))))
    for step in range(6):
        P.step(gen.hidden_states(61, 0, "decode", 50 + step, 1 + step % 3, d))
    # a bf16 store cannot be registered on this handle, nor 4-bit slots made for a width the kernel does not split
    with pytest.raises(Exception):
        P.gpu.layer.register_host_experts([0] * E, 3 * d * F * 2)
    P.close()
    from paper_2602_11192_b200 import MoELayer
    with pytest.raises(Exception):
        MoELayer(1536, 64, 8, 2, 4, slots="q4")


@pytest.mark.parametrize("d,F,E,k,n_shared,T", [(512, 72, 6, 2, 1, 40), (2048, 264, 5, 4, 0, 72), (1024, 64, 3, 3, 2, 300)])
def test_4bit_tokens_get_the_same_result_from_long_and_short_calls(d, F, E, k, n_shared, T):
    """A prompt through the grouped GEMM against the same tokens in decode calls of 8: both round gate * h to bf16, so
    only fp32 sums of the tensor cores differ in their order.  Where such sums differ by delta of themselves, a share of
    delta / 2^-8 of the roundings of h and y falls the other way, by 2^-8 of a value: sqrt(2^-8 * delta) in the 2-norm, 1e-3
    for delta = 2^-12 (twice the 4.9e-4 measured at d_model 2048); rounding h without its gate would be 3.2e-3."""
    P = _pair(d, F, E, k, E, seed=700 + d // 256, n_shared=n_shared, store="q4slots")
    P.set_bias(_bias(24, E, 0.5, 1), None)
    x = gen.hidden_states(701, 0, "prefill", 0, T, d)
    long_call = gen.bf16_bits_to_f32(P.gpu.forward_np(x)["out_bits"]).astype(np.float64)
    short = np.concatenate([gen.bf16_bits_to_f32(P.gpu.forward_np(x[i:i + 8])["out_bits"]) for i in range(0, T, 8)]).astype(np.float64)
    err = np.linalg.norm(long_call - short) / np.linalg.norm(short)
    assert err <= 1e-3, err
    P.close()


@pytest.mark.parametrize("T", [24, 100, 300])
def test_4bit_prompts_give_the_same_bits_every_time(T):
    """Weight tiles that one CTA of a pair expands and the other's thread multiplies (24 tokens: its own), many per CTA: a tile
    that was read before it was complete would change some output."""
    d, F, E, k = 2048, 1408, 12, 4
    P = _pair(d, F, E, k, E, seed=66, store="q4slots")
    x = gen.hidden_states(66, 0, "prefill", 0, T, d)
    res, _ = P.step(x, tokens=[0, T // 2, T - 1])
    for _ in range(30):
        assert np.array_equal(P.gpu.forward_np(x)["out_bits"], res["out_bits"])
    P.close()


def test_parity_without_programmatic_launch():
    """The decode kernels are launched with programmatic stream serialisation by default; the
    same parity must hold with the attribute switched off (the switch is read once per process,
    hence the child process)."""
    import os
    import subprocess
    import sys
    here = os.path.dirname(os.path.abspath(__file__))
    code = (
        "import sys; sys.path.insert(0, %r); sys.path.insert(0, %r)\n"
        "import numpy as np, gen\n"
        "from parity_util import Pair\n"
        "P = Pair(512, 64, 16, 2, 4, seed=61)\n"
        "for step, T in enumerate((1, 4, 1, 8, 2, 1, 12, 1)):\n"
        "    P.step(gen.hidden_states(61, 0, 'decode', step, T, 512))\n"
        "P.close()\n"
        "print('child ok')\n" % (os.path.dirname(here), here))
    env = dict(os.environ, MELINOE_MOE_NO_PDL="1")
    r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "child ok" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]


def _child(code_body, env_extra):
    import os
    import subprocess
    import sys
    here = os.path.dirname(os.path.abspath(__file__))
    code = ("import sys; sys.path.insert(0, %r); sys.path.insert(0, %r)\n"
            "import numpy as np, gen\nfrom parity_util import Pair\n" % (os.path.dirname(here), here)) + code_body + "print('child ok')\n"
    r = subprocess.run([sys.executable, "-c", code], env=dict(os.environ, **env_extra), capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0 and "child ok" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]


def test_parity_with_every_transfer_issued_by_the_host():
    """MELINOE_MOE_HOST_COPIES: decode calls, too, wait for their plan on the host and fetch with
    cudaMemcpyAsync (the switch is read once per process, hence the child process)."""
    _child("P = Pair(512, 64, 16, 2, 4, seed=62)\n"
           "for step, T in enumerate((1, 2, 1, 8, 2, 1, 12, 1)):\n"
           "    P.step(gen.hidden_states(62, 0, 'decode', step, T, 512))\n"
           "P.close()\n", {"MELINOE_MOE_HOST_COPIES": "1"})


@pytest.mark.parametrize("policy,T", [("lru", 1), ("count", 1), ("lru", 3)])
def test_host_issued_transfers_of_calls_queued_back_to_back(policy, T):
    """A 4-bit store feeding bf16 slots: the host queues the copies of a call while its planner is still writing the cache
    state, and then the next call.  Bits and cache are those of calls that are waited for."""
    import torch
    from paper_2602_11192_b200.runner import current_stream_ptr, to_dev_bf16
    d, F, E, k, C, n = 512, 40, 16, 2, 4, 40
    P = _pair(d, F, E, k, C, seed=64, store="q4")
    P.set_policy(policy, 0.9 if policy == "count" else 0.0)
    xs = [gen.hidden_states(64, 0, "decode", i, T, d) for i in range(n)]
    want = [P.step(x)[0]["out_bits"].copy() for x in xs]
    P.reset()
    xd, out = [to_dev_bf16(x) for x in xs], torch.empty((n, T, d), dtype=torch.int16, device="cuda")
    for i in range(n):
        P.gpu.layer.forward(current_stream_ptr(), xd[i], T, out[i])
        P.cache.call(oracle.route(xs[i], P.w_r, k)[0])
    torch.cuda.synchronize()
    got = out.cpu().numpy().view(np.uint16)
    for i in range(n):
        assert np.array_equal(got[i], want[i]), i
    eos, _, tot = P.cache.state()
    eos_g, tot_g = P.gpu.layer.cache_state()
    assert np.array_equal(eos_g, eos) and tot_g == tot and tot["misses"] > n // 4
    P.close()


def test_parity_of_the_single_cta_gemm_on_a_call_of_many_tokens():
    """MELINOE_MOE_GEMM_SINGLE: a call that would pair CTAs (300 tokens per expert) through the
    cta_group::1 form of the grouped GEMM."""
    _child("P = Pair(512, 256, 4, 2, 4, seed=63)\n"
           "x = gen.hidden_states(63, 0, 'prefill', 0, 600, 512)\n"
           "P.step(x, tokens=sorted(set([0, 1, 598, 599] + list(range(0, 600, 7)))))\n"
           "assert P.gpu.layer.last_call_used_gemm()\n"
           "P.close()\n", {"MELINOE_MOE_GEMM_SINGLE": "1"})


def test_trace_miss_proxies_match_the_oracle():
    """Soft (Section 3.1) and hard (Definition C.1) miss proxies of recorded traces, every cache size
    at once: hard misses exact, soft proxy to fp64 rounding; then a budget split over the layers."""
    from paper_2602_11192_b200.budget import miss_curves, allocate_slots
    rs = np.random.default_rng(71)
    L, T, K, E = 3, 300, 2, 12
    trace = np.empty((L, T, K), np.int32)
    for l, alpha in enumerate((0.05, 0.5, 50.0)):             # from concentrated to uniform routing
        pref = rs.dirichlet(np.full(E, alpha)) + 1e-6
        pref /= pref.sum()
        for t in range(T):
            trace[l, t] = rs.choice(E, size=K, replace=False, p=pref)
    sizes = list(range(K, E + 1))
    for gamma in (1.0, 0.9, 0.0):
        soft, hard = miss_curves(trace, E, gamma, sizes)
        for l in range(L):
            for j, c in enumerate(sizes):
                so, ho = oracle.miss_proxies(trace[l], E, c, gamma)
                assert hard[l, j] == int(ho.sum()), (gamma, l, c)
                assert abs(soft[l, j] - so.mean()) <= 1e-10 * max(1.0, abs(so.mean())), (gamma, l, c)
        assert np.all(np.diff(hard, axis=1) <= 0)            # a larger gamma-cache never transfers more
    _, hard = miss_curves(trace, E, 0.9, sizes)
    slots = allocate_slots(hard, sizes, 3 * K + 9)
    assert sum(slots) == 3 * K + 9 and slots[0] <= slots[1]   # concentrated routing needs the fewest slots
    # a configuration that names nothing is marked, not evaluated
    import torch
    from paper_2602_11192_b200 import binding as B
    from paper_2602_11192_b200.runner import current_stream_ptr
    cfg = (B.ProxyConfig * 2)(B.ProxyConfig(7, 4, 0.9), B.ProxyConfig(0, 0, 0.9))
    cfg_dev = torch.frombuffer(bytearray(bytes(cfg)), dtype=torch.uint8).cuda()
    so = torch.zeros(2, dtype=torch.float64, device="cuda")
    ha = torch.zeros(2, dtype=torch.int64, device="cuda")
    B.melinoe_trace_miss_proxies(current_stream_ptr(), torch.from_numpy(trace).cuda(), L, T, K, E, cfg_dev, 2, so, ha)
    torch.cuda.synchronize()
    assert bool(torch.isnan(so).all()) and ha.tolist() == [-1, -1]


@pytest.mark.parametrize("T,K,E,gamma,sizes", [
    (1, 1, 1, 0.5, [1]),
    (31, 3, 33, 0.9, [1, 3, 32, 33]),           # fewer tokens than one batch of 32; three configurations rank with two warps
    (1100, 8, 64, 0.9, list(range(8, 65))),     # tokens held 512 at a time; 57 sizes share the ranking
    (513, 40, 64, 1.0, [40, 41, 63, 64]),       # more requests per token than a warp has lanes
    (700, 1, 64, 0.9, [5, 10, 11, 64]),         # the norm tends to K / (1 - gamma) = 10: just below, never above
    (200, 6, 40, 0.0, [6, 7, 40]),              # nothing is remembered
])
def test_trace_miss_proxies_at_the_edges_of_their_batches(T, K, E, gamma, sizes):
    """Hard misses exact, soft proxy to fp64 rounding (a sum of at most 64 T terms of at most 1 each)."""
    from paper_2602_11192_b200 import binding as B
    from paper_2602_11192_b200.runner import current_stream_ptr
    import torch
    rs = np.random.default_rng(T)
    pref = rs.dirichlet(np.full(E, 0.5)) + 1e-3
    trace = np.stack([rs.choice(E, size=K, replace=False, p=pref / pref.sum()) for _ in range(T)]).astype(np.int32)
    n = len(sizes)
    cfg = (B.ProxyConfig * n)(*[B.ProxyConfig(0, c, gamma) for c in sizes])
    cfg_dev = torch.frombuffer(bytearray(bytes(cfg)), dtype=torch.uint8).cuda()
    soft = torch.zeros(n, dtype=torch.float64, device="cuda")
    hard = torch.full((n,), 7, dtype=torch.int64, device="cuda")
    B.melinoe_trace_miss_proxies(current_stream_ptr(), torch.from_numpy(trace).cuda(), 1, T, K, E, cfg_dev, n, soft, hard)
    soft, hard = soft.cpu().numpy(), hard.cpu().numpy()
    for j, c in enumerate(sizes):
        so, ho = oracle.miss_proxies(trace, E, c, gamma)
        assert hard[j] == int(ho.sum()), (c, hard[j], int(ho.sum()))
        assert abs(soft[j] - so.mean()) <= 1e-10 * max(1.0, abs(so.mean())), (c, soft[j], so.mean())


@pytest.mark.parametrize("total", [600, 1200])
def test_trace_miss_proxies_of_groups_of_all_sizes(total):
    """Many configurations, so that not every block ranks, in groups (of a layer and gamma) of 15, 16, 31, 32, 48 and 57 sizes and
    of one to three, in an order that mixes them: hard misses exact, soft proxy to fp64 rounding."""
    from paper_2602_11192_b200 import binding as B
    from paper_2602_11192_b200.runner import current_stream_ptr
    import torch
    rs = np.random.default_rng(total)
    T, K, E, L = 90, 2, 64, 12
    trace = np.stack([np.stack([rs.choice(E, size=K, replace=False) for _ in range(T)]) for _ in range(L)]).astype(np.int32)
    cfgs = [(l, c, 0.9) for l, n in enumerate((15, 16, 31, 32, 48, 57)) for c in range(K, K + n)]
    for i in range(total):
        if len(cfgs) >= total:
            break
        cfgs += [(i % L, c, 0.5 + i / (4.0 * total)) for c in (3, 16, 40)[:1 + i % 3]]
    cfgs = [cfgs[i] for i in rs.permutation(len(cfgs))]
    n = len(cfgs)
    cfg_dev = torch.frombuffer(bytearray(bytes((B.ProxyConfig * n)(*[B.ProxyConfig(*c) for c in cfgs]))), dtype=torch.uint8).cuda()
    soft = torch.zeros(n, dtype=torch.float64, device="cuda")
    hard = torch.full((n,), 7, dtype=torch.int64, device="cuda")
    B.melinoe_trace_miss_proxies(current_stream_ptr(), torch.from_numpy(trace).cuda(), L, T, K, E, cfg_dev, n, soft, hard)
    soft, hard = soft.cpu().numpy(), hard.cpu().numpy()
    for j, (l, c, gamma) in enumerate(cfgs):
        so, ho = oracle.miss_proxies(trace[l], E, c, gamma)
        assert hard[j] == int(ho.sum()), (l, c, gamma, hard[j], int(ho.sum()))
        assert abs(soft[j] - so.mean()) <= 1e-10 * max(1.0, abs(so.mean())), (l, c, gamma, soft[j], so.mean())


@pytest.mark.parametrize("n_layers,E,n", [(1, 64, 57), (3, 5, 700)])
def test_trace_miss_proxies_of_no_tokens_are_zero(n_layers, E, n):
    """A trace without tokens: no misses and a mean of 0 for every configuration, whatever an earlier kernel left in
    shared memory (a trace of many tokens is evaluated ahead of each); a configuration that names nothing is marked."""
    from paper_2602_11192_b200 import binding as B
    from paper_2602_11192_b200.runner import current_stream_ptr
    import torch
    cfg = (B.ProxyConfig * (n + 1))(*[B.ProxyConfig(i % n_layers, 1 + i % E, 0.9) for i in range(n)], B.ProxyConfig(n_layers, 1, 0.9))
    cfg_dev = torch.frombuffer(bytearray(bytes(cfg)), dtype=torch.uint8).cuda()
    trace = (torch.arange(n_layers * 600 * 2, dtype=torch.int32, device="cuda") % E).contiguous()
    soft = torch.empty(n + 1, dtype=torch.float64, device="cuda")
    hard = torch.empty(n + 1, dtype=torch.int64, device="cuda")
    for _ in range(10):
        B.melinoe_trace_miss_proxies(current_stream_ptr(), trace, n_layers, 600, 2, E, cfg_dev, n + 1, soft, hard)
        soft.fill_(7.0)
        B.melinoe_trace_miss_proxies(current_stream_ptr(), trace, n_layers, 0, 2, E, cfg_dev, n + 1, soft, hard)
        assert not bool(soft[:n].any()) and not bool(hard[:n].any())
        assert bool(torch.isnan(soft[n])) and int(hard[n]) == -1


def test_argument_and_state_errors():
    import torch
    from paper_2602_11192_b200 import MoELayer, MelinoeError, melinoe_moe_expert_bytes
    from paper_2602_11192_b200.runner import current_stream_ptr
    for bad in ((250, 64, 8, 2, 4), (256, 63, 8, 2, 4), (256, 64, 65, 2, 4), (256, 64, 8, 3, 2), (256, 64, 8, 2, 9)):
        with pytest.raises(MelinoeError):
            MoELayer(*bad)
    L = MoELayer(256, 64, 4, 2, 2)
    x = torch.zeros((1, 256), dtype=torch.int16, device="cuda")
    y = torch.zeros((1, 256), dtype=torch.int16, device="cuda")
    with pytest.raises(MelinoeError) as ei:
        L.forward(current_stream_ptr(), x, 1, y)
    assert ei.value.status == 2                       # router / experts not set
    eb = melinoe_moe_expert_bytes(256, 64)
    pageable = torch.zeros((4, eb), dtype=torch.uint8)
    with pytest.raises(MelinoeError) as ei:
        L.register_host_experts([pageable.data_ptr() + i * eb for i in range(4)], eb)
    assert ei.value.status == 1                       # pageable memory is rejected, never staged
    pinned = torch.zeros((4, eb), dtype=torch.uint8, pin_memory=True)
    with pytest.raises(MelinoeError):
        L.register_host_experts([pinned.data_ptr() + i * eb for i in range(4)], eb - 2)
    L.register_host_experts([pinned.data_ptr() + i * eb for i in range(4)], eb, keep=pinned)
    w = torch.zeros((4, 256), dtype=torch.int16, device="cuda")
    L.set_router(w)
    L.forward(current_stream_ptr(), x, 0, y)          # zero tokens: no-op
    L.forward(current_stream_ptr(), x, 1, y)
    torch.cuda.synchronize()
    assert int(y.abs().max()) == 0                    # all-zero weights give exactly zero
    idx, gate = L.last_routing(1)
    assert idx.tolist() == [[0, 1]] and np.allclose(gate, 0.5)   # all-equal logits: lowest ids, equal gates
    L.destroy()
