"""The passes that cover several blocks of rows at once (the full blocks of a prompt; the sequences of a decode step) and
the attention kernels large launches take, against the paths small ones take (need a B200)."""
import numpy as np
import pytest
import torch

import synth
import paper_2603_17942_b200 as P
from tests.test_gpu_operators import R, _anc_words, _run_attention, _tree_block
from tests.test_gpu_parity import BF16_SMALL, TOL_BF16

pytestmark = pytest.mark.gpu


def _handle(w, max_seq, spec, batch=1):
    h = P.Handle(BF16_SMALL, spec, w, max_seq_len=max_seq, max_batch=batch)
    logits = torch.zeros(batch, R, BF16_SMALL.vocab, dtype=torch.float32, device="cuda")
    P.esp_debug_capture(h.h, logits)
    return h, logits


@pytest.fixture(scope="module")
def weights():
    return synth.make_weights(BF16_SMALL, seed=3, device="cuda", gain_jitter=True, std=0.05)


@pytest.mark.parametrize("n_prompt", [120, 121, 240, 241, 361, 1081, 1200])
def test_wide_prefill_against_cuda_core_path(weights, n_prompt):
    """Prompts whose full blocks make no wide pass, one of 2, of 3 (a ragged row tile), of 8, and one of 8 with a single
    block left over: the last prompt row's and the probe rows' logits against the CUDA-core GEMMs, which never take it.
    Both round the same activations to bf16 once or twice, so they agree to the bar bf16 logits are held to anywhere."""
    spec = P.spec_cfg(n_probes=3, topk=5, max_nodes=16, expand_width=0, n_anchor=1)
    prompt = synth.make_prompt(BF16_SMALL.vocab, n_prompt, 7)
    rows = slice((n_prompt - 1) % P.ESP_PREFILL_CHUNK, (n_prompt - 1) % P.ESP_PREFILL_CHUNK + 4)
    got = []
    for impl in (0, 1):
        h, logits = _handle(weights, 1300, spec)
        P.esp_debug_set_gemm(h.h, impl)
        h.prefill(prompt)
        got.append(logits[0, rows].clone())
        assert h.stats().device_error == 0 and h.state()["L"] == n_prompt
        h.close()
    span = float(got[1].max() - got[1].min())
    assert (got[0] - got[1]).abs().max() <= TOL_BF16 * span


@pytest.mark.parametrize("n_seq,nodes,n_anchor,idle", [(2, 16, 1, None), (2, 16, 1, 1), (5, 16, 1, 2), (33, 16, 1, 16), (4, 40, 1, 0), (2, 60, 1, 0), (4, 70, 1, None),
                                                        (4, 70, 1, 2), (5, 70, 1, 3), (7, 70, 1, 2), (8, 70, 1, None), (13, 70, 1, 12), (3, 25, 0, None), (3, 25, 0, 1)])
def test_batch_steps_against_each_sequence_alone(weights, n_seq, nodes, n_anchor, idle):
    """One step of a handle with several sequences (row tiles of every shape, ragged ones, more sequences than a
    pass covers, blocks of 100 rows) against the step each sequence takes in a handle of its own: the same trees (the
    prefill does not depend on the batch), logits equal to the bar bf16 logits are held to, for every sequence of every row
    tile, LM-head group and pass.  All of them take part, or all but one: the first or the last of a row tile, of a pass, of
    the handle."""
    spec = P.spec_cfg(n_probes=3, topk=5, max_nodes=nodes, expand_width=0 if n_anchor else 1, n_anchor=n_anchor)
    h, logits = _handle(weights, 400, spec, n_seq)
    prompts = [synth.make_prompt(BF16_SMALL.vocab, 17 + 40 * (i % 5), 10 + i) for i in range(n_seq)]
    who = [i for i in range(n_seq) if i != idle]
    for i in who:
        h.prefill(prompts[i], i)
    rows = {i: h.state(i)["n_rows"] for i in who}
    P.esp_step(h.h, h.tokens_out, h.n_out)
    assert h.stats().device_error == 0 and [i for i in range(n_seq) if h.n_out[i]] == who
    for i in who:
        one, alone = _handle(weights, 400, spec)
        one.prefill(prompts[i])
        assert one.state()["n_rows"] == rows[i]
        one.step()
        span = float(alone[0, :rows[i]].max() - alone[0, :rows[i]].min())
        assert (logits[i, :rows[i]] - alone[0, :rows[i]]).abs().max() <= TOL_BF16 * span, f"sequence {i}"
        one.close()
    h.close()


@pytest.mark.parametrize("n_seq", [2, 3, 5, 7, 13])
def test_batch_rows_have_the_bits_of_the_greedy_handle(weights, n_seq):
    """The split of k of a handle with several sequences does not follow the rows of its blocks: the first row of a step
    (the last committed token) has the same logits bit for bit in the greedy handle and with trees of every block size,
    128-row blocks that take two turns included."""
    prompts = [synth.make_prompt(BF16_SMALL.vocab, 30 + 7 * i, 20 + i) for i in range(n_seq)]
    first = []
    for kw in (dict(n_probes=0, max_nodes=1), *(dict(n_probes=3, topk=5, max_nodes=n, expand_width=0, n_anchor=1) for n in (16, 40, 70, 110))):
        h, logits = _handle(weights, 400, P.spec_cfg(**kw), n_seq)
        for i in range(n_seq):
            h.prefill(prompts[i], i)
        P.esp_step(h.h, h.tokens_out, h.n_out)
        assert h.stats().device_error == 0
        first.append(logits[:, 0].clone())
        h.close()
    for f in first[1:]:
        assert torch.equal(f, first[0])


@pytest.mark.parametrize("group,n_rows,batch,L", [(4, 68, 3, 500), (2, 128, 5, 130), (1, 41, 24, 64), (8, 9, 70, 250), (4, 120, 8, 15)])
def test_attention_tail_of_large_launches_bitwise(group, n_rows, batch, L):
    """(Lengths for which the split grid does not follow the batch.)  The tail kernel of launches with many (row, head)
    pairs adds in the order of the one that takes a warp per pair: every sequence of a batch has the bits it has in a
    launch of its own, for every group size and ragged row counts."""
    Hkv = 8 if group > 1 else 16
    Hq, h, cap = Hkv * group, 128, L + R
    n_probes = min(4, n_rows - 1)
    _, depth1, vis = _tree_block(n_rows - n_probes, n_probes, 5, n_rows)
    g = torch.Generator(device="cuda").manual_seed(group)
    q = torch.randn(batch, R, Hq, h, generator=g, device="cuda").bfloat16()
    kc, vc = (torch.randn(batch, Hkv, cap, h, generator=g, device="cuda").bfloat16() for _ in range(2))
    anc = np.stack([_anc_words(vis)] * batch)
    depth = np.zeros((batch, R), np.int32)
    depth[:, :n_rows] = depth1
    out = _run_attention(1, q, kc, vc, anc, depth, n_rows, L, Hq, Hkv, h)
    for s in (0, batch - 1):
        alone = _run_attention(1, q[s:s + 1].contiguous(), kc[s:s + 1].contiguous(), vc[s:s + 1].contiguous(), anc[:1], depth[:1],
                               n_rows, L, Hq, Hkv, h)
        assert torch.equal(out[s, :n_rows], alone[0, :n_rows]), f"sequence {s}"


@pytest.mark.parametrize("group,n_rows,batch,dcap", [(4, 68, 3, 32), (4, 128, 2, 128), (8, 41, 12, 48)])
def test_attention_tail_of_large_launches_with_deep_trees_bitwise(group, n_rows, batch, dcap):
    """More than 16 positions behind the root: tails of up to several 32-key chunks, in the instance that large launches take
    for them.  Every sequence has the bits of a launch of its own (one cache split, whatever the batch)."""
    Hkv, h, L = 8, 128, 250
    Hq, cap = Hkv * group, L + R
    vis = np.tril(np.ones((n_rows, n_rows), np.uint8)) if dcap == 128 else None
    if vis is None:
        _, depth1, vis = _tree_block(n_rows, 0, dcap, n_rows)
    else:
        depth1 = np.arange(n_rows)
    g = torch.Generator(device="cuda").manual_seed(dcap)
    q = torch.randn(batch, R, Hq, h, generator=g, device="cuda").bfloat16()
    kc, vc = (torch.randn(batch, Hkv, cap, h, generator=g, device="cuda").bfloat16() for _ in range(2))
    anc = np.stack([_anc_words(vis)] * batch)
    depth = np.zeros((batch, R), np.int32)
    depth[:, :n_rows] = depth1
    out = _run_attention(1, q, kc, vc, anc, depth, n_rows, L, Hq, Hkv, h, dcap)
    for s in (0, batch - 1):
        alone = _run_attention(1, q[s:s + 1].contiguous(), kc[s:s + 1].contiguous(), vc[s:s + 1].contiguous(), anc[:1], depth[:1],
                               n_rows, L, Hq, Hkv, h, dcap)
        # (a launch of 128 rows x 32 heads takes the same instance: checked against fp64 as well)
        assert torch.equal(out[s, :n_rows], alone[0, :n_rows]), f"sequence {s}"
    sc = torch.einsum("rhd,hcd->hrc", q[0, :n_rows].double(), kc[0].repeat_interleave(group, 0)[:, :L + n_rows].double()) / h ** 0.5
    hide = torch.zeros(n_rows, L + n_rows, dtype=torch.bool)
    hide[:, L:] = torch.from_numpy(vis == 0)
    ref = torch.einsum("hrc,hcd->rhd", sc.masked_fill_(hide.cuda(), -float("inf")).softmax(-1), vc[0].repeat_interleave(group, 0)[:, :L + n_rows].double())
    # bf16 probabilities of the chunks below the tail (2^-9 each, sums of at most their number) and the result's own rounding
    assert (out[0, :n_rows].double() - ref).abs().max() <= 2e-2


@pytest.mark.parametrize("group,n_rows,batch", [(4, 68, 3), (1, 120, 9)])
def test_attention_tail_of_large_launches_without_a_cache(group, n_rows, batch):
    """No cached position, so no bulk kernel in front of the tail kernel: it waits before it reads (the queries and keys come
    from the kernel in front of it), and every sequence has the bits of a launch of its own."""
    Hkv, h, L = 8, 128, 0
    Hq, cap = Hkv * group, R
    _, depth1, vis = _tree_block(n_rows, 0, 5, n_rows)
    g = torch.Generator(device="cuda").manual_seed(group)
    q = torch.randn(batch, R, Hq, h, generator=g, device="cuda").bfloat16()
    kc, vc = (torch.randn(batch, Hkv, cap, h, generator=g, device="cuda").bfloat16() for _ in range(2))
    anc = np.stack([_anc_words(vis)] * batch)
    depth = np.zeros((batch, R), np.int32)
    depth[:, :n_rows] = depth1
    out = _run_attention(1, q, kc, vc, anc, depth, n_rows, L, Hq, Hkv, h)
    for s in range(batch):
        alone = _run_attention(1, q[s:s + 1].contiguous(), kc[s:s + 1].contiguous(), vc[s:s + 1].contiguous(), anc[:1], depth[:1],
                               n_rows, L, Hq, Hkv, h)
        assert torch.equal(out[s, :n_rows], alone[0, :n_rows]), f"sequence {s}"


@pytest.mark.parametrize("group,n_rows,batch", [(4, 68, 16), (1, 128, 5), (8, 41, 12)])
def test_attention_tail_of_large_launches_rows_in_any_order(group, n_rows, batch):
    """The rows of the operator come in any order, so a row may stand before its ancestors, and its CTA has to fetch keys
    of rows that other CTAs work on (with the rows reversed the root is the last one): the bits and the clean status of a
    launch of its own, whose kernel takes every key from the cache."""
    Hkv, h, L = 8, 128, 250          # (one cache split, whatever the batch)
    Hq, cap = Hkv * group, L + R
    _, depth1, vis = _tree_block(n_rows - 3, 3, 5, n_rows)
    depth1, vis = depth1[::-1], vis[::-1, ::-1]
    g = torch.Generator(device="cuda").manual_seed(group)
    q = torch.randn(batch, R, Hq, h, generator=g, device="cuda").bfloat16()
    kc, vc = (torch.randn(batch, Hkv, cap, h, generator=g, device="cuda").bfloat16() for _ in range(2))
    anc = np.stack([_anc_words(vis)] * batch)
    depth = np.zeros((batch, R), np.int32)
    depth[:, :n_rows] = depth1
    out = _run_attention(1, q, kc, vc, anc, depth, n_rows, L, Hq, Hkv, h)
    for s in (0, batch - 1):
        alone = _run_attention(1, q[s:s + 1].contiguous(), kc[s:s + 1].contiguous(), vc[s:s + 1].contiguous(), anc[:1], depth[:1],
                               n_rows, L, Hq, Hkv, h)
        assert torch.equal(out[s, :n_rows], alone[0, :n_rows]), f"sequence {s}"


@pytest.mark.parametrize("n_seq,early", [(34, 33), (34, 32), (130, 129)])
def test_prefill_leaves_every_other_sequence_alone(weights, n_seq, early):
    """Prefilling one sequence changes nothing of another that is waiting, whatever their places in a large handle: length,
    draft tree, mask vectors and Top-K' lists stay, and its next step is that of a handle in which it was prefilled last."""
    spec = P.spec_cfg(n_probes=3, topk=5, max_nodes=16, expand_width=0, n_anchor=1)
    prompts = {early: synth.make_prompt(BF16_SMALL.vocab, 45, 1), 0: synth.make_prompt(BF16_SMALL.vocab, 130, 2)}
    seen = []
    for order in ((early, 0), (0, early)):
        h, logits = _handle(weights, 200, spec, n_seq)
        for i in order:
            h.prefill(prompts[i], i)
            if i == early:
                before = h.state(early)
        after = h.state(early)
        for key in before:
            assert np.array_equal(before[key], after[key]), key
        h.step(early)
        assert h.stats().device_error == 0
        seen.append((h.n_out.copy(), h.tokens_out[early].copy(), logits[early, :after["n_rows"]].clone()))
        h.close()
    assert np.array_equal(seen[0][0], seen[1][0]) and np.array_equal(seen[0][1], seen[1][1]) and torch.equal(seen[0][2], seen[1][2])


@pytest.mark.parametrize("n_seq,nodes,n_anchor", [(2, 16, 1), (3, 16, 1), (12, 16, 1), (5, 40, 1), (8, 60, 1), (4, 70, 1), (8, 70, 1), (13, 70, 1), (14, 70, 1),
                                                   (3, 110, 1), (5, 110, 1), (13, 25, 0)])
def test_rows_do_not_depend_on_who_else_takes_part(weights, n_seq, nodes, n_anchor):
    """A step in which some sequences of the handle are idle packs the others into row tiles of their own: every row has the
    bits it has when all take part, whoever is idle (the first, the last, all but one, every second), for every block size."""
    spec = P.spec_cfg(n_probes=3, topk=5, max_nodes=nodes, expand_width=0 if n_anchor else 1, n_anchor=n_anchor)
    prompts = [synth.make_prompt(BF16_SMALL.vocab, 17 + 40 * (i % 4), 30 + i) for i in range(n_seq)]
    everyone = list(range(n_seq))
    full = None
    for who in (everyone, [0], [n_seq - 1], [n_seq // 2], everyone[:-1], everyone[1:], everyone[::2], [0, n_seq - 1], everyone[1::2], everyone[1:3]):
        h, logits = _handle(weights, 300, spec, n_seq)
        for i in who:
            h.prefill(prompts[i], i)
        rows = {i: h.state(i)["n_rows"] for i in who}
        logits.zero_()
        P.esp_step(h.h, h.tokens_out, h.n_out)
        assert h.stats().device_error == 0 and [i for i in everyone if h.n_out[i]] == who
        if full is None:
            full = logits.clone()
        for i in who:
            assert torch.equal(logits[i, :rows[i]], full[i, :rows[i]]), f"{who}: sequence {i}"
        h.close()


def test_steps_of_a_partly_filled_handle_cost_what_takes_part():
    """One sequence of eight: the layer GEMMs and the LM head run over its block alone.  (Layers of 0.44 GB; the step took
    0.73 of the full one's time when a pass carried all of its blocks, 0.32 with the one that takes part.)"""
    shape = synth.LLAMA3_8B.replace(n_layers=2, vocab=8192)
    w = synth.make_weights(shape, 1, device="cuda")
    spec = P.spec_cfg(n_probes=4, topk=10, max_nodes=64, expand_width=0, n_anchor=1)
    us = []
    for who in (range(8), [3]):
        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        h = P.Handle(shape, spec, w, 700, 8, stream)
        for i in who:
            h.prefill(synth.make_prompt(shape.vocab, 100, i), i)
        best = 1e9
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            h.step()
            a.record(stream)
            for _ in range(10):
                h.step_async()
            b.record(stream)
            for _ in range(10):
                h.read()
            best = min(best, a.elapsed_time(b))
        us.append(best)
        h.close()
    assert us[1] < 0.55 * us[0]


def test_rows_have_the_bits_of_the_greedy_handle_in_every_instance(weights):
    """One sequence: the layer GEMMs load as many rows as the handle's blocks have, in steps of 8 to 16, and 128-row plans take
    the blocks of more than 80 rows; the split of k is the same in all of them, so the first row of a step has the bits it has in
    the greedy handle."""
    prompt = synth.make_prompt(BF16_SMALL.vocab, 150, 4)
    first = []
    for nodes in (0, 13, 14, 29, 30, 45, 46, 53, 61, 62, 69, 70, 77, 78, 93, 94, 109, 110, 125):
        kw = dict(n_probes=0, max_nodes=1) if not nodes else dict(n_probes=3, topk=10, max_nodes=nodes, expand_width=0, n_anchor=1)
        h, logits = _handle(weights, 400, P.spec_cfg(**kw))
        h.prefill(prompt)
        assert h.state()["n_rows"] == (nodes + 3 if nodes else 1)
        h.step()
        assert h.stats().device_error == 0
        first.append(logits[0, 0].clone())
        h.close()
    for f in first[1:]:
        assert torch.equal(f, first[0])


@pytest.mark.parametrize("d", [2056, 2944, 4096])
def test_a_row_normed_by_two_blocks_has_the_bits_of_one_block(d):
    """Rows of more than 2048 features: up to 74 of them are normed by a pair of blocks each, 75 by one block each (17, 23 and
    32 groups of 128; the first row of the step, bit for bit)."""
    shape = BF16_SMALL.replace(name="bf16-wide-rows", d_model=d, n_layers=2, n_q_heads=16, n_kv_heads=4, d_ffn=1376)
    w = synth.make_weights(shape, seed=4, device="cuda", gain_jitter=True, std=0.03)
    prompt = synth.make_prompt(shape.vocab, 60, 4)
    first = []
    for nodes in (72, 71, 13, 0):
        kw = dict(n_probes=0, max_nodes=1) if not nodes else dict(n_probes=3, topk=10, max_nodes=nodes, expand_width=0, n_anchor=1)
        h = P.Handle(shape, P.spec_cfg(**kw), w, max_seq_len=300, max_batch=1)
        logits = torch.zeros(1, R, shape.vocab, dtype=torch.float32, device="cuda")
        P.esp_debug_capture(h.h, logits)
        h.prefill(prompt)
        assert h.state()["n_rows"] == (nodes + 3 if nodes else 1)
        h.step()
        assert h.stats().device_error == 0 and torch.isfinite(logits[0, 0]).all()
        first.append(logits[0, 0].clone())
        h.close()
    assert first[0].abs().max() > 0
    for f in first[1:]:
        assert torch.equal(f, first[0])


def test_rows_of_two_sequences_normed_by_pairs_of_blocks():
    """Two sequences of up to 37 rows have their norms taken by a pair of blocks per row, of 38 by one block per row: the root rows' bits
    of both sequences are those of the greedy handle of as many sequences."""
    shape = BF16_SMALL.replace(name="bf16-wide-rows", d_model=2944, n_layers=2, n_q_heads=16, n_kv_heads=4, d_ffn=1376)
    w = synth.make_weights(shape, seed=4, device="cuda", gain_jitter=True, std=0.03)
    torch.cuda.synchronize()
    first = []
    for nodes in (0, 13, 34, 35):
        kw = dict(n_probes=0, max_nodes=1) if not nodes else dict(n_probes=3, topk=10, max_nodes=nodes, expand_width=0, n_anchor=1)
        h = P.Handle(shape, P.spec_cfg(**kw), w, max_seq_len=300, max_batch=2)
        logits = torch.zeros(2, R, shape.vocab, dtype=torch.float32, device="cuda")
        P.esp_debug_capture(h.h, logits)
        for i in range(2):
            h.prefill(synth.make_prompt(shape.vocab, 60 + i, 4 + i), i)
        assert all(h.state(i)["n_rows"] == (nodes + 3 if nodes else 1) for i in range(2))
        h.step()
        assert h.stats().device_error == 0 and torch.isfinite(logits[:, 0]).all()
        first.append(logits[:, 0].clone())
        h.close()
    assert (first[0][0] != first[0][1]).any()
    for f in first[1:]:
        assert torch.equal(f, first[0])
