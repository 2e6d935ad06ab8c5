"""Rounds of small decoders inside one thread-block cluster (csrc/cluster_pass.cuh) at the edges of its shares, steps and splits."""
import time

import numpy as np
import pytest

import paper_2602_05499_b200 as pkg
import synth_inputs as si
from gpu_common import check_stream_against_oracle, make_pair
from oracle import sdfp_oracle as orc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads,head_dim,ffn,vocab,dtype,prompt,k", [
    (2, 64, 64, 16, "f32", 1, 3),        # the smallest shares: four pairs per CTA, CTAs without a token of the vocabulary; a draft row in front of the text
    (2, 64, 64, 16, "bf16", 300, 4),     # ... K of half a step; four CTAs per head
    (3, 128, 528, 400, "f32", 200, 4),   # shares of different size, a ragged last K step, CTAs without a head; blocks of four keys
    (3, 128, 1040, 400, "bf16", 60, 8),  # ... 9 rows: a second sweep of the weights
    (7, 64, 1200, 272, "bf16", 90, 0),   # several steps and batches of pairs per warp
    (17, 64, 80, 272, "bf16", 20, 0),    # more heads than CTAs
])
def test_greedy_rounds_at_the_edges(heads, head_dim, ffn, vocab, dtype, prompt, k):
    """One launch for all rounds; every token is the oracle's choice given the tokens before it (near-ties of bf16 within
    1e-2 as everywhere; fp32 within 1e-3, five times the logit error that 1e-4 in 2-norm can put on one of these vocabularies),
    and speculative and autoregressive decoding agree."""
    shape = si.ModelShape("edge", 3, heads * head_dim, heads, head_dim, ffn, vocab, dtype=dtype)
    eng, m, _ = make_pair(shape, (1,), max_seq=prompt + 40 + k, k_max=k, random_gains=True)
    try:
        text = si.make_prompts(vocab, 1, prompt, seed=31)
        out = eng.sdfp_generate(text, k, 36)
        assert out.timing["kernel_launches"] == 1 and len(out.tokens[0]) == 36
        assert eng.sdfp_generate(text, 0, 36).tokens == out.tokens
        check_stream_against_oracle(m, text[0].tolist(), out.tokens[0], gap_tol=1e-3 if dtype == "f32" else 1e-2)
        if k and dtype == "f32":
            ref = orc.spec_generate(orc.CachedLM(m, max_seq=prompt + 60), orc.CachedLM(m, orc.keep_layers(3, (1,)), max_seq=prompt + 60),
                                    text[0].tolist(), k, 36)
            if ref.tokens == out.tokens[0]:  # no near-tie among them: the same drafts were accepted
                assert [int(a) for a in out.stats[:, 0, 1]] == [r.accepted for r in ref.rounds]
    finally:
        eng.close()


@pytest.mark.parametrize("dtype,batch,k,prompt", [("f32", 1, 4, 1), ("bf16", 3, 4, 70), ("bf16", 4, 2, 9), ("bf16", 8, 0, 2), ("f32", 4, 0, 33)])
def test_rounds_of_a_batch(dtype, batch, k, prompt):
    """speculative == autoregressive == one sequence alone, with the draft's own cache and with the target's; the sequences are
    teacher-forced with the oracle; sampled decoding with the full model as its own draft accepts everything."""
    shape = si.TINY if dtype == "f32" else si.TINY_BF16
    eng, m, _ = make_pair(shape, (1, 2), max_seq=prompt + 40, max_batch=batch, k_max=k)
    try:
        prompts = si.make_prompts(m.vocab, batch, prompt, seed=50 + batch)
        out = eng.sdfp_generate(prompts, k, 24)
        assert out.timing["kernel_launches"] == 1
        ar = eng.sdfp_generate(prompts, 0, 24)
        assert ar.tokens == out.tokens and all(len(t) == 24 for t in out.tokens)
        assert np.array_equal(out.stats[:, :, 2].sum(axis=0), np.full(batch, 24))
        solo = eng.sdfp_generate(prompts[-1:], k, 24)
        assert solo.tokens[0] == out.tokens[-1]
        for b in (0, batch - 1):
            check_stream_against_oracle(m, prompts[b].tolist(), out.tokens[b])
        if k:
            eng.sdfp_set_draft_kv_sharing(True)
            assert eng.sdfp_generate(prompts, k, 24).tokens == out.tokens
            eng.sdfp_set_draft_kv_sharing(False)
            eng.sdfp_set_draft_layers(np.ones(shape.n_layers, dtype=np.uint8))
            s = eng.sdfp_generate(prompts, k, 20, temperature=1.0, seed=5)
            assert (s.stats[:-1, 0, 1] == k).all()
    finally:
        eng.close()


@pytest.mark.parametrize("heads,head_dim,ffn,vocab,dtype,batch,k,new", [
    (2, 64, 64, 16, "f32", 1, 3, 90),       # draft rows in front of the text, two chunks of keys
    (4, 64, 688, 528, "f32", 1, 8, 40),     # nine rows
    (3, 128, 528, 400, "f32", 2, 0, 150),
    (2, 64, 64, 16, "bf16", 1, 3, 90),      # k-classes and CTAs without a unit, half a tile per CTA
    (4, 64, 688, 528, "bf16", 1, 8, 40),    # two column groups; sums in three pieces
    (4, 64, 688, 2048, "bf16", 2, 2, 140),
    (3, 128, 1040, 400, "bf16", 1, 5, 70),
    (8, 64, 1376, 4096, "bf16", 1, 0, 600),  # ten chunks: the first splits walk two
])
def test_rounds_have_the_bits_of_the_other_passes(heads, head_dim, ffn, vocab, dtype, batch, k, new):
    """Keys and values that rounds leave in either cache, the tokens they choose and the counts they accept are those of the
    kernels that run prompts and sdfp_forward_logits: logits behind a generated text are, bit for bit, the ones of the same
    text fed from its first token, and every token is the first largest of its row.  A text goes on the same in a second call."""
    shape = si.ModelShape("bits", 4, heads * head_dim, heads, head_dim, ffn, vocab, dtype=dtype)
    eng, m, _ = make_pair(shape, (1, 2), max_seq=new + k + 8, max_batch=batch, k_max=k, random_gains=True)
    try:
        first = si.make_prompts(vocab, batch, 1, seed=61)
        out = eng.sdfp_generate(first, k, new)
        assert out.timing["kernel_launches"] == 1
        text = first[0].tolist() + list(out.tokens[0])
        tail = 12  # (behind a round the caches hold all keys in front of the last token)
        for draft in ([False, True] if k else [False]):
            got = eng.sdfp_forward_logits(text[-tail:-1], len(text) - tail, draft=draft)
            whole = np.concatenate([eng.sdfp_forward_logits(text[i:i + 80], i, draft=draft) for i in range(0, len(text) - 1, 80)])[:len(text) - 1]
            assert np.array_equal(got.view(np.uint32), whole[-tail + 1:].view(np.uint32))
            if not draft:
                assert text[1:] == [int(np.argmax(row)) for row in whole]
        if batch == 1:
            half = new // 2
            if dtype == "f32" or half + 1 <= 16:  # (longer bf16 prompts run on the tcgen05 path)
                on = eng.sdfp_generate(np.asarray([text[:1 + half]], dtype=np.int32), k, new - half)
                assert on.tokens[0] == out.tokens[0][half:]
        if k:  # drafted tokens are the draft's first largest
            eng.sdfp_set_draft_layers(np.ones(shape.n_layers, dtype=np.uint8))
            assert (eng.sdfp_generate(first, k, 20).stats[:-1, :, 1] == k).all()
    finally:
        eng.close()


@pytest.mark.parametrize("shape,prompt,temperature", [(si.TINY, 1, 0.0), (si.TINY, 30, 0.0), (si.TINY_BF16, 1, 0.0), (si.TINY_BF16, 24, 0.0), (si.TINY_BF16, 1, 1.0)])
def test_a_wait_that_runs_out(shape, prompt, temperature):
    """The cluster kernel's own waits, without faulting anything: every CTA's first one expects more bytes than are sent, with a 20 ms
    limit.  (The prompts have no pass that would take the hook: one token, per-operation kernels, or long enough for the tcgen05
    path.)  The CTAs walk to their end, the call comes back with SDFP_ETIMEOUT and the wait's name, the context works again."""
    eng, _, _ = make_pair(shape, (1, 2), max_seq=96, max_batch=1, k_max=4)
    try:
        text = si.make_prompts(shape.vocab, 1, prompt, seed=91)
        before = eng.sdfp_generate(text, 4, 24, temperature=temperature, seed=3)
        for _ in range(2):
            eng.sdfp_debug_expire_next_wait(20_000_000)
            t0 = time.perf_counter()
            with pytest.raises(pkg.SdfpError) as ei:
                eng.sdfp_generate(text, 4, 24, temperature=temperature, seed=3)
            assert time.perf_counter() - t0 < 1.0
            assert ei.value.code == -5 and "in the cluster" in str(ei.value)
            after = eng.sdfp_generate(text, 4, 24, temperature=temperature, seed=3)
            assert after.tokens == before.tokens and np.array_equal(after.stats, before.stats)
    finally:
        eng.close()


@pytest.mark.parametrize("shape", [si.TINY, si.TINY_BF16], ids=["f32", "bf16"])
def test_the_flag_that_leaves_the_cluster_kernel_out(shape):
    """Greedy and sampled rounds on the kernels of every other pass: the same tokens, statistics and, from the caches they leave, logits."""
    prompts = si.make_prompts(shape.vocab, 2, 9, seed=67)
    got = []
    for flags in (0, pkg.FLAG_NO_CLUSTER):
        eng, _, _ = make_pair(shape, (1, 2), max_seq=96, max_batch=1, k_max=5, flags=flags, random_gains=True)
        greedy = eng.sdfp_generate(prompts[:1], 5, 70)
        logits = [eng.sdfp_forward_logits(greedy.tokens[0][-9:], 70, draft=draft).view(np.uint32) for draft in (False, True)]
        sampled = eng.sdfp_generate(prompts[1:], 5, 60, temperature=1.0, seed=9)
        got.append((greedy, sampled, logits))
        eng.close()
    (a, sa, la), (b, sb, lb) = got
    assert a.timing["kernel_launches"] == 1 < b.timing["kernel_launches"]
    assert a.tokens == b.tokens and sa.tokens == sb.tokens and np.array_equal(a.stats, b.stats) and np.array_equal(sa.stats, sb.stats)
    assert all(np.array_equal(x, y) for x, y in zip(la, lb))


@pytest.mark.parametrize("d,vocab,dtype,max_seq,batch,k,inside", [
    (256, 4096, "bf16", 96, 1, 4, True), (256, 4096, "f32", 96, 1, 4, True), (512, 4096, "bf16", 96, 1, 4, True),
    (512, 32000, "bf16", 96, 1, 4, False),    # measured 0.76 of the whole-pass kernel's speed
    (256, 32000, "f32", 96, 1, 4, False),     # 0.86
    (256, 32000, "bf16", 96, 1, 0, True),     # 1.4
    (512, 4096, "bf16", 2080, 1, 8, False),   # 0.78
    (256, 4096, "bf16", 2080, 1, 8, True),    # 1.2
    (256, 4096, "bf16", 2080, 4, 0, False),   # 0.80
    (384, 4096, "f32", 2080, 1, 4, False),    # 0.65
    (640, 4096, "bf16", 96, 1, 4, False),     # 0.92
    (512, 4096, "f32", 96, 1, 0, True),       # 1.03
])
def test_which_decoders_run_inside_a_cluster(d, vocab, dtype, max_seq, batch, k, inside):
    """The line takes the size of the vocabulary, the positions and the sequences of a call into account, not a layer's weights alone."""
    shape = si.ModelShape("line", 4, d, d // 64, 64, 16 * int(d * 2.7 / 16), vocab, dtype=dtype)
    eng, m, _ = make_pair(shape, (1, 2), max_seq=max_seq, max_batch=batch, k_max=k, draw_device="cuda:0")
    try:
        out = eng.sdfp_generate(si.make_prompts(vocab, batch, max_seq - 20, seed=5), k, 10)
        assert (out.timing["kernel_launches"] == 1) == inside
    finally:
        eng.close()


@pytest.mark.parametrize("flags", [0, pkg.FLAG_NO_CLUSTER], ids=["cluster", "whole-pass"])
def test_an_end_token(flags):
    """A sequence that ends early stays where it is while the other goes on; calls behind it start afresh."""
    eng, m, _ = make_pair(si.TINY_BF16, (1, 2), max_seq=64, max_batch=2, k_max=4, flags=flags)
    prompts = si.make_prompts(m.vocab, 2, 12, seed=77)
    free = eng.sdfp_generate(prompts, 4, 30)
    eng.close()
    eos = free.tokens[0][7]
    eng, _, _ = make_pair(si.TINY_BF16, (1, 2), max_seq=64, max_batch=2, k_max=4, eos_id=int(eos), flags=flags)
    try:
        for k in (4, 0):
            out = eng.sdfp_generate(prompts, k, 30)
            assert (out.timing["kernel_launches"] == 1) == (flags == 0)
            for b in range(2):
                want = free.tokens[b]
                cut = want.index(eos) + 1 if eos in want else len(want)
                assert out.tokens[b] == want[:cut]
    finally:
        eng.close()


def test_a_logit_that_is_not_a_number_hides_no_other():
    """fp32, one row of the lm-head not numbers: its neighbour in the pair (eight rows on), often the largest, is still chosen, as on the
    kernels of every other pass."""
    shape = si.TINY
    w = si.make_weights(shape, (1, 2))
    w["lm_head"][0] = float("nan")
    w["lm_head"][8] *= 40.0
    got = []
    for flags in (0, pkg.FLAG_NO_CLUSTER):
        eng = pkg.Sdfp(shape, si.weights_to(w, "cuda:0"), max_seq=64, k_max=4, flags=flags)
        eng.sdfp_set_draft_layers(si.keep_mask(shape.n_layers, (1, 2)))
        outs = [eng.sdfp_generate(si.make_prompts(shape.vocab, 1, 5, seed=s), 4, 12) for s in range(4)]
        assert all((o.timing["kernel_launches"] == 1) == (flags == 0) for o in outs)
        got.append([o.tokens[0] for o in outs])
        eng.close()
    assert got[0] == got[1] and any(8 in t for t in got[0])
