"""Stage A of Algorithm 1 on the GPU (sdfp_fit_scores) against the CPU oracle's FIT scores, which
are themselves pinned by finite differences (tests/test_oracle_fit.py)."""
import threading

import numpy as np
import pytest
import torch

import paper_2602_05499_b200 as pkg
import synth_inputs as si
from oracle import fit
from oracle import sdfp_oracle as orc

pytestmark = pytest.mark.gpu


def _both(shape, w, calib):
    pkg.build_library()
    got_T, got_F = pkg.sdfp_fit_scores(shape, si.weights_to(w, "cuda:0"), calib)
    m = orc.Model.from_shape(shape, si.weights_to(w, "cpu"))
    ref_T, ref_F = fit.fit_scores(m, [list(map(int, r)) for r in calib])
    return got_T, got_F, ref_T, ref_F


def test_fit_scores_small_model_with_large_gradients():
    """The finite-difference test's model (weights x 10, so that every tensor's gradient is well
    above rounding), odd sizes: 2 layers, d 32, 2 heads x 16, FFN 40, vocabulary 50; sequences of
    12 tokens.  Every layer's trace and FIT value against the fp64 oracle: off by 2.4e-7 when measured
    (fp32 sums, two passes), four times that allowed."""
    shape = si.ModelShape("fd", 2, 32, 2, 16, 40, 50)
    w = si.make_weights(shape, [], random_gains=True)
    for lw in w["layers"]:
        for k in lw:
            if k.startswith("w"):
                lw[k] *= 10.0
    calib = si.make_prompts(shape.vocab, 3, 12, seed=7)
    got_T, got_F, ref_T, ref_F = _both(shape, w, calib)
    assert got_T == pytest.approx(ref_T, rel=1e-6)
    assert got_F == pytest.approx(ref_F, rel=1e-6)


@pytest.mark.parametrize("shape", [si.TINY, si.TINY_BF16])
def test_fit_scores_tiny_config_and_ranking(shape):
    """The tiny configuration (fp32 and bf16 storage), 8 calibration sequences of 32 tokens: scores
    against the oracle (off by 8e-8 when measured), the two down-scaled layers rank lowest (Algorithm 1 with r = 0.5 selects
    exactly them), and the result does not depend on the order of the calibration set."""
    w = si.make_weights(shape, (1, 2))
    calib = si.make_prompts(shape.vocab, 8, 32, seed=99)
    got_T, got_F, ref_T, ref_F = _both(shape, w, calib)
    assert got_T == pytest.approx(ref_T, rel=4e-7)
    assert got_F == pytest.approx(ref_F, rel=4e-7)
    assert fit.prune_set(got_F, 0.5) == [1, 2]
    assert max(got_F[1], got_F[2]) < 0.2 * min(got_F[0], got_F[3])
    again_T, again_F = pkg.sdfp_fit_scores(shape, si.weights_to(w, "cuda:0"), calib[::-1].copy())
    assert again_T == pytest.approx(got_T, rel=1e-12) and again_F == pytest.approx(got_F, rel=1e-12)
    same_T, _ = pkg.sdfp_fit_scores(shape, si.weights_to(w, "cuda:0"), calib)
    assert same_T == got_T                                   # run to run: bit-identical


@pytest.mark.parametrize("d,heads,ffn,vocab,n_seq,seq_len,dtype", [
    (32, 2, 40, 50, 3, 2, "f32"),        # one token per sequence, a vocabulary that is no multiple of 8
    (36, 2, 41, 64, 2, 34, "f32"),       # rows that are no whole 16-byte pieces, two Gram tiles with a remainder
    (128, 2, 264, 96, 11, 66, "bf16"),   # more rows than go through at a time: a full and a smaller group
    (136, 1, 72, 130, 1, 130, "bf16"),   # one head wider than a block, five Gram tiles, cut contractions
    (64, 4, 2048, 4096, 2, 18, "f32"),   # long contractions over few tiles: the widest split
    (256, 2, 4096, 2048, 4, 65, "f32"),  # contractions of thousands, wide tiles
])
def test_fit_scores_at_the_edges(d, heads, ffn, vocab, n_seq, seq_len, dtype):
    """Tile remainders, unaligned rows, groups of sequences and split contractions against the fp64 oracle.  Off by
    2.9e-7 at most when measured (the random walk of fp32 sums of up to 4096 terms, two passes); four times that is allowed, so
    that a GEMM of fewer bits shows."""
    shape = si.ModelShape("edge", 2, d, heads, d // heads, ffn, vocab, dtype=dtype)
    w = si.make_weights(shape, [], random_gains=True)
    for lw in w["layers"]:
        for k in lw:
            if k.startswith("w"):
                lw[k] *= 4.0
    calib = si.make_prompts(shape.vocab, n_seq, seq_len, seed=5)
    got_T, got_F, ref_T, ref_F = _both(shape, w, calib)
    assert got_T == pytest.approx(ref_T, rel=1.2e-6)
    assert got_F == pytest.approx(ref_F, rel=1.2e-6)
    back_T, _ = pkg.sdfp_fit_scores(shape, si.weights_to(w, "cuda:0"), calib[::-1].copy())
    assert back_T == pytest.approx(got_T, rel=1e-12)   # nor on where in the set a sequence stands


def test_fit_scores_on_two_threads_with_different_lengths():
    """Calls on other threads, of other sequence lengths, do not disturb one another: a long sequence's launches go
    through, and to the same bits, while a second thread scores sequences of a few tokens."""
    pkg.build_library()
    shape = si.ModelShape("threads", 8, 64, 1, 64, 80, 64)
    w = si.weights_to(si.make_weights(shape, []), "cuda:0")
    long_set, short_set = si.make_prompts(shape.vocab, 4, 1501, seed=1), si.make_prompts(shape.vocab, 2, 5, seed=2)
    want = pkg.sdfp_fit_scores(shape, w, long_set)
    stop, errors = threading.Event(), []

    def score_short():
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                while not stop.is_set():
                    pkg.sdfp_fit_scores(shape, w, short_set)
        except Exception as e:  # noqa: BLE001 (reported by the test's own thread)
            errors.append(e)

    other = threading.Thread(target=score_short)
    other.start()
    try:
        for _ in range(20):
            assert pkg.sdfp_fit_scores(shape, w, long_set) == want
    finally:
        stop.set()
        other.join()
    assert not errors


def test_fit_scores_give_their_memory_back():
    """What a call holds when it returns, before anything else synchronises: nothing of a working set above 256 MB, at most
    256 MB of a smaller one, and that until sdfp_fit_release or the end of a context."""
    pkg.build_library()
    small, large = si.ModelShape("small", 2, 64, 1, 64, 80, 64), si.ModelShape("large", 2, 64, 1, 64, 80, 1 << 17)
    w_small, w_large = (si.weights_to(si.make_weights(m, []), "cuda:0") for m in (small, large))
    sets = {m.name: si.make_prompts(m.vocab, 2, 600, seed=1) for m in (small, large)}  # large: 599 x 131072 logits, 314 MB
    keep = 256 << 20

    def kept(call):
        call()                         # kernels and device tables loaded
        pkg.sdfp_fit_release()
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        call()
        return before - torch.cuda.mem_get_info()[0], before

    assert kept(lambda: pkg.sdfp_fit_scores(large, w_large, sets["large"]))[0] <= 0
    held, before = kept(lambda: pkg.sdfp_fit_scores(small, w_small, sets["small"]))
    assert 0 < held <= keep
    pkg.sdfp_fit_release()
    assert torch.cuda.mem_get_info()[0] == before
    eng = pkg.Sdfp(si.TINY, si.weights_to(si.make_weights(si.TINY, []), "cuda:0"), max_seq=64)
    pkg.sdfp_fit_scores(small, w_small, sets["small"])
    eng.close()
    pkg.sdfp_fit_scores(small, w_small, sets["small"])
    pkg.sdfp_fit_release()
    pkg.sdfp_fit_release()             # nothing left: no error


def test_fit_scores_do_not_depend_on_free_memory():
    """With room for only some of the sequences at a time the scores have the same bits as with room for all: 8 sequences
    of 64 tokens need 537 MB of logits, half of them fit into what a hold on the rest of the device leaves."""
    pkg.build_library()
    shape = si.ModelShape("memory", 3, 64, 1, 64, 336, 1 << 18)
    w = si.weights_to(si.make_weights(shape, []), "cuda:0")
    calib = si.make_prompts(shape.vocab, 9, 65, seed=3)  # a full group of eight and one more
    want = pkg.sdfp_fit_scores(shape, w, calib)
    pkg.sdfp_fit_release()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (420 << 20), dtype=torch.uint8, device="cuda:0")
    try:
        assert pkg.sdfp_fit_scores(shape, w, calib) == want
    finally:
        del hold
        torch.cuda.empty_cache()
        pkg.sdfp_fit_release()


def test_fit_scores_drive_the_draft_mask():
    """Stage A feeding Stage B: the prune set chosen from the GPU scores is handed to
    sdfp_set_draft_layers and the speculative output stays the target's."""
    shape = si.TINY
    w = si.make_weights(shape, (1, 2))
    calib = si.make_prompts(shape.vocab, 8, 32, seed=99)
    _, F = pkg.sdfp_fit_scores(shape, si.weights_to(w, "cuda:0"), calib)
    skip = fit.prune_set(F, 0.5)
    assert skip == [1, 2]
    eng = pkg.Sdfp(shape, si.weights_to(w, "cuda:0"), max_seq=128, k_max=4)
    try:
        eng.sdfp_set_draft_layers(si.keep_mask(shape.n_layers, skip))
        prompt = si.make_prompts(shape.vocab, 1, 16)
        out = eng.sdfp_generate(prompt, 4, 32)
        assert out.tokens == eng.sdfp_generate(prompt, 0, 32).tokens
        assert out.acceptance_rate > 0.15
    finally:
        eng.close()


def test_fit_scores_rejects_bad_arguments():
    shape = si.TINY
    w = si.weights_to(si.make_weights(shape, (1, 2)), "cuda:0")
    with pytest.raises(pkg.SdfpError):
        pkg.sdfp_fit_scores(shape, w, np.full((2, 8), shape.vocab, dtype=np.int32))     # token out of range
    with pytest.raises(pkg.SdfpError):
        pkg.sdfp_fit_scores(shape, w, np.zeros((2, 1), dtype=np.int32))                 # nothing to predict
