"""Forms of a call that the boundary accepts and that depend on where or when it is made: weights anywhere in a larger buffer, a
handle that has seen other calls, n-gram calls behind a greedy loop."""
import numpy as np
import pytest
import torch

from helpers import gpu_model, new_stream, require_gpu
from workloads import ModelShape, make_weights, markov_prompt

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def A():
    require_gpu()
    from paper_2404_08698_b200 import binding
    return binding


def _prompt_and_logits(A, shape, m, kv, n=40):
    prompt = markov_prompt(n, shape.vocab, 2, 31).tolist()
    A.anpd_kv_truncate(kv, 0, 0)
    first = A.anpd_prefill(m, kv, prompt)
    return first, A.anpd_verify_logits(m, kv, first, [3, 9, 4], shape.vocab)


# device matrices at 2, 8 and 14 bytes behind a 16-byte boundary; 0 beside them
@pytest.mark.parametrize("bf16", [True, False])
@pytest.mark.parametrize("offset", [0, 1, 4, 7])
def test_device_weights_at_any_element_of_a_buffer(A, offset, bf16):
    shape = ModelShape(2, 64, 2, 1, 64, 96, 160)
    w = make_weights(shape, 3, bf16, std=0.08)

    def inside(t):
        if t.dim() != 2:
            return t.cuda()
        flat = torch.zeros(t.numel() + 16, dtype=t.dtype, device="cuda")
        at = flat[offset:offset + t.numel()].view(t.shape)
        at.copy_(t)
        assert (at.data_ptr() - offset * t.element_size()) % 16 == 0
        return at

    got = []
    for form in ({k: v.cuda() for k, v in w.items()}, {k: inside(v) for k, v in w.items()}):
        torch.cuda.synchronize()
        m = gpu_model(A, shape, form, new_stream())
        kv = A.anpd_kv_create(m, 128)
        got.append(_prompt_and_logits(A, shape, m, kv))
        A.anpd_kv_destroy(kv)
        A.anpd_model_destroy(m)
    assert got[0][0] == got[1][0]
    assert np.array_equal(got[0][1], got[1][1])


# widths whose last k-block of 64 is part empty: the residual stream's, the FFN's, both
@pytest.mark.parametrize("d,f", [(72, 128), (64, 96), (72, 96)])
def test_an_overflow_stays_with_its_call(A, d, f):
    """A prompt with a token whose FFN activations overflow, then ordinary calls of other row counts on the same handle: bit for bit
    what a handle gives that has not seen it.  The token's keys and values are overwritten by the second prompt."""
    shape = ModelShape(2, d, 1, 1, 64, f, 160)
    w = make_weights(shape, 7, False, std=0.08)
    bad, dim = 100, 5
    w["embed"][:, dim] = 0.0
    w["embed"][bad, dim] = 1.0
    w["l0.wo"][dim] = 0.0                                       # the dimension is the token's alone where layer 0 reads it
    w["l0.w_gate"][:, dim] = 1e25
    w["l0.w_up"][:, dim] = 1e25
    good = [t if t != bad else 3 for t in markov_prompt(80, shape.vocab, 2, 12).tolist()]
    m = gpu_model(A, shape, w, new_stream())
    used, fresh = A.anpd_kv_create(m, 128), A.anpd_kv_create(m, 128)
    try:
        A.anpd_prefill(m, used, good[:3] + [bad] + good[4:])    # 80 rows
        assert not np.isfinite(A.anpd_verify_logits(m, used, 3, [5], shape.vocab)).all()
        got = []
        for kv in (used, fresh):
            A.anpd_kv_truncate(kv, 0, 0)
            first = A.anpd_prefill(m, kv, good[:40])            # 40 rows
            got.append((first, A.anpd_verify_logits(m, kv, 3, [5, 9], shape.vocab)))
        assert np.isfinite(got[1][1]).all()
        assert got[0][0] == got[1][0] and np.array_equal(got[0][1], got[1][1])
    finally:
        A.anpd_kv_destroy(used)
        A.anpd_kv_destroy(fresh)
        A.anpd_model_destroy(m)


# the first call after a greedy loop finds prompt and output unfolded: more than a call's one block takes
@pytest.mark.parametrize("first", ["update", "draft"])
def test_ngram_calls_after_a_greedy_loop(A, first):
    shape = ModelShape(1, 64, 1, 1, 64, 96, 160)
    st = new_stream()
    m = gpu_model(A, shape, make_weights(shape, 9, False, std=0.08), st)
    n, new = 700, 20
    kv = A.anpd_kv_create(m, n + new + 32)
    got, want = (A.anpd_ngram_create(2, 5, n + new + 64, 0, st) for _ in range(2))
    prompt = markov_prompt(n, shape.vocab, 2, 44)
    more = [7, 8, 9]
    try:
        tokens = np.append(prompt, A.anpd_generate(m, kv, want, prompt, new + 1, 0)[0])
        A.anpd_generate(m, kv, got, prompt, new, 0)             # its context ends with the token behind the output
        assert A.anpd_ngram_len(got) == len(tokens)
        A.anpd_launch_count(True)
        d = A.anpd_ngram_draft(got, 5) if first == "draft" else A.anpd_ngram_update(got, more)
        assert A.anpd_launch_count() == 3                       # the two bulk passes, and the call's kernel
        A.anpd_ngram_reset(want)
        A.anpd_ngram_update(want, tokens)
        if first == "draft":
            assert A.anpd_ngram_draft(want, 5) == d
            A.anpd_ngram_update(got, more)
        A.anpd_ngram_update(want, more)
        for level in range(2, 6):
            assert A.anpd_ngram_dump(want, level) == A.anpd_ngram_dump(got, level)
            assert A.anpd_ngram_dump_best(want, level) == A.anpd_ngram_dump_best(got, level)
    finally:
        for c in (got, want):
            A.anpd_ngram_destroy(c)
        A.anpd_kv_destroy(kv)
        A.anpd_model_destroy(m)
