"""Decode attention of head dimension 128 where several query heads share a kv head: a cluster of CTAs per query head."""
import numpy as np
import pytest
import torch

from helpers import as_bf16_values, check_stream_against_oracle, gpu_model, new_stream, require_gpu
from oracle.decoder import Decoder
from workloads import ModelShape, make_weights, markov_prompt

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def A():
    require_gpu()
    from paper_2404_08698_b200 import binding
    return binding


@pytest.mark.parametrize("group", [2, 4, 8])
def test_logits_at_page_and_share_edges(A, group):
    """Contexts around a page of 128, two pages, a round of the four shares and a second one; kv heads of their own keys."""
    shape = ModelShape(1, 64, 3 * group, 3, 128, 96, 160)
    w = make_weights(shape, 5, False, std=0.08)
    dec = Decoder(shape, as_bf16_values(w), torch.float64, kv_dtype=torch.bfloat16)
    m = gpu_model(A, shape, w, new_stream())
    kv = A.anpd_kv_create(m, 1100, 1, 1)
    prompt = markov_prompt(1030, shape.vocab, 2, 17).tolist()
    draft = [5, 9, 2, 7, 30, 77, 4]
    try:
        for n in (1, 15, 120, 121, 128, 250, 257, 511, 520, 1030):
            A.anpd_kv_truncate(kv, 0, 0)
            A.anpd_prefill(m, kv, prompt[:n])
            cache = dec.new_cache()
            dec.forward(prompt[:n], cache)
            want = dec.forward([3] + draft, cache)
            got = torch.from_numpy(A.anpd_verify_logits(m, kv, 3, draft, shape.vocab)).double()
            # both sides round the cache to bf16; what is left are entries that round the other way (2^-8 of one key or value)
            err = float((got - want).abs().max())
            assert err <= 5e-3 * max(1.0, float(want.abs().max())), (n, err)
    finally:
        A.anpd_kv_destroy(kv)
        A.anpd_model_destroy(m)


# enough heads for one CTA each, and few; two candidates (slots and masks of their own) with one sequence
@pytest.mark.parametrize("hkv,group,batch", [(2, 8, 9), (1, 4, 3), (2, 2, 1)])
def test_streams_against_the_oracle(A, hkv, group, batch):
    shape = ModelShape(2, 64, hkv * group, hkv, 128, 96, 160)
    w = make_weights(shape, 6, False, std=0.08)
    dec = Decoder(shape, as_bf16_values(w), torch.float64, kv_dtype=torch.bfloat16)
    st = new_stream()
    m = gpu_model(A, shape, w, st)
    n, new = 120, 14
    kv = A.anpd_kv_create(m, n + new + 24, batch, 1)
    ctxs = [A.anpd_ngram_create(2, 4, n + new + 24, 0, st) for _ in range(batch)]
    prompts = np.stack([markov_prompt(n, shape.vocab, 2, 100 + b) for b in range(batch)])
    try:
        greedy, _ = A.anpd_generate_batch(m, kv, ctxs, prompts, new, 0)
        for candidates in (1, 2):
            A.anpd_kv_set_candidates(kv, candidates)
            out, _ = A.anpd_generate_batch(m, kv, ctxs, prompts, new, 5)
            assert np.array_equal(out, greedy)
        checked = sum(check_stream_against_oracle(dec, prompts[b].tolist(), greedy[b].tolist()) for b in {0, batch - 1})
        assert checked >= 4
    finally:
        for c in ctxs:
            A.anpd_ngram_destroy(c)
        A.anpd_kv_destroy(kv)
        A.anpd_model_destroy(m)


@pytest.mark.parametrize("hd,group", [(64, 1), (64, 2), (64, 8), (128, 1), (128, 4)])
def test_page_partials_on_mma_sync_cross_check_the_step_kernel(A, monkeypatch, hd, group):
    """The same step through the page-wise kernel and its merge (one launch more per layer).  One layer: both read the same cache."""
    shape = ModelShape(1, 64, 2 * group, 2, hd, 96, 160)
    w = make_weights(shape, 8, False, std=0.08)
    m = gpu_model(A, shape, w, new_stream())
    prompt = markov_prompt(300, shape.vocab, 2, 18).tolist()
    got, launches = [], []
    try:
        for sync in (False, True):
            if sync:
                monkeypatch.setenv("ANPD_ATTN_MMA_SYNC", "1")
            kv = A.anpd_kv_create(m, 400, 1, 1)
            A.anpd_prefill(m, kv, prompt)
            A.anpd_launch_count(True)
            got.append(A.anpd_verify_logits(m, kv, 3, [5, 9, 2, 7], shape.vocab))
            launches.append(A.anpd_launch_count())
            A.anpd_kv_destroy(kv)
    finally:
        A.anpd_model_destroy(m)
    assert launches[1] == launches[0] + 1
    # fp32 sums of two-term products (2^-17 of a term) in another order, through one layer
    assert float(np.abs(got[0] - got[1]).max()) <= 2.0 ** -12 * max(1.0, float(np.abs(got[0]).max()))
