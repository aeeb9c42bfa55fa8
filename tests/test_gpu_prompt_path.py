"""Prompt passes at the row counts where their kernels change: the decode projections up to 128 rows, above that row tiles cut into
equal multiples of 16 and up to eight parts along K."""
import numpy as np
import pytest
import torch

from helpers import as_bf16_values, check_stream_against_oracle, gpu_model, new_stream, require_gpu, top2_margin
from oracle.anpd import argmax_lowest
from oracle.decoder import Decoder
from workloads import ModelShape, make_weights, markov_prompt

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def A():
    require_gpu()
    from paper_2404_08698_b200 import binding
    return binding


@pytest.fixture(scope="module", params=[ModelShape(2, 1024, 8, 8, 128, 2816, 1000), ModelShape(2, 1024, 16, 2, 64, 1400, 1000)], ids=["hd128", "hd64g8"])
def rig(A, request):
    shape = request.param
    w = make_weights(shape, 23, False, std=0.025)
    m = gpu_model(A, shape, w, new_stream())
    kv = A.anpd_kv_create(m, 640)
    yield shape, m, kv, Decoder(shape, as_bf16_values(w), torch.float64, kv_dtype=torch.bfloat16)
    A.anpd_kv_destroy(kv)
    A.anpd_model_destroy(m)


# 9: two groups of 8; 121 / 129: 128 rows on the decode projections, 136 on the prompt GEMM; 257: two tiles of 144 rows where one of
# 256 would be a row short; 513: three; one handle for all, so that every cut follows another
@pytest.mark.parametrize("plen", [9, 64, 121, 128, 129, 200, 256, 257, 513, 15])
def test_prompt_logits_at_row_tile_edges(A, rig, plen):
    shape, m, kv, dec = rig
    prompt = markov_prompt(plen, shape.vocab, 2, 300 + plen).tolist()
    draft = [int(t) for t in markov_prompt(7, shape.vocab, 2, 301 + plen)]
    A.anpd_kv_truncate(kv, 0, 0)
    first = A.anpd_prefill(m, kv, prompt)
    got = torch.from_numpy(A.anpd_verify_logits(m, kv, first, draft, shape.vocab)).double()
    cache = dec.new_cache()
    lp = dec.forward(prompt, cache)
    if top2_margin(lp[-1]) > 5e-2:
        assert first == argmax_lowest(lp[-1])
    want = dec.forward([first] + draft, cache)
    # the two sides round the same cache to bf16; what is left is fp32 sums of two-term products (2^-17 of a term) and cache
    # entries that round the other way (2^-9 of an entry, one in hundreds): well below 2^-9 of the logits' scale
    err = float((got - want).abs().max())
    assert err <= 2 ** -8 * max(1.0, float(want.abs().max())), err


# rows per sequence: a group of 8 (as many rows as a step has: not to be taken for one), over it, over a tile of 32 and of 128 rows;
# five sequences of 600 do not fit one pass of 2048 rows, three of 1030 take a pass each
@pytest.mark.parametrize("hd,group", [(64, 4), (128, 1)])
@pytest.mark.parametrize("batch,plen", [(3, 5), (4, 16), (8, 8), (2, 41), (5, 139), (5, 600), (3, 1030)])
def test_prompts_of_several_sequences_share_a_pass(A, batch, plen, hd, group):
    shape = ModelShape(2, 256, 2 * group, 2, hd, 520, 300)
    w = make_weights(shape, 29, False, std=0.04)
    st = new_stream()
    m = gpu_model(A, shape, w, st)
    kv = A.anpd_kv_create(m, plen + 24, batch, 1)
    ctxs = [A.anpd_ngram_create(2, 3, plen + 24, 0, st) for _ in range(batch)]
    dec = Decoder(shape, as_bf16_values(w), torch.float64, kv_dtype=torch.bfloat16)
    prompts = np.stack([markov_prompt(plen, shape.vocab, 2, 400 + plen + b) for b in range(batch)])
    try:
        out, _ = A.anpd_generate_batch(m, kv, ctxs, prompts, 4, 3)
        greedy, _ = A.anpd_generate_batch(m, kv, ctxs, prompts, 4, 0)
        assert np.array_equal(out, greedy)
        checked = sum(check_stream_against_oracle(dec, prompts[b].tolist(), out[b].tolist()) for b in range(batch))
        assert checked >= 2
    finally:
        for c in ctxs:
            A.anpd_ngram_destroy(c)
        A.anpd_kv_destroy(kv)
        A.anpd_model_destroy(m)


# The gate-up projection finishes the activations of tiles that are not cut along K: all cut (twice), none cut and a ragged end, more tiles
# than SMs (the last, partly filled round cut in two: 213 tiles of 256 features x 176 rows); residual rows of more than 1024 chunks of
# four: one over, the most of two chunks per thread with two rows to an SM, one over that and 8192 (two chunks where there is an SM per row,
# 144 rows, four beyond, 200), one over 8192
@pytest.mark.parametrize("d,F,plen", [(256, 136, 129), (512, 1400, 300), (2048, 9000, 513), (4104, 136, 140), (6144, 136, 140), (6152, 136, 140), (8200, 136, 140),
                                      (512, 1400, 1100), (6152, 136, 200), (8192, 136, 140), (8192, 136, 200)])
def test_prompt_logits_at_feature_tile_and_row_width_edges(A, d, F, plen):
    shape = ModelShape(1, d, 2, 2, 128, F, 500)
    w = make_weights(shape, 31, False, std=0.02)
    m = gpu_model(A, shape, w, new_stream())
    kv = A.anpd_kv_create(m, plen + 16)
    try:
        test_prompt_logits_at_row_tile_edges(A, (shape, m, kv, Decoder(shape, as_bf16_values(w), torch.float64, kv_dtype=torch.bfloat16)), plen)
    finally:
        A.anpd_kv_destroy(kv)
        A.anpd_model_destroy(m)


# whole tiles of gate-up, finished by the projection: an odd number of 16-row chunks, a last tile's chunks that are partly or not there
@pytest.mark.parametrize("plen", [129, 150, 182, 340, 393])
def test_gate_up_tiles_finished_by_the_projection(A, plen):
    shape = ModelShape(2, 256, 2, 2, 128, 9608, 300)               # (the second layer reads every row of the first)
    w = make_weights(shape, 31, False, std=0.03)
    m = gpu_model(A, shape, w, new_stream())
    kv = A.anpd_kv_create(m, plen + 16)
    prompt = markov_prompt(plen, shape.vocab, 2, 500 + plen).tolist()
    draft = [int(t) for t in markov_prompt(7, shape.vocab, 2, 501 + plen)]
    try:
        first = A.anpd_prefill(m, kv, prompt)
        got = torch.from_numpy(A.anpd_verify_logits(m, kv, first, draft, shape.vocab)).double()
    finally:
        A.anpd_kv_destroy(kv)
        A.anpd_model_destroy(m)
    dec = Decoder(shape, as_bf16_values(w), torch.float64, kv_dtype=torch.bfloat16)
    cache = dec.new_cache()
    lp = dec.forward(prompt, cache)
    if top2_margin(lp[-1]) > 5e-2:
        assert first == argmax_lowest(lp[-1])
    want = dec.forward([first] + draft, cache)
    err = float((got - want).abs().max())
    assert err <= 2 ** -8 * max(1.0, float(want.abs().max())), err          # (the bound of the row tile edges above)
