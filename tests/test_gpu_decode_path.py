"""The decode step's own kernels at the sizes where they can go wrong: projections split over clusters (fused exchange for one
sequence, partial sums for several) and the attention over shares of the key pages."""
import numpy as np
import pytest
import torch

from helpers import as_bf16_values, check_stream_against_oracle, gpu_model, new_stream, require_gpu
from oracle.decoder import Decoder
from workloads import ModelShape, make_weights, markov_prompt
from workloads.rng import normal_tensor

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def A():
    require_gpu()
    from paper_2404_08698_b200 import binding
    return binding


# N: fewer groups of 8 than clusters, ragged, one feature over a group, one group over a tile, several passes (40000);
# K: fewer k-blocks than CTAs of a cluster, tails; rows: one sequence, two, an odd count, the most
@pytest.mark.parametrize("N,K,rows", [
    (8, 64, 8), (30, 72, 8), (257, 192, 8), (300, 200, 8), (4096, 256, 8), (4104, 4096, 8), (32000, 512, 8), (40000, 128, 8),
    (30, 72, 16), (512, 512, 128), (1000, 2048, 128), (704, 320, 40), (4352, 640, 64), (27648, 640, 64), (1024, 4096, 24), (33000, 192, 16),
])
def test_projection_matches_fp64_product(A, N, K, rows):
    w = normal_tensor(N * 7 + K, 1, N * K, 0.05).view(N, K).to(torch.bfloat16)
    a = normal_tensor(N + K * 3, 2, rows * K, 1.0).view(rows, K)
    a[0, :] = 0.0
    a[1, 0] = 1000.0
    want = a.double() @ w.double().T
    scale = float(want.abs().max()) + 1e-6
    got = torch.from_numpy(A.anpd_debug_gemm(w, a.numpy(), plain=3)).double()
    # hi + lo carries about 16 mantissa bits: 2e-5, the bar of the other projection kernels
    assert float((got - want).abs().max()) <= 2e-5 * scale + 1e-6
    assert float(got[0].abs().max()) == 0.0


# one sequence, 5 to 8 k-blocks per CTA (one activation slot; all weights in the ring with few features), 4 and 9 beside them;
# an SM of its own (many features) with more k-blocks than one slot of 8 holds; half an SM with more than 8, steps of 4, 2 and 1 k-blocks
@pytest.mark.parametrize("N,K", [(64, 1024), (64, 1088), (300, 1344), (2560, 2048), (2816, 2000), (5640, 2048), (700, 2056), (12296, 2200), (1000, 2600), (2048, 5632), (4096, 4104)])
def test_projection_slots_of_one_sequence(A, N, K):
    test_projection_matches_fp64_product(A, N, K, 8)


@pytest.mark.parametrize("rows", [8, 64])
def test_projection_rows_are_independent(A, rows):
    N, K = 1536, 1024
    w = normal_tensor(15, 1, N * K, 0.05).view(N, K).to(torch.bfloat16)
    a = normal_tensor(16, 2, rows * K, 1.0).view(rows, K).numpy()
    full = A.anpd_debug_gemm(w, a, plain=3)
    other = a.copy()
    other[1:] = 0.0
    alone = A.anpd_debug_gemm(w, other, plain=3)
    assert np.array_equal(full[0], alone[0]) and float(np.abs(alone[1:]).max()) == 0.0


# (head_dim, query heads per kv head): every instance of the attention kernel; head dimension 128 with grouped heads takes the
# page-wise kernels
@pytest.mark.parametrize("hd,group", [(64, 1), (64, 2), (64, 4), (64, 8), (128, 1), (128, 2)])
def test_decode_logits_at_block_page_and_share_edges(A, hd, group):
    """Contexts around a block of 16 keys, a page of 128, a share's pair of pages (256), a round of the shares (1024)."""
    shape = ModelShape(1, 64, 2 * group, 2, hd, 96, 160)
    w = make_weights(shape, 5, False, std=0.08)
    dec = Decoder(shape, as_bf16_values(w), torch.float64, kv_dtype=torch.bfloat16)
    m = gpu_model(A, shape, w, new_stream())
    kv = A.anpd_kv_create(m, 1400, 1, 1)                       # shuffled pages
    prompt = markov_prompt(1290, shape.vocab, 2, 17).tolist()
    draft = [5, 9, 2, 7, 30, 77, 4]
    try:
        for n in (1, 7, 8, 9, 16, 23, 121, 127, 128, 129, 250, 256, 380, 511, 1020, 1024, 1290):
            A.anpd_kv_truncate(kv, 0, 0)
            A.anpd_prefill(m, kv, prompt[:n])
            cache = dec.new_cache()
            dec.forward(prompt[:n], cache)
            want = dec.forward([3] + draft, cache)
            got = torch.from_numpy(A.anpd_verify_logits(m, kv, 3, draft, shape.vocab)).double()
            # activations and weights carry about 16 mantissa bits, the cache's bf16 rounding is the oracle's own: what is left
            # are values that round to the neighbouring bf16 number in the cache (2^-8 of one key or value)
            err = float((got - want).abs().max())
            assert err <= 5e-3 * max(1.0, float(want.abs().max())), (n, err)
    finally:
        A.anpd_kv_destroy(kv)
        A.anpd_model_destroy(m)


@pytest.mark.parametrize("hkv,group,batch", [(16, 1, 8), (8, 8, 16), (2, 4, 3)])
def test_batched_streams_against_the_oracle(A, hkv, group, batch):
    """Enough heads for one CTA per head (128), and few (a cluster per head); ragged acceptance over a page boundary."""
    shape = ModelShape(2, 64, hkv * group, hkv, 64, 96, 160)
    w = make_weights(shape, 6, False, std=0.08)
    dec = Decoder(shape, as_bf16_values(w), torch.float64, kv_dtype=torch.bfloat16)
    st = new_stream()
    m = gpu_model(A, shape, w, st)
    n, new = 120, 14
    kv = A.anpd_kv_create(m, n + new + 24, batch, 1)
    ctxs = [A.anpd_ngram_create(2, 4, n + new + 24, 0, st) for _ in range(batch)]
    prompts = np.stack([markov_prompt(n, shape.vocab, 2, 100 + b) for b in range(batch)])
    try:
        out, _ = A.anpd_generate_batch(m, kv, ctxs, prompts, new, 5)
        greedy, _ = A.anpd_generate_batch(m, kv, ctxs, prompts, new, 0)
        assert np.array_equal(out, greedy)
        checked = sum(check_stream_against_oracle(dec, prompts[b].tolist(), out[b].tolist()) for b in (0, batch - 1))
        assert checked >= 4
    finally:
        for c in ctxs:
            A.anpd_ngram_destroy(c)
        A.anpd_kv_destroy(kv)
        A.anpd_model_destroy(m)
