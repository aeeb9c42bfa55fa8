"""Device memory of a kv handle: what its passes use, not the widest output times the most rows."""
import numpy as np
import pytest
import torch

from helpers import gpu_model, new_stream, require_gpu
from workloads import ModelShape, make_weights, markov_prompt

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module")
def A():
    require_gpu()
    from paper_2404_08698_b200 import binding
    return binding


def _taken(make):
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    kv = make()
    return before - torch.cuda.mem_get_info()[0], kv


def test_the_vocabulary_does_not_size_the_prompt_passes(A):
    """Sixteen short sequences: prompt passes of 2048 rows, a vocabulary of 32000 for 128 of them."""
    shape = ModelShape(1, 256, 4, 4, 64, 688, 32000)
    m = gpu_model(A, shape, make_weights(shape, 1, True), new_stream())
    taken, kv = _taken(lambda: A.anpd_kv_create(m, 128, 16))
    A.anpd_kv_destroy(kv)
    A.anpd_model_destroy(m)
    # four partial sums and the logits of 128 rows: 82 MB; the passes' activations and sums at widths up to 1376: 60 MB
    assert taken < 160 * MB, taken // MB


def test_long_contexts_keep_no_page_partials_of_prompt_rows(A):
    shape = ModelShape(1, 1024, 16, 16, 64, 2816, 1000)
    m = gpu_model(A, shape, make_weights(shape, 1, True), new_stream())
    taken, kv = _taken(lambda: A.anpd_kv_create(m, 4096, 1))
    A.anpd_kv_destroy(kv)
    A.anpd_model_destroy(m)
    # cache 17 MB, activations of 2048 rows 56 MB, two sums of 2048 x 5632 92 MB (page partials of 2048 rows: 277 MB more)
    assert taken < 220 * MB, taken // MB


def test_a_handle_without_room_for_joint_prompts_takes_them_one_by_one(A):
    shape = ModelShape(1, 64, 1, 1, 64, 65536, 160)
    st = new_stream()
    m = gpu_model(A, shape, make_weights(shape, 4, True, std=0.08), st)
    batch, n, new = 16, 100, 8
    ctxs = [A.anpd_ngram_create(2, 3, 160, 0, st) for _ in range(batch)]
    prompts = np.stack([markov_prompt(n, shape.vocab, 2, 70 + b) for b in range(batch)])
    got, fill = [], None
    try:
        for full in (False, True):
            if full:
                torch.cuda.synchronize()
                fill = torch.empty(torch.cuda.mem_get_info()[0] - 900 * MB, dtype=torch.uint8, device="cuda")
            taken, kv = _taken(lambda: A.anpd_kv_create(m, n + new + 20, batch))
            got.append((A.anpd_generate_batch(m, kv, ctxs, prompts, new, 3)[0], taken))
            A.anpd_kv_destroy(kv)
        assert got[0][1] > 900 * MB > got[1][1]
        # the pass's row count chooses how its sums are cut: equal but for near-ties
        assert np.mean(got[0][0] == got[1][0]) > 0.9
    finally:
        del fill
        torch.cuda.empty_cache()
        for c in ctxs:
            A.anpd_ngram_destroy(c)
        A.anpd_model_destroy(m)
