"""A single sequence's step as one kernel (csrc/step_cl.cu) against the same step as a kernel per projection: the same sums in the same
order, so equal bit for bit.  The chain of kernels is held to the oracle by the other tests."""
import numpy as np
import pytest

from helpers import gpu_model, new_stream, require_gpu
from workloads import ModelShape, make_weights, markov_prompt

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def A():
    require_gpu()
    from paper_2404_08698_b200 import binding
    return binding


# head dimension and heads per kv head: every instance; widths: fewest k-blocks and units there may be, tails of a k-block in every
# projection, several tiles per projection, one segment (kb >= 64), a vocabulary that is no multiple of anything; four, two and one CTAs per head
@pytest.mark.parametrize("shape", [
    ModelShape(1, 256, 4, 4, 64, 256, 256), ModelShape(3, 328, 6, 3, 64, 904, 1037), ModelShape(2, 2048, 32, 4, 64, 5632, 3200),
    ModelShape(2, 512, 40, 40, 64, 1000, 5000), ModelShape(2, 1024, 8, 8, 128, 2816, 3000), ModelShape(2, 4096, 32, 8, 128, 11008, 32000),
    ModelShape(3, 1024, 80, 80, 64, 512, 700),
], ids=lambda s: f"{s.n_layers}x{s.d_model}h{s.n_q_heads}-{s.n_kv_heads}-{s.head_dim}")
def test_one_kernel_equals_a_kernel_per_projection(A, monkeypatch, shape):
    m = gpu_model(A, shape, make_weights(shape, 21, True), new_stream())
    prompt = markov_prompt(1160, shape.vocab, 2, 31).tolist()
    draft = [5, 9, 2, 7, 30, 77, 4]
    try:
        got, launches = [], []
        for chain in (True, False):
            if chain:
                monkeypatch.setenv("ANPD_STEP_CHAIN", "1")
            else:
                monkeypatch.delenv("ANPD_STEP_CHAIN")
            kv = A.anpd_kv_create(m, 1200, 1, True)                    # shuffled pages
            res, n_launch = [], 0
            for n in (1, 8, 121, 125, 128, 250, 512, 1150):            # the step's rows before, on and behind the edges of a page
                A.anpd_kv_truncate(kv, 0, 0)
                last = A.anpd_prefill(m, kv, prompt[:n])
                A.anpd_launch_count(True)
                for k in (7, 0, 3):                                    # commits shift the next step's rows; the second layer's buffers serve again
                    res.append(A.anpd_verify_logits(m, kv, last, draft[:k], shape.vocab))
                    res.append(np.array(A.anpd_verify(m, kv, last, draft[:k])))
                    last = int(res[-1][1])
                res.append(np.array(A.anpd_verify_two_candidates(m, kv, last, [1, 2], [3, 4, 5])[:3]))
                n_launch += A.anpd_launch_count()
            got.append(res)
            launches.append(n_launch)
            A.anpd_kv_destroy(kv)
    finally:
        A.anpd_model_destroy(m)
    assert launches[1] < launches[0]                                   # the path under test really ran
    for a, b in zip(*got):
        assert np.array_equal(a, b)
