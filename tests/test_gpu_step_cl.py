"""A single sequence's step as one kernel (csrc/step_cl.cu) against the same step as a kernel per projection, which the other tests
hold to the oracle."""
import time
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest
import torch

from helpers import gpu_model, new_stream, require_gpu
from workloads import ModelShape, make_weights, markov_prompt

pytestmark = pytest.mark.gpu

DRAFT = [5, 9, 2, 7, 30, 77, 4]


@pytest.fixture(scope="module")
def A():
    require_gpu()
    from paper_2404_08698_b200 import binding
    return binding


def _both(A, monkeypatch, shape, run, stream=None, max_len=1200, weights=None):
    """run(kv) on a handle of either kind: its results, and the kernels it launched."""
    m = gpu_model(A, shape, weights or make_weights(shape, 21, True), stream or new_stream())
    got, launches = [], []
    try:
        for chain in (True, False):
            if chain:
                monkeypatch.setenv("ANPD_STEP_CHAIN", "1")
            else:
                monkeypatch.delenv("ANPD_STEP_CHAIN")
            kv = A.anpd_kv_create(m, max_len, 1, True)                 # shuffled pages
            A.anpd_launch_count(True)
            got.append(run(m, kv))
            launches.append(A.anpd_launch_count())
            A.anpd_kv_destroy(kv)
    finally:
        A.anpd_model_destroy(m)
    assert launches[1] < launches[0]                                   # the path under test really ran
    return got


def _id(s):
    return f"{s.n_layers}x{s.d_model}h{s.n_q_heads}-{s.n_kv_heads}-{s.head_dim}"


# Fewest k-blocks and units there may be, tails of a k-block in every projection, several tiles per projection, one segment (kb >= 64), a
# vocabulary that is no multiple of anything; four and two CTAs per head; a layer of few copies (no prefetch) and of many.
@pytest.mark.parametrize("shape", [
    ModelShape(1, 256, 4, 4, 64, 256, 256), ModelShape(3, 328, 6, 6, 64, 904, 1037), ModelShape(2, 512, 40, 40, 64, 1000, 5000),
    ModelShape(2, 4096, 32, 8, 128, 11008, 32000),
], ids=_id)
def test_the_same_sums_in_the_same_order(A, monkeypatch, shape):
    prompt = markov_prompt(1160, shape.vocab, 2, 31).tolist()

    def run(m, kv):
        res = []
        for n in (1, 8, 121, 125, 128, 250, 512, 1150):                # the step's rows before, on and behind the edges of a page
            A.anpd_kv_truncate(kv, 0, 0)
            last = A.anpd_prefill(m, kv, prompt[:n])
            for k in (7, 0, 3):                                        # commits shift the next step's rows; the exchange buffers serve again
                res.append(A.anpd_verify_logits(m, kv, last, DRAFT[:k], shape.vocab))
                res.append(np.array(A.anpd_verify(m, kv, last, DRAFT[:k])))
                last = int(res[-1][1])
            res.append(np.array(A.anpd_verify_two_candidates(m, kv, last, [1, 2], [3, 4, 5])[:3]))
        return res

    for a, b in zip(*_both(A, monkeypatch, shape, run)):
        assert np.array_equal(a, b)


# Two and four k-blocks of the residual projections in one product (64 and 32 features per cluster), with a stage that is not full; two tiles
# of the residual stream; query heads of dimension 64 that share a kv head; one CTA per head.
@pytest.mark.parametrize("shape", [
    ModelShape(1, 2048, 32, 4, 64, 5632, 3200), ModelShape(1, 1024, 8, 8, 128, 2824, 3000), ModelShape(1, 1024, 80, 80, 64, 512, 700),
    ModelShape(1, 512, 8, 2, 64, 1376, 1000), ModelShape(1, 5120, 40, 40, 128, 1024, 500),
], ids=_id)
def test_sums_in_another_order(A, monkeypatch, shape):
    prompt = markov_prompt(1160, shape.vocab, 2, 31).tolist()

    def run(m, kv):
        res = []
        for n in (9, 121, 128, 512, 1150):
            A.anpd_kv_truncate(kv, 0, 0)
            A.anpd_prefill(m, kv, prompt[:n])
            res.append(A.anpd_verify_logits(m, kv, 3, DRAFT, shape.vocab))
        return res

    for a, b in zip(*_both(A, monkeypatch, shape, run)):
        # fp32 sums of two-term products (2^-17 of a term) in another order, through one layer whose cached keys and values are the same
        assert float(np.abs(a - b).max()) <= 2.0 ** -12 * max(1.0, float(np.abs(a).max()))


# Words that are all ones mean "not written yet" between the CTAs: infinities and NaN of that pattern go through a step like any other value.
@pytest.mark.parametrize("where", ["embed", "l1.attn_norm", "l1.ffn_norm", "final_norm", "l0.wv"])
@pytest.mark.parametrize("shape", [ModelShape(3, 328, 6, 6, 64, 904, 1037), ModelShape(2, 512, 4, 4, 128, 1000, 5000)], ids=_id)
def test_infinities_and_nan(A, monkeypatch, shape, where):
    w = make_weights(shape, 21, True)
    ones = {2: torch.tensor([-1], dtype=torch.int16).view(torch.bfloat16), 4: torch.tensor([-1], dtype=torch.int32).view(torch.float32)}
    t = w[where]
    if where == "embed":
        t[7, 3], t[9, 4:6], t[2, 5] = float("inf"), ones[2], float("-inf")
    elif t.dim() == 2:
        t[5, 11] = float("inf")
    else:
        t[8:10], t[17] = ones[4], float("-inf")

    def run(m, kv):
        res = []
        for n in (3, 126, 300):
            A.anpd_kv_truncate(kv, 0, 0)
            A.anpd_prefill(m, kv, markov_prompt(n, shape.vocab, 2, 31).tolist())
            for k in (7, 0, 3):                                        # the rows' keys and values stay in the cache
                res.append(A.anpd_verify_logits(m, kv, 3, DRAFT[:k], shape.vocab))
                A.anpd_verify(m, kv, 3, DRAFT[:k])
        return res

    chain, one = _both(A, monkeypatch, shape, run, weights=w)
    assert any(np.isnan(a).any() for a in chain)
    for a, b in zip(chain, one):
        assert np.array_equal(a, b, equal_nan=True)


# Two-tile and packed projections and grouped heads of dimension 64 over several layers: the step's results against the chain's.  A layer
# changes what it is given by no more than rounding; sums in another order differ by 2^-17 of a term, of which the residual stream holds three per layer.
@pytest.mark.parametrize("shape", [ModelShape(4, 2048, 32, 4, 64, 5632, 3200), ModelShape(3, 5120, 40, 40, 128, 1024, 500)], ids=_id)
def test_several_layers_in_another_order(A, monkeypatch, shape):
    prompt = markov_prompt(600, shape.vocab, 2, 31).tolist()

    def run(m, kv):
        res = []
        for n in (9, 128, 590):
            A.anpd_kv_truncate(kv, 0, 0)
            A.anpd_prefill(m, kv, prompt[:n])
            for k in (7, 2, 7):
                res.append(A.anpd_verify_logits(m, kv, 3, DRAFT[:k], shape.vocab))
        return res

    for a, b in zip(*_both(A, monkeypatch, shape, run)):
        # the step's own keys and values are rounded to bf16: a sum next to a boundary falls to either side, 2^-8 of that one element
        assert float(np.abs(a - b).max()) <= 2.0 ** -9 * max(1.0, float(np.abs(a).max()))


# A page of head dimension 128 is four stages of the ring, of ten, nine and eight stages here: which stage of an earlier page lies where a
# stage goes differs from page to page.  A dozen pages per CTA, and one CTA for all of a head's.
@pytest.mark.parametrize("shape, n", [
    (ModelShape(2, 256, 2, 2, 128, 688, 300), 6000), (ModelShape(2, 256, 2, 2, 128, 688, 16000), 6000), (ModelShape(2, 256, 2, 2, 128, 688, 32000), 6000),
    (ModelShape(1, 1024, 80, 10, 128, 1024, 300), 2000),
], ids=["10", "9", "8", "one-cta"])
def test_many_pages_through_a_short_ring(A, monkeypatch, shape, n):
    prompt = markov_prompt(n, shape.vocab, 2, 31).tolist()

    def run(m, kv):
        last = A.anpd_prefill(m, kv, prompt)
        return [A.anpd_verify_logits(m, kv, last, DRAFT[:i % 8], shape.vocab) for i in range(50)]

    for a, b in zip(*_both(A, monkeypatch, shape, run, max_len=n + 16)):
        # 1024 wide: sums in another order, with the bound above; else bit for bit
        assert np.array_equal(a, b) if shape.d_model == 256 else float(np.abs(a - b).max()) <= 2.0 ** -12 * max(1.0, float(np.abs(a).max()))


# What one step leaves in the exchange buffers, the next must not find: many steps, of one layer (its down projection writes what the same
# layer sets back) and of the fewest that alternate between the copies.
@pytest.mark.parametrize("shape", [
    ModelShape(1, 256, 4, 4, 64, 256, 256), ModelShape(1, 4096, 32, 32, 128, 1024, 500), ModelShape(2, 256, 2, 2, 128, 4096, 300),
], ids=_id)
def test_many_steps_one_after_the_other(A, monkeypatch, shape):
    prompt = markov_prompt(200, shape.vocab, 2, 31).tolist()
    stream = new_stream()

    def run(m, kv):
        ctx = A.anpd_ngram_create(2, 4, 1200, 0, stream)
        res = []
        for n, K in ((3, 0), (200, 5)):                                # one launch for all steps
            res.append(A.anpd_generate(m, kv, ctx, prompt[:n], 900, K)[0])
        A.anpd_ngram_destroy(ctx)
        A.anpd_kv_truncate(kv, 0, 0)
        last = A.anpd_prefill(m, kv, prompt)
        for i in range(60):
            res.append(A.anpd_verify_logits(m, kv, last, DRAFT[:i % 8], shape.vocab))
            res.append(np.array(A.anpd_verify(m, kv, last, DRAFT[:i % 3])))
            last = int(res[-1][1])
        return res

    for a, b in zip(*_both(A, monkeypatch, shape, run, stream)):
        assert np.array_equal(a, b)


# The handle of a model that takes more shared memory than the one whose handle is made after it, in either instance of the kernel (223488 and
# 217344 bytes, 224512 and 219392).
@pytest.mark.parametrize("first, second", [
    (ModelShape(2, 512, 40, 40, 64, 1000, 5000), ModelShape(1, 256, 4, 4, 64, 256, 256)),
    (ModelShape(1, 1024, 8, 8, 128, 2824, 3000), ModelShape(2, 512, 4, 4, 128, 1376, 1000)),
], ids=["hd64", "hd128"])
def test_handles_of_two_models_do_not_disturb_each_other(A, first, second):
    def steps(m, kv, vocab):                                           # the first step is launched, the others replay a graph
        A.anpd_kv_truncate(kv, 0, 0)
        last = A.anpd_prefill(m, kv, [1, 2, 3])
        return [A.anpd_verify_logits(m, kv, last, DRAFT[:k], vocab) for k in (0, 5, 5)]

    models, kvs, want = [], [], []
    try:
        for shape in (first, second):
            models.append(gpu_model(A, shape, make_weights(shape, 21, True), new_stream()))
            kv = A.anpd_kv_create(models[-1], 256)
            want.append(steps(models[-1], kv, shape.vocab))            # alone
            A.anpd_kv_destroy(kv)
        kvs = [A.anpd_kv_create(m, 256) for m in models]
        for _ in range(2):
            for m, kv, shape, alone in zip(models, kvs, (first, second), want):
                assert all(np.array_equal(x, y) for x, y in zip(steps(m, kv, shape.vocab), alone))
    finally:
        for kv in kvs:
            A.anpd_kv_destroy(kv)
        for m in models:
            A.anpd_model_destroy(m)


def test_two_models_step_at_the_same_time(A):
    """Either model's kernel needs most of the GPU: on two streams, from two threads, they take turns."""
    shapes = [ModelShape(3, 512, 8, 8, 64, 1376, 2000), ModelShape(2, 1024, 8, 8, 128, 2816, 3000)]
    models, kvs = [], []
    try:
        for shape in shapes:
            models.append(gpu_model(A, shape, make_weights(shape, 21, True), new_stream()))
            kvs.append(A.anpd_kv_create(models[-1], 512))

        def steps(i):
            res = []
            for _ in range(20):
                A.anpd_kv_truncate(kvs[i], 0, 0)
                last = A.anpd_prefill(models[i], kvs[i], [1, 2, 3])
                for k in range(30):                                    # the first are launched, the others replay a graph
                    res.append(A.anpd_verify_logits(models[i], kvs[i], last, DRAFT[:k % 8], shapes[i].vocab))
                    last = A.anpd_verify(models[i], kvs[i], last, DRAFT[:k % 3])[1]
            return res

        alone = [steps(i) for i in range(2)]
        with ThreadPoolExecutor(2) as pool:
            together = list(pool.map(steps, range(2)))
        for a, b in zip(alone, together):
            assert all(np.array_equal(x, y) for x, y in zip(a, b))
    finally:
        for kv in kvs:
            A.anpd_kv_destroy(kv)
        for m in models:
            A.anpd_model_destroy(m)


# A step whose inputs never come ends by itself, soon, and with an error that stays with its handle.
@pytest.mark.parametrize("shape", [
    ModelShape(2, 256, 4, 4, 64, 256, 256), ModelShape(16, 2048, 16, 16, 128, 2048, 8000),
], ids=_id)
def test_a_step_that_hears_nothing(A, shape):
    m = gpu_model(A, shape, make_weights(shape, 21, True), new_stream())
    kvs = [A.anpd_kv_create(m, 600) for _ in range(2)]
    try:
        last = [A.anpd_prefill(m, kv, markov_prompt(500, shape.vocab, 2, 31).tolist()) for kv in kvs][0]
        want = [A.anpd_verify_logits(m, kv, last, DRAFT, shape.vocab) for kv in kvs][0]
        t0 = time.perf_counter()
        with pytest.raises(A.AnpdError, match="209"):
            A.anpd_debug_lost_step(m, kvs[0])
        assert time.perf_counter() - t0 < 20.0                         # 2^21 polls, and what is left of the step
        with pytest.raises(A.AnpdError, match="209"):
            A.anpd_verify_logits(m, kvs[0], last, DRAFT, shape.vocab)
        assert np.array_equal(A.anpd_verify_logits(m, kvs[1], last, DRAFT, shape.vocab), want)
    finally:
        for kv in kvs:
            A.anpd_kv_destroy(kv)
        A.anpd_model_destroy(m)


def test_a_kernel_per_projection_under_nsight_compute(A, monkeypatch):
    """A profiler that runs launches again does not get a kernel whose CTAs wait for one another."""
    shape = ModelShape(1, 256, 4, 4, 64, 256, 256)
    m = gpu_model(A, shape, make_weights(shape, 21, True), new_stream())
    launches = []
    try:
        for var in ("ANPD_STEP_CHAIN", "NV_COMPUTE_PROFILER_PERFWORKS_DIR"):
            with monkeypatch.context() as env:
                env.delenv("NV_COMPUTE_PROFILER_PERFWORKS_DIR", raising=False)
                env.setenv(var, "1")
                kv = A.anpd_kv_create(m, 64)
            last = A.anpd_prefill(m, kv, [1, 2, 3])
            A.anpd_launch_count(True)
            A.anpd_verify(m, kv, last, DRAFT[:3])
            launches.append(A.anpd_launch_count())
            A.anpd_kv_destroy(kv)
    finally:
        A.anpd_model_destroy(m)
    assert launches[0] == launches[1]


def test_the_one_kernel_elsewhere(A, monkeypatch):
    """The shape of the test above, with neither variable: fewer kernels than with either."""
    monkeypatch.delenv("NV_COMPUTE_PROFILER_PERFWORKS_DIR", raising=False)
    shape = ModelShape(1, 256, 4, 4, 64, 256, 256)
    _both(A, monkeypatch, shape, lambda m, kv: [A.anpd_verify(m, kv, A.anpd_prefill(m, kv, [1, 2, 3]), DRAFT[:3])])
