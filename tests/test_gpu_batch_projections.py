"""Projections of several sequences' steps as a stream-K sweep over the model's storage: long contractions from 32 rows on."""
import numpy as np
import pytest
import torch

from helpers import as_bf16_values, gpu_model, new_stream, require_gpu
from oracle.decoder import Decoder
from workloads import ModelShape, make_weights, markov_prompt
from workloads.rng import normal_tensor

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def A():
    require_gpu()
    from paper_2404_08698_b200 import binding
    return binding


# one segment with a full last tile, with a part-filled one, with one group over a tile; K tail; 20 groups per cluster: a segment each,
# tiles across their seams; the widths of the 7B model; rows: the fewest, no multiple of 16, the most
@pytest.mark.parametrize("N,K,rows", [
    (4096, 4096, 32), (4000, 4096, 40), (4104, 4104, 104), (4200, 4160, 128), (5120, 4096, 64), (5112, 13824, 72),
    (22016, 4096, 128), (32000, 4096, 56), (4096, 11008, 64),
])
def test_product_matches_fp64(A, N, K, rows):
    w = normal_tensor(N * 7 + K, 1, N * K, 0.05).view(N, K).to(torch.bfloat16)
    a = normal_tensor(N + K * 3, 2, rows * K, 1.0).view(rows, K)
    a[0, :] = 0.0
    a[1, 0] = 1000.0
    got = torch.from_numpy(A.anpd_debug_gemm(w, a.numpy(), plain=3)).double()
    pick = torch.unique(torch.cat([torch.arange(0, N, max(1, N // 1500)), torch.arange(max(0, N - 140), N)]))       # and all of the last tile
    want = a.double() @ w[pick].double().T
    # hi + lo carries about 16 mantissa bits: 2e-5, the bar of the other projection kernels
    assert float((got[:, pick] - want).abs().max()) <= 2e-5 * (float(want.abs().max()) + 1e-6) + 1e-6
    assert float(got[0].abs().max()) == 0.0


def test_rows_are_independent(A):
    N, K = 4096, 4096
    w = normal_tensor(15, 1, N * K, 0.05).view(N, K).to(torch.bfloat16)
    a = normal_tensor(16, 2, 40 * K, 1.0).view(40, K).numpy()
    full = A.anpd_debug_gemm(w, a, plain=3)
    other = a.copy()
    other[1:] = 0.0
    alone = A.anpd_debug_gemm(w, other, plain=3)
    assert np.array_equal(full[0], alone[0]) and float(np.abs(alone[1:]).max()) == 0.0


# every projection on the sweep (rotary, SwiGLU, residual and argmax add a tile's own number of sums), a ragged vocabulary; four sequences
# (32 rows) and fifteen (120)
@pytest.mark.parametrize("batch", [4, 15])
def test_verified_rows_of_a_wide_layer(A, batch, d=4096):
    shape = ModelShape(1, d, 32, 32, 128, 4096, 4100)
    w = make_weights(shape, 3, True, std=0.02)
    dec = Decoder(shape, as_bf16_values(w), torch.float64, kv_dtype=torch.bfloat16)
    st = new_stream()
    m = gpu_model(A, shape, w, st)
    kv = A.anpd_kv_create(m, 128, batch, 1)
    prompts = [markov_prompt(11 + b, shape.vocab, 2, 60 + b).tolist() for b in range(batch)]
    try:
        last, drafts, want = [], [], []
        for b in range(batch):
            A.anpd_prefill(m, kv, prompts[b], b)
            last.append(3 + b)
            drafts.append([7, 9 + b, 11])
        acc, nxt = A.anpd_verify_batch(m, kv, last, drafts)
        checked = 0
        for b in {0, 1, batch - 1}:
            cache = dec.new_cache()
            dec.forward(prompts[b], cache)
            rows = dec.forward([last[b]] + drafts[b], cache)
            top = torch.topk(rows[0], 2).values
            if float(top[0] - top[1]) > 5e-2:                  # decided: the first row's prediction says what is accepted
                pred = int(rows[0].argmax())
                assert (acc[b] > 0) == (drafts[b][0] == pred)
                if acc[b] == 0:
                    assert nxt[b] == pred
                checked += 1
        assert checked >= 2
    finally:
        A.anpd_kv_destroy(kv)
        A.anpd_model_destroy(m)


# residual rows of two chunks of four features per thread with an SM to themselves: little over the rows that share one, and the most (with
# these weights the oracle's margins are 0.31, 0.21, 0.17 at 6160 and 0.04, 1.2, 2.1 at 8192; at 6152 the first three sequences have one above 5e-2)
@pytest.mark.parametrize("batch,d", [(3, 6160), (3, 8192)])
def test_verified_rows_of_wider_rows(A, batch, d):
    test_verified_rows_of_a_wide_layer(A, batch, d)
