"""GPU parity of the ping-pong kernel on tiles gathered from several narrow entries of the tile list (two of 64 keys,
four of 32): list lengths around multiples of the entries per tile, ragged last blocks, every row-block size, both
head dimensions and element types, Split-K partitions that start anywhere in the list."""
import numpy as np
import pytest
import torch

from paper_2609_25869_b200 import bsa
from paper_2609_25869_b200 import inputs as I
from tests import helpers as Hh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B_Q,B_KV,N,N_kv,d,dtype,plan_id", [
    (16, 16, 1000, 0, 64, "bf16", 39), (16, 32, 777, 1300, 128, "bf16", 39), (32, 16, 900, 0, 128, "fp16", 40),
    (32, 32, 3000, 0, 128, "bf16", 42), (64, 32, 1300, 1111, 64, "fp16", 41), (128, 32, 1000, 0, 128, "bf16", 39),
    (256, 16, 900, 0, 64, "bf16", 43), (32, 32, 2000, 3001, 128, "bf16", 43),
    (16, 16, 1000, 0, 128, "bf16", 23), (32, 32, 1500, 0, 64, "fp16", 26), (64, 64, 1301, 0, 128, "bf16", 33),
    (128, 64, 2000, 999, 128, "fp16", 32), (16, 64, 1000, 0, 64, "bf16", 28), (256, 256, 1100, 0, 128, "bf16", 23),
    (64, 128, 1000, 0, 128, "bf16", 27)])
def test_gathered_tiles_match_the_oracle(B_Q, B_KV, N, N_kv, d, dtype, plan_id):
    H = 3
    M = I.random_mask(B_Q + 7 * B_KV + N, H, I.cdiv(N, B_Q), I.cdiv(N_kv or N, B_KV), 0.3, empty_rows=0.15)
    Hh.run_request(I.Request("gather", H, N, d, B_Q, B_KV, M, qkv_seed=N, N_kv=N_kv, dtype=dtype), plan_id=plan_id)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,plan_id", [(32, 39), (64, 23), (128, 22)])
def test_list_lengths_around_whole_tiles(B, plan_id, d):
    """Query block i has i + 1 active key blocks: lists of 1, 2, ... entries, each with the ragged last block or not."""
    n = 13
    M = np.zeros((2, n, n), np.uint8)
    for i in range(n):
        M[0, i, n - 1 - i:] = 1
        M[1, i, :i + 1] = 1
    Hh.run_request(I.Request("lengths", 2, n * B - 5, d, B, B, M, qkv_seed=B), plan_id=plan_id)
    # 128-row query blocks: every list length belongs to one work item
    Hh.run_request(I.Request("lengths", 2, n * 128, d, 128, B, M, qkv_seed=B + 1, N_kv=n * B - 5), plan_id=plan_id)


@pytest.mark.parametrize("d", [64, 128])
def test_rows_that_only_every_other_tile_reaches(d):
    """Two row blocks of one work item whose tiles alternate: each of the two softmax warpgroups sees only masked tiles
    for half of its rows, in lists of two tiles and more."""
    M = np.zeros((2, 6, 9), np.uint8)
    M[0, 0::2, 0::2] = 1
    M[0, 1::2, 1::2] = 1
    M[1, 0, 0] = M[1, 1, 1] = M[1, 2, 3] = M[1, 3, 8] = M[1, 5, 8] = 1
    req = I.Request("alternating", 2, 6 * 64, d, 64, 128, M, qkv_seed=3, N_kv=9 * 128 - 40)
    for plan_id in (22, 24):
        Hh.run_request(req, plan_id=plan_id)


@pytest.mark.parametrize("B,d,dtype,plan_id", [(32, 64, "fp16", 39), (32, 128, "bf16", 43), (64, 64, "bf16", 23), (64, 128, "fp16", 28)])
def test_token_major_gathered_tiles(B, d, dtype, plan_id):
    """The copies of narrow entries out of token-major tensors: the same bits as head-major, which the oracle checks."""
    H, N, N_kv = 3, 1000, 1301
    M = I.random_mask(B + d, H, I.cdiv(N, B), I.cdiv(N_kv, B), 0.35, empty_rows=0.1)
    req = I.Request("nhd", H, N, d, B, B, M, qkv_seed=B, N_kv=N_kv, dtype=dtype)
    Hh.run_request(req, plan_id=plan_id)
    mask, q, k, v, _ = Hh.to_dev(req)
    kw = {"N_kv": N_kv, "dtype": dtype, "plan_id": plan_id}
    with bsa.plan_create(mask, B, B, N, H, d, **kw) as plan:
        O, L = plan.forward(q, k, v)
    with bsa.plan_create(mask, B, B, N, H, d, layout="nhd", **kw) as plan:
        Ot, Lt = plan.forward(*(t.permute(1, 0, 2).contiguous() for t in (q, k, v)))
    torch.cuda.synchronize()
    assert torch.equal(Ot.permute(1, 0, 2), O) and torch.equal(Lt, L)
