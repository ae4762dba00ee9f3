"""GPU parity of the 16-row-tile kernel around its copy rings: lists shorter and longer than a ring, entries cut into
steps, N_kv that ends inside any step, both head dimensions, token-major tensors."""
import numpy as np
import pytest
import torch

from paper_2609_25869_b200 import bsa
from paper_2609_25869_b200 import inputs as I
from tests import helpers as Hh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,B_KV,plan_id", [(64, 64, 34), (64, 32, 35), (64, 16, 36), (128, 32, 35), (128, 16, 36)])
@pytest.mark.parametrize("cut", [0, 1, 17, 63])
def test_list_lengths_around_the_ring(d, B_KV, plan_id, cut):
    n = 7
    M = np.zeros((2, n, n), np.uint8)
    for i in range(n):
        M[0, i, n - 1 - i:] = 1  # i + 1 entries, the last one cut
        M[1, i, :i] = 1          # i entries, none for the first block
    req = I.Request("ring", 2, n * 16 - 3, d, 16, B_KV, M, qkv_seed=d + cut, N_kv=n * B_KV - cut % B_KV)
    Hh.run_request(req, plan_id=plan_id)


def test_token_major_tensors():
    H, N, d = 3, 700, 64
    M = I.random_mask(5, H, I.cdiv(N, 32), I.cdiv(N, 64), 0.4)
    req = I.Request("nhd", H, N, d, 32, 64, M, qkv_seed=9)
    mask, q, k, v, _ = Hh.to_dev(req)
    with bsa.plan_create(mask, 32, 64, N, H, d, plan_id=34) as a:
        O, L = a.forward(q, k, v)
    with bsa.plan_create(mask, 32, 64, N, H, d, plan_id=34, layout="nhd") as b:
        Ot, Lt = b.forward(*(t.permute(1, 0, 2).contiguous() for t in (q, k, v)))
    torch.cuda.synchronize()
    assert torch.equal(Ot.permute(1, 0, 2), O) and torch.equal(Lt, L)


@pytest.mark.parametrize("d,B_KV,plan_id,dtype", [(64, 64, 34, "bf16"), (64, 16, 36, "fp16"), (128, 32, 35, "bf16")])
@pytest.mark.parametrize("growing", [True, False])
def test_scores_that_move_the_running_maximum(d, B_KV, plan_id, dtype, growing):
    """Keys whose length grows or falls along the list: the running maximum moves at nearly every step, or after the first
    ones hardly at all, in some rows of a fragment and not in the rest."""
    n = 12
    M = np.ones((1, 3, n), np.uint8)
    req = I.Request("reference", 1, 40, d, 16, B_KV, M, qkv_seed=3, N_kv=n * B_KV, dtype=dtype)
    q, k, v = req.qkv()
    steps = torch.linspace(0.1, 4.0, n)
    scale = (steps if growing else steps.flip(0)).repeat_interleave(B_KV)[None, :, None]
    Hh.run_request(req, plan_id=plan_id, qkv=(q, (k.float() * scale).to(k.dtype), v), guards=False)
