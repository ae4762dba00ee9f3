"""An item's bits depend on the item alone: not on the items its CTA had before, and not on where the kernel keeps Q, which
follows from the length of the whole request's lists."""
import numpy as np
import pytest
import torch

from paper_2609_25869_b200 import bsa
from paper_2609_25869_b200 import inputs as I
from tests import helpers as Hh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,d,dtype,plan_id", [(128, 64, "bf16", 22), (64, 64, "fp16", 23), (32, 64, "bf16", 39),
                                               (128, 64, "bf16", 24), (128, 128, "bf16", 22), (64, 128, "fp16", 23)])
@pytest.mark.parametrize("N_kv", [1500, 4000])  # about 5 and 13 tiles per item
def test_heads_of_a_whole_request_equal_the_heads_alone(B, d, dtype, plan_id, N_kv):
    H, N = 16, 45 * 128 - 9  # at least 720 work items; a head alone has at most one per CTA, or two (Split-K, 4000 keys)
    M = I.random_mask(d + B, H, I.cdiv(N, B), I.cdiv(N_kv, B), 0.4, empty_rows=0.05)
    req = I.Request("position", H, N, d, B, B, M, qkv_seed=B, N_kv=N_kv, dtype=dtype)
    mask, q, k, v, _ = Hh.to_dev(req)
    kw = {"N_kv": N_kv, "dtype": dtype, "plan_id": plan_id}
    with bsa.plan_create(mask, B, B, N, H, d, **kw) as plan:
        O, L = plan.forward(q, k, v)
        assert plan.info()["nitems"] > 4 * torch.cuda.get_device_properties(0).multi_processor_count
    for h in range(H):
        one = slice(h, h + 1)
        with bsa.plan_create(mask[one].contiguous(), B, B, N, 1, d, **kw) as plan:
            Oh, Lh = plan.forward(q[one].contiguous(), k[one].contiguous(), v[one].contiguous())
        torch.cuda.synchronize()
        assert torch.equal(Lh, L[one]) and torch.equal(Oh, O[one]), h


@pytest.mark.parametrize("B,dtype,plan_id", [(128, "bf16", 22), (64, "fp16", 23), (32, "bf16", 39), (128, "bf16", 24)])
def test_short_lists_next_to_long_ones(B, dtype, plan_id):
    """Head 0 has lists of one to four 128-key tiles; two dense heads beside it lift the average above the length from which
    Q goes through tensor memory.  Both against the oracle, head 0 bit for bit."""
    N, N_kv = 21 * 128 - 5, 40 * 128 - 17
    M = np.ones((3, I.cdiv(N, B), I.cdiv(N_kv, B)), np.uint8)
    M[0] = 0
    for i in range(M.shape[1]):
        M[0, i, (5 * i) % M.shape[2]:][: 1 + (i * B // 128) % 4] = 1
    args, kw = (B, B, N), {"N_kv": N_kv, "dtype": dtype, "plan_id": plan_id}
    req = I.Request("short", 3, N, 128, B, B, M, qkv_seed=B, N_kv=N_kv, dtype=dtype)
    Hh.run_request(req, plan_id=plan_id)
    mask, q, k, v, _ = Hh.to_dev(req)
    with bsa.plan_create(mask, *args, 3, 128, **kw) as plan:
        O, L = plan.forward(q, k, v)
    with bsa.plan_create(mask[:1].contiguous(), *args, 1, 128, **kw) as plan:
        O0, L0 = plan.forward(q[:1].contiguous(), k[:1].contiguous(), v[:1].contiguous())
    torch.cuda.synchronize()
    assert torch.equal(O0, O[:1]) and torch.equal(L0, L[:1])
