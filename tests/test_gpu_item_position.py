"""An item's bits depend on the item alone: whole requests, whose CTAs walk several items one after the other, against
their heads run one at a time, where no CTA has more than one item."""
import pytest
import torch

from paper_2609_25869_b200 import bsa
from paper_2609_25869_b200 import inputs as I
from tests import helpers as Hh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,d,dtype,plan_id", [(128, 64, "bf16", 22), (64, 64, "fp16", 23), (32, 64, "bf16", 39),
                                               (128, 64, "bf16", 24), (128, 128, "bf16", 22), (64, 128, "fp16", 23)])
def test_heads_of_a_whole_request_equal_the_heads_alone(B, d, dtype, plan_id):
    H, N, N_kv = 16, 45 * 128 - 9, 1500  # at least 720 work items, at most 135 for a head alone
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
            assert plan.info()["nitems"] <= 148
        torch.cuda.synchronize()
        assert torch.equal(Lh, L[one]) and torch.equal(Oh, O[one]), h
