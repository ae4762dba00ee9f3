"""Tensors that lie on the 16-byte boundary the entry points ask for, and on no wider one."""
import pytest
import torch

from paper_2609_25869_b200 import bsa
from paper_2609_25869_b200 import inputs as I
from tests import helpers as Hh

pytestmark = pytest.mark.gpu


def _shifted(t):
    """The same values 16 bytes behind an allocation's start."""
    step = 16 // t.element_size()
    buf = torch.empty(t.numel() + step, dtype=t.dtype, device=t.device)
    out = buf[step:].view(t.shape)
    out.copy_(t)
    assert out.data_ptr() % 32 == 16
    return out


@pytest.mark.parametrize("B_Q,B_KV,d,plan_id", [(128, 128, 128, 22), (64, 64, 64, 23), (64, 64, 128, 27), (32, 32, 64, 39),
                                                (64, 64, 64, 19), (16, 64, 64, 34), (128, 128, 256, -1)])
def test_tensors_on_16_byte_boundaries(B_Q, B_KV, d, plan_id):
    H, N = 2, 900
    M = I.random_mask(B_Q + d, H, I.cdiv(N, B_Q), I.cdiv(N, B_KV), 0.4)
    req = I.Request("align", H, N, d, B_Q, B_KV, M, qkv_seed=d)
    mask, q, k, v, _ = Hh.to_dev(req)
    with bsa.plan_create(mask, B_Q, B_KV, N, H, d, plan_id=plan_id) as plan:
        O, L = plan.forward(q, k, v)
        O2 = _shifted(torch.zeros_like(O))
        _, L2 = plan.forward(_shifted(q), _shifted(k), _shifted(v), O2, torch.empty_like(L))
        torch.cuda.synchronize()
    assert torch.equal(O, O2) and torch.equal(L, L2)


@pytest.mark.parametrize("B_Q,B_KV,d,plan_id", [(128, 128, 128, 22), (64, 64, 64, 23), (32, 32, 128, 39)])
def test_token_major_half_tensors_on_16_byte_boundaries(B_Q, B_KV, d, plan_id):
    H, N = 3, 900
    M = I.random_mask(B_Q + d, H, I.cdiv(N, B_Q), I.cdiv(N, B_KV), 0.4)
    req = I.Request("align", H, N, d, B_Q, B_KV, M, qkv_seed=d, dtype="fp16")
    mask, q, k, v, _ = Hh.to_dev(req)
    q, k, v = (t.permute(1, 0, 2).contiguous() for t in (q, k, v))
    with bsa.plan_create(mask, B_Q, B_KV, N, H, d, dtype="fp16", layout="nhd", plan_id=plan_id) as plan:
        O, L = plan.forward(q, k, v)
        O2 = _shifted(torch.zeros_like(O))
        _, L2 = plan.forward(_shifted(q), _shifted(k), _shifted(v), O2, torch.empty_like(L))
        torch.cuda.synchronize()
    assert torch.equal(O, O2) and torch.equal(L, L2)
