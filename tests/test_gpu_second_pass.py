"""The ping-pong kernel's second pass on lists of several items per CTA: marked items stand behind, between and in front of items
that are not computed again, and must get their own list's tiles and membership bits, whatever was left out before them."""
import numpy as np
import pytest
import torch

from paper_2609_25869_b200 import bsa
from paper_2609_25869_b200 import inputs as I
from tests import helpers as Hh

pytestmark = pytest.mark.gpu

H, Q_TILES = 16, 42
MARKED = [(h, (11 * h + 3) % Q_TILES) for h in range(H)] + [(3, 37), (15, 41)]  # (head, Q tile) of the items computed again


def _request(B, d, plan_id):
    """672 items, four to five per CTA, of 12 tiles and more (d = 128) or 38 (d = 64): the form that keeps first references."""
    N = Q_TILES * 128 - 3
    N_kv = (24 if d == 128 else 80) * 128 - 9
    M = I.random_mask(B[0] + d, H, I.cdiv(N, B[0]), I.cdiv(N_kv, B[1]), 0.5, empty_rows=0.03)
    req = I.Request("second", H, N, d, B[0], B[1], M, qkv_seed=B[1] + d, N_kv=N_kv)
    # the estimate by which the kernel's form is chosen
    T_KV = {22: 128, 23: 64, 39: 32}[plan_id]
    entries = I.cdiv(N_kv, T_KV) * (1 - (1 - M.mean()) ** (max(1, 128 // B[0]) * max(1, T_KV // B[1])))
    assert entries * T_KV >= (8 if d == 128 else 32) * 128
    return req


CASES = [((64, 64), 128, 23), ((32, 32), 128, 39), ((64, 128), 128, 22), ((128, 64), 128, 22), ((32, 32), 64, 39),
         ((64, 128), 64, 22), ((128, 128), 64, 22)]


@pytest.mark.parametrize("B,d,plan_id", CASES)
def test_marked_items_between_others(B, d, plan_id):
    """Scores of some rows of a few Q tiles outgrow their first tile by more than 2^100; every row against the oracle."""
    req = _request(B, d, plan_id)
    q, k, v = req.qkv()
    factor = torch.ones(H, req.N, 1)
    for h, t in MARKED:
        factor[h, t * 128 + 96:(t + 1) * 128] = 200.0
    q = (q.float() * factor).to(q.dtype)
    # those rows are one key's: up to 2^-8 |v| off, below the contract's 2e-2 for |v| < 3 (as for the first tile's references)
    Hh.run_request(req, plan_id=plan_id, qkv=(q, k, v * 0.5), structure=False, guards=False)


@pytest.mark.parametrize("B,d,plan_id", CASES)
def test_undefined_rows_stay_alone(B, d, plan_id):
    """A NaN in one query row of a few items: they are computed again, and all their other rows are right."""
    req = _request(B, d, plan_id)
    q, k, v = req.qkv()
    bad = q.clone()
    for h, t in MARKED:
        bad[h, t * 128 + 7, 3] = float("nan")
    mask, qd, kd, vd, cpu = Hh.to_dev(req, (q, k, v))
    with bsa.plan_create(mask, *B, req.N, H, d, plan_id=plan_id, N_kv=req.N_kv) as plan:
        O, L = plan.forward(qd, kd, vd)
        Ob, Lb = plan.forward(bad.cuda(), kd, vd)
        assert plan.info()["device_status"] == 0
    for h, t in MARKED:
        Ob[h, t * 128 + 7], Lb[h, t * 128 + 7] = O[h, t * 128 + 7], L[h, t * 128 + 7]
    Hh.compare_with_oracle(req, Ob, Lb, cpu)
