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


def _against_64_bits(scores_of_keys, values, d, N_kv):
    """One head of 300 rows, dense, every row with (about) the given score per key; outputs against 64 bits."""
    gen = torch.Generator().manual_seed(d)
    q, k, v = (torch.randn(1, n, d, generator=gen) for n in (300, N_kv, N_kv))
    q[..., 0] = 8.0
    k[..., 0] = scores_of_keys * (d ** 0.5 / 8.0)
    q, k, v = (t.bfloat16().cuda() for t in (q, k * torch.tensor([1.0] + [0.1] * (d - 1)), v * values[None, :, None]))
    mask = torch.ones(1, 3, I.cdiv(N_kv, 128), dtype=torch.uint8, device="cuda")
    with bsa.plan_create(mask, 128, 128, 300, 1, d, plan_id=22, N_kv=N_kv) as plan:
        O, L = plan.forward(q, k, v)
        assert plan.info()["device_status"] == 0
    S = q[0].double() @ k[0].double().t() / d ** 0.5
    ref = torch.softmax(S, dim=1) @ v[0].double()
    assert torch.isfinite(O.float()).all()
    assert (L[0].double() - torch.logsumexp(S, dim=1)).abs().max() <= 1e-4
    # P and O are rounded to bf16 (2^-9 each, P's share of the normalisation another 2^-9), relative to the largest |v|
    assert (O[0].double() - ref).abs().max() <= 4 * 2.0 ** -9 * v.double().abs().max()


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("low", [0, 1])  # the tiles of this parity start low and catch up
def test_one_half_of_the_tiles_outgrows_its_first(d, low):
    """At d = 64 each half of an item's tiles has its own reference and accumulator.  One half starts 2^87 below the other and
    reaches it at its second tile: its sum stays below 2^100 and the item's total is small, its accumulator overflows."""
    N_kv = 40 * 128
    s = torch.zeros(40)
    s[1 - low], s[low + 2] = 60.0, 60.0
    _against_64_bits(s.repeat_interleave(128), torch.full((N_kv,), 2.0 ** 60), d, N_kv)


@pytest.mark.parametrize("d", [64, 128])
def test_one_large_value_behind_a_moderate_weight(d):
    """A weight of 2^20 against the first tile on a value of about 2^110: their product overflows, the row's sum is small."""
    N_kv = 40 * 128
    s, x = torch.zeros(N_kv), torch.ones(N_kv)
    s[700], x[700] = 14.0, 2.0 ** 110
    _against_64_bits(s, x, d, N_kv)


def test_marks_are_not_shared_in_long_lists():
    """More than 1024 items per SM: items computed again change no bit of any other, whose scores outgrow their first tile too."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    H, d, nk = 64, 128, 12
    nq = 1024 * sms // H + 5
    N, N_kv = nq * 128, nk * 128
    gen = torch.Generator(device="cuda").manual_seed(9)
    q = torch.randn(H, N, d, device="cuda", generator=gen, dtype=torch.bfloat16)
    k, v = (torch.randn(H, N_kv, d, device="cuda", generator=gen, dtype=torch.bfloat16) for _ in range(2))
    k[:, -200:] *= 8
    mask = torch.ones(H, nq, nk, dtype=torch.uint8, device="cuda")
    marked = [(0, 1), (17, nq // 2), (40, 3), (63, nq - 1)]
    with bsa.plan_create(mask, 128, 128, N, H, d, plan_id=22, N_kv=N_kv) as plan:
        O, L = plan.forward(q, k, v)
        for h, t in marked:
            q[h, t * 128:(t + 1) * 128] *= 60
        Ob, Lb = plan.forward(q, k, v)
        assert plan.info()["device_status"] == 0 and plan.info()["nitems"] > 1024 * sms
    same = torch.ones(H, nq, dtype=torch.bool, device="cuda")
    for h, t in marked:
        same[h, t] = False
        assert not torch.equal(Lb[h, t * 128:(t + 1) * 128], L[h, t * 128:(t + 1) * 128])
    assert ((O.view(H, nq, -1) == Ob.view(H, nq, -1)).all(dim=2) | ~same).all()
    assert ((L.view(H, nq, -1) == Lb.view(H, nq, -1)).all(dim=2) | ~same).all()
