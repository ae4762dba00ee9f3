"""The ping-pong kernel's items whose reference maximum, taken from the first tile that reaches a row, does not serve: weights
that overflow against it, accumulators that overflow, rows that no tile reaches, rows that a late tile reaches first."""
import numpy as np
import pytest
import torch

from paper_2609_25869_b200 import bsa
from paper_2609_25869_b200 import inputs as I
from tests import helpers as Hh

pytestmark = pytest.mark.gpu


def _request(B, N_kv, late_rows, seed=5, d=128):
    """Three heads of 300 query rows, lists long enough for the form that keeps a row's first reference."""
    N = 300
    nq, nk = I.cdiv(N, B), I.cdiv(N_kv, B)
    M = I.random_mask(seed + B, 3, nq, nk, 0.8, empty_rows=0.1)
    if late_rows:  # every other row block is reached by the last blocks only, its neighbours from the first on
        M[:, ::2, : nk - 3] = 0
        M[:, 1::2] = 1
    return I.Request("first", 3, N, d, B, B, M, qkv_seed=seed, N_kv=N_kv)


@pytest.mark.parametrize("B,plan_id,d", [(128, 22, 128), (64, 23, 128), (32, 39, 128), (128, 22, 64), (32, 39, 64)])
@pytest.mark.parametrize("late_rows", [False, True])
@pytest.mark.parametrize("top", [1.0, 8.0, 60.0])  # scores up to about 5, 40 and 300 (in units of e)
def test_scores_that_outgrow_the_first_tile(B, plan_id, d, late_rows, top):
    req = _request(B, (25 if d == 128 else 45) * 128 - 7, late_rows, d=d)
    q, k, v = req.qkv()
    scale = torch.ones(req.n_kv)
    scale[-200:] = top
    k = (k.float() * scale[None, :, None]).to(k.dtype)
    q[0, 100:] *= 0.05  # these rows never leave the range of their first tile
    # a row that one key dominates is off by up to half a unit of its weight and half of its output, 2^-8 |v| in all:
    # with |v| < 3 below the contract's 2e-2
    v = v * 0.5
    Hh.run_request(req, plan_id=plan_id, qkv=(q, k, v), guards=False)


def test_values_that_overflow_an_accumulator_of_large_weights():
    """Weights of 2^40 against the first tile and values of 2^100: the sum fits, the accumulator does not."""
    req = _request(128, 24 * 128, False)
    q, k, v = req.qkv()
    scale = torch.ones(req.n_kv)
    scale[-130:] = 8.0
    k = (k.float() * scale[None, :, None]).to(k.dtype)
    mask, qd, kd, vd, _ = Hh.to_dev(req, (q, k, v))
    with bsa.plan_create(mask, 128, 128, req.N, req.H, 128, plan_id=22, N_kv=req.N_kv) as plan:
        O, L = plan.forward(qd, kd, vd)
        Ob, Lb = plan.forward(qd, kd, (vd.float() * 2.0 ** 100).to(vd.dtype))
        assert plan.info()["device_status"] == 0
    assert torch.isfinite(Ob.float()).all()
    assert torch.allclose(Lb, L, atol=1e-4, rtol=0, equal_nan=True) or torch.equal(torch.isinf(Lb), torch.isinf(L))
    # two forms of the same rows: each is within half a unit of 2^-8 of P and of O
    assert (Ob.double() * 2.0 ** -100 - O.double()).abs().max() <= 4 * 2.0 ** -8 * O.double().abs().max()


def test_infinite_and_undefined_inputs_stay_in_their_rows():
    req = _request(128, 24 * 128, False)
    q, k, v = req.qkv()
    clean = Hh.to_dev(req, (q, k, v))
    q = q.clone()
    q[1, 5, 0] = float("inf")
    q[2, 7, 3] = float("nan")
    mask, qd, kd, vd, _ = Hh.to_dev(req, (q, k, v))
    with bsa.plan_create(mask, 128, 128, req.N, req.H, 128, plan_id=22, N_kv=req.N_kv) as plan:
        O, L = plan.forward(*clean[1:4])
        Oi, Li = plan.forward(qd, kd, vd)
        assert plan.info()["device_status"] == 0
    same = torch.ones((3, req.N), dtype=torch.bool, device="cuda")
    same[1, :128] = same[2, :128] = False  # (the items of the two rows are computed again)
    assert torch.equal(Oi[same], O[same])
    rest = ~same
    rest[1, 5] = rest[2, 7] = False
    assert (Oi[rest].double() - O[rest].double()).abs().max() <= 4 * 2.0 ** -8 * O[rest].double().abs().max()
    assert torch.equal(torch.isneginf(Li[rest]), torch.isneginf(L[rest]))
