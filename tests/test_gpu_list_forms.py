"""Lists whose rows are reached late, or by no tile at all, on both sides of the lines where the ping-pong kernel changes its
form: a few active blocks per row block, in lists of many tiles that its neighbours need."""
import numpy as np
import pytest
import torch

from paper_2609_25869_b200 import bsa
from paper_2609_25869_b200 import inputs as I
from tests import helpers as Hh

pytestmark = pytest.mark.gpu


# (d, blocks, plan, 128-key tiles in all, density): about 9, 25 and 70 tiles per item at d = 128, 34 and 180 at d = 64
@pytest.mark.parametrize("d,B,plan_id,n_kt,density", [
    (128, (16, 64), 23, 75, 0.016), (128, (16, 64), 23, 180, 0.02), (128, (16, 64), 23, 180, 0.06),
    (128, (32, 64), 23, 75, 0.032), (128, (32, 64), 23, 75, 0.1), (128, (16, 128), 22, 75, 0.016), (128, (16, 128), 22, 180, 0.06),
    (128, (16, 32), 39, 75, 0.02), (64, (16, 128), 22, 75, 0.08), (64, (16, 128), 22, 400, 0.09), (64, (32, 128), 22, 180, 0.15),
    (64, (16, 32), 39, 75, 0.08), (64, (128, 32), 39, 100, 0.4), (64, (128, 32), 39, 100, 0.6)])
def test_rows_reached_late(d, B, plan_id, n_kt, density):
    H, N, N_kv = 2, 5 * 128 - 7, n_kt * 128 - 11
    M = I.random_mask(d + B[0] + n_kt, H, I.cdiv(N, B[0]), I.cdiv(N_kv, B[1]), density, empty_rows=0.05)
    M[1, ::3, : -M.shape[2] // 8] = 0  # every third row block of one head: the last eighth of the keys only
    Hh.run_request(I.Request("late", H, N, d, B[0], B[1], M, qkv_seed=n_kt, N_kv=N_kv), plan_id=plan_id)


@pytest.mark.parametrize("d,B,plan_id", [(64, 128, 22), (64, 32, 39), (128, 64, 23), (128, 128, 22)])
def test_heads_of_a_whole_request_equal_the_heads_alone(d, B, plan_id):
    """Long lists that keep first references, some of their items computed again: 720 items against 45, bit for bit."""
    H, N, N_kv = 16, 45 * 128 - 9, 63 * 128 - 5
    M = I.random_mask(d + B, H, I.cdiv(N, B), I.cdiv(N_kv, B), 0.85, empty_rows=0.05)
    req = I.Request("position", H, N, d, B, B, M, qkv_seed=B, N_kv=N_kv)
    mask, q, k, v, _ = Hh.to_dev(req)
    for h in range(H):
        for t in {(7 * h + 2) % 45, (11 * h) % 45, 44}:
            q[h, t * 128 + 9:t * 128 + 30] *= 200
    kw = {"N_kv": N_kv, "plan_id": plan_id}
    with bsa.plan_create(mask, B, B, N, H, d, **kw) as plan:
        O, L = plan.forward(q, k, v)
        assert plan.info()["nitems"] > 4 * torch.cuda.get_device_properties(0).multi_processor_count
    for h in range(H):
        one = slice(h, h + 1)
        with bsa.plan_create(mask[one].contiguous(), B, B, N, 1, d, **kw) as plan:
            Oh, Lh = plan.forward(q[one].contiguous(), k[one].contiguous(), v[one].contiguous())
            assert plan.info()["device_status"] == 0
        assert torch.equal(Lh, L[one]) and torch.equal(Oh, O[one]), h


@pytest.mark.parametrize("d,B,plan_id", [(128, (16, 64), 23), (128, (32, 64), 23), (128, (32, 128), 22), (128, (64, 64), 23),
                                         (64, (32, 32), 39), (64, (64, 128), 22)])
@pytest.mark.parametrize("layout", ["hnd", "nhd"])
def test_runs_that_differ_from_row_to_row(d, B, plan_id, layout):
    """Two runs of keys per row block, wherever they begin: many more blocks in runs than independent ones would have."""
    H, N, N_kv = 2, 4 * 128 - 3, 130 * 128 - 21
    nq, nk = I.cdiv(N, B[0]), I.cdiv(N_kv, B[1])
    rng = np.random.RandomState(d + B[0])
    M = np.zeros((H, nq, nk), np.uint8)
    for h in range(H):
        for i in range(nq):
            for a in rng.randint(0, nk - nk // 6, 2):
                M[h, i, a:a + nk // 6] = 1
    req = I.Request("runs", H, N, d, B[0], B[1], M, qkv_seed=d, N_kv=N_kv)
    mask, q, k, v, cpu = Hh.to_dev(req)
    nhd = layout == "nhd"
    with bsa.plan_create(mask, *B, N, H, d, plan_id=plan_id, N_kv=N_kv, layout=layout) as plan:
        O, L = plan.forward(*(t.transpose(0, 1).contiguous() if nhd else t for t in (q, k, v)))
        assert plan.info()["device_status"] == 0
    Hh.compare_with_oracle(req, O.transpose(0, 1).contiguous() if nhd else O, L, cpu)
