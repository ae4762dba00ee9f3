"""Order of the work items against a stable sort on the host: lists around the ranking kernel's rows and tiles, and on
both sides of the length from which the sorts take over (2^28 comparisons: several CTAs for the global orders, one per
head for the head-major ones); every order; exported items, no forward."""
import numpy as np
import pytest
import torch

from paper_2609_25869_b200 import bsa

pytestmark = pytest.mark.gpu


def _bucket(n):  # half-octaves: 0, 1, 2, 3, 4-5, 6-7, 8-11, 12-15, ...
    n = np.asarray(n)
    lz = np.floor(np.log2(np.maximum(n, 2))).astype(int)
    return np.where(n <= 1, n, 2 * lz + ((n >> (lz - 1)) & 1))


@pytest.mark.parametrize("plan_id", [22, 25, 29, 30, 31])
@pytest.mark.parametrize("H,rows", [(1, 1), (3, 31), (2, 33), (5, 64), (1, 2047), (2, 2049), (4, 4100), (7, 2900), (2, 12000)])
def test_items_are_in_stable_order(H, rows, plan_id):
    nk = 37
    r = np.random.RandomState(H * 10000 + rows)
    M = (r.rand(H, rows, nk) < r.choice([0.0, 0.1, 0.5, 1.0], size=(H, rows, 1))).astype(np.uint8)
    with bsa.plan_create(torch.from_numpy(M).cuda(), 128, 128, rows * 128, H, 64, N_kv=nk * 128, plan_id=plan_id) as plan:
        items = plan.export_items()
    n = M.sum(axis=2).reshape(-1).astype(int)
    key = _bucket(n) if plan_id in (30, 31) else n
    head = np.repeat(np.arange(H), rows)
    if plan_id == 29:
        want = np.arange(H * rows)
    elif plan_id in (25, 31):
        want = np.argsort(-key, kind="stable")
    else:
        want = np.lexsort((-key, head))
    assert len(items) == H * rows
    assert np.array_equal(items[:, 0] * rows + items[:, 1], want)
    assert np.array_equal(items[:, 7], n[want]) and np.array_equal(items[:, 3] - items[:, 2], n[want])
    assert (items[:, 4] == 0).all() and (items[:, 5] == 1).all()
